"""Kernels that are launched while the kernel before them may still run: each opens with grid_begin(), or takes its tensor memory
and then calls it, before anything else, and declares nothing it reads __restrict__, const or not, nor reads it through __ldg (a load of
such data may be moved above the wait).  The kernels that fetch something ahead of their wait are named with what that is.  Read
off the sources: on a GPU a missing wait is a race that need not show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_05528_b200", "csrc")
TEXT = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def _by_hand(text):
    """Kernels of functions that set the attribute themselves."""
    for body in re.split(r"\n}\n", text):
        if "cudaLaunchAttributeProgrammaticStreamSerialization" in body:
            yield from re.findall(r"cudaLaunchKernelEx\(&\w+, (\w+_kernel)", body)


LAUNCHED = sorted({(f, k) for f, t in TEXT.items() for k in re.findall(r"launch_dependent\((\w+_kernel)", t)})
BY_HAND = sorted({(f, k) for f, t in TEXT.items() for k in _by_hand(t)})

# The kernels that do not open with grid_begin() in every form: all of the names of their parameters that may stand ahead of the
# wait, and why what is read there is complete.
AHEAD = {
    # the packed wrappers: the pass's first kernel, two launches earlier, has waited for whatever wrote them
    "fwd_small_kernel": {"Q"},
    # the packed core: the kernel before lets this one in behind its own wait, so whatever wrote the core has ended.  (mapB, the
    # tokens' map, stands there in a function that is called behind the wait.)
    "tc_sparse_small_kernel": {"mapA", "mapE", "mapB", "k_per_piece", "p"},
    # a Gram's product behind the kernel that looks at the channels, which starts when all before it has ended and writes
    # nothing but the scales
    "tc_gemm_kernel": {"mapA", "mapAlo", "mapB", "mapBlo", "p"},
}
# Outputs that are written through a pointer formed from them, as the reader finds; the kernels load nothing there
WRITTEN = {"sum_slabs_kernel": {"out0", "out1"}, "bgemm_tile_kernel": {"part_out"}, "split_rows_kernel": {"hi", "lo"}}
# Data read through __ldg, and why that is older than the kernel before
LDG = {
    ("split_f16.cu", "__ldg(reinterpret_cast<const uint4*>(X + r * ldx + col))"): "gram_range_kernel, launched without the attribute",
}


def _closing(text, at):
    depth = 0
    for i in range(at, len(text)):
        depth += {"(": 1, ")": -1, "[": 1, "]": -1}.get(text[i], 0)
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def _bare(text):
    return re.sub(r"//[^\n]*", "", text)


def _kernel(text, name):
    """(parameter list, body) of a __global__ function."""
    for m in re.finditer(r"__global__", text):
        d = re.compile(r"(\w+_kernel)\s*\(").search(text, m.end())
        if d.group(1) == name:
            end = _closing(text, d.end() - 1)
            body = text[text.index("{", end) + 1:]
            return _bare(text[d.end():end]), _bare(body[:body.index("\n}\n")])
    raise AssertionError(name)


def _only_written(name, body):
    """Every mention of the pointer is the left side of an assignment, an address for an atomic operation or a comparison with null."""
    for m in re.finditer(rf"\b{name}\b", body):
        rest = body[m.end():]
        if re.search(r"(atomicAdd|atomicOr|atomicMax|atomicCAS)\(&$", body[:m.start()]):
            continue
        if re.search(r"\bif \($", body[:m.start()]) and rest.startswith(")"):
            continue
        vector = re.search(r"\*reinterpret_cast<[\w* ]+>\($", body[:m.start()])
        if vector:
            rest = body[_closing(body, vector.end() - 1) + 1:]
        elif rest.startswith("["):
            rest = body[_closing(body, m.end()) + 1:]
        elif not re.search(r"[;)]\s*\*$", body[:m.start()]):
            return False
        rest = re.sub(r"^\.\w+", "", rest)
        if not re.match(r"\s*=(?!=)", rest):
            return False
    return True


def test_there_are_such_kernels():
    assert len(LAUNCHED) > 30
    assert {k for _, k in BY_HAND} == {"tc_gemm_kernel", "tc_gemm_fixup_kernel", "tc_blockpair_kernel", "fwd_small_kernel",
                                       "tc_sparse_small_kernel"}


@pytest.mark.parametrize("name,kernel", LAUNCHED + BY_HAND)
def test_nothing_that_is_read_is_restrict(name, kernel):
    params, body = _kernel(TEXT[name], kernel)
    for p in params.split(","):
        if "__restrict__" in p:
            assert not re.search(r"\bconst\b", p), p
            out = re.search(r"(\w+)\s*$", p).group(1)
            assert out in WRITTEN.get(kernel, ()) or _only_written(out, body), p
    assert "__restrict__" not in body


@pytest.mark.parametrize("name,kernel", LAUNCHED + [(f, k) for f, k in BY_HAND if k not in AHEAD])
def test_waits_before_it_reads(name, kernel):
    params, body = _kernel(TEXT[name], kernel)
    before = re.sub(r"constexpr[^;]*;", "", body[:body.index("grid_begin();")])
    if before.strip():
        # what may stand before it: setting up shared memory, barriers and tensor memory
        assert "tcgen05.alloc" in before and "return" not in before
        assert not re.search(r"tma_load|tma_store|tmem_ld|ld\.global|st\.global", before)


@pytest.mark.parametrize("name,kernel", [(f, k) for f, k in BY_HAND if k in AHEAD])
def test_reads_ahead_of_the_wait_only_what_is_named(name, kernel):
    params, body = _kernel(TEXT[name], kernel)
    before = body[:body.rindex("grid_dependency_wait();")]
    names = [re.search(r"(\w+)\s*$", p).group(1) for p in params.split(",") if re.search(r"\*|CUtensorMap|Params", p)]
    assert {n for n in names if re.search(rf"\b{n}\b", before)} <= AHEAD[kernel]
    assert not re.search(r"tma_store|st\.global|ld\.global", before)
    if "tcgen05.alloc" in before:        # tensor memory before the next kernel is let in
        lets_in = [before.index(s) for s in ("grid_launch_dependents();", "grid_begin();") if s in before]
        assert lets_in and before.index("tcgen05.alloc") < min(lets_in)


def test_order_of_the_forward_of_few_tokens():
    """The first product of a pass lets the core product in behind its wait; the core product asks for tokens behind its own."""
    _, body = _kernel(TEXT["fwd_tcgen05.cu"], "fwd_small_kernel")
    assert body.index("if (!SUM) grid_dependency_wait();") < body.index("grid_launch_dependents();")
    _, body = _kernel(TEXT["sparse_tcgen05.cu"], "tc_sparse_small_kernel")
    calls = [m.start() for m in re.finditer(r"\bload_z\(", body)]
    assert calls and body.index("grid_dependency_wait();") < min(calls)
    # a Gram's product reads its scales behind the wait, and the kernel before it is launched without the attribute
    _, body = _kernel(TEXT["gemm_tcgen05.cu"], "tc_gemm_kernel")
    assert "row_scale" not in body[:body.index("if (p.dependent) grid_dependency_wait();")]
    assert ("split_f16.cu", "gram_range_kernel") not in LAUNCHED + BY_HAND


def test_loads_through_the_read_only_path():
    found = {(f, m.group(0)) for f, t in TEXT.items() for m in re.finditer(r"__ldg\((?:[^()]|\([^()]*\))*\)", _bare(t))}
    assert found == set(LDG)
    assert "ld.global.nc" not in "".join(TEXT.values())
