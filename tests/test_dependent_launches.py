"""Kernels that are launched while the kernel before them may still run: each opens with grid_begin(), or takes its tensor memory
and then calls it, before anything else, and declares nothing it reads __restrict__ (a load of such data may be moved above the
wait).  Read off the sources: on a GPU a missing wait is a race that need not show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_05528_b200", "csrc")
TEXT = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")}
LAUNCHED = sorted({(f, k) for f, t in TEXT.items() for k in re.findall(r"launch_dependent\((\w+)", t)})


def _closing(text, at):
    depth = 0
    for i in range(at, len(text)):
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def _kernel(text, name):
    """(parameter list, body) of a __global__ function."""
    for m in re.finditer(r"__global__", text):
        d = re.compile(r"(\w+_kernel)\s*\(").search(text, m.end())
        if d.group(1) == name:
            end = _closing(text, d.end() - 1)
            body = text[text.index("{", end) + 1:]
            return text[d.end():end], body[:body.index("\n}\n")]
    raise AssertionError(name)


def test_there_are_such_kernels():
    assert len(LAUNCHED) > 30


@pytest.mark.parametrize("name,kernel", LAUNCHED)
def test_waits_before_it_reads(name, kernel):
    params, body = _kernel(TEXT[name], kernel)
    for p in params.split(","):
        assert not (re.search(r"\bconst\b.*\*", p) and "__restrict__" in p), p
    before = body[:body.index("grid_begin();")]
    if before.strip():
        # what may stand before it: setting up shared memory, barriers and tensor memory
        assert "tcgen05.alloc" in before and "return" not in before
        assert not re.search(r"tma_load|tma_store|tmem_ld|ld\.global|st\.global", before)
