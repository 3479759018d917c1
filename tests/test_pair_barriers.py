"""Barriers of the kernels on pairs of CTAs: what can be read from the source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_05528_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "map_to_cta(" in open(os.path.join(CSRC, f)).read())


@pytest.mark.parametrize("name", FILES)
def test_a_barrier_that_the_partner_signals_is_waited_for_at_cluster_scope(name):
    """A barrier that is signalled through map_to_cta takes arrivals from both CTAs.  mbar_wait acquires at the scope of the
    own CTA only, so what the partner did before its arrival would not be ordered before what follows the wait."""
    text = open(os.path.join(CSRC, name)).read()
    seen = 0
    for kernel in re.split(r"\b__global__\b", text)[1:]:
        shared = set(re.findall(r"map_to_cta\(\s*(\w+)", kernel))
        waited = set(re.findall(r"\bmbar_wait\(\s*(\w+)", kernel))
        at_cluster = set(re.findall(r"\bmbar_wait_cluster\(\s*(\w+)", kernel))
        assert not shared & waited, (name, shared & waited)
        assert shared <= at_cluster, (name, shared - at_cluster)
        seen += len(shared)
    assert seen


def test_the_kernels_on_pairs_are_found():
    assert {"gemm_tcgen05.cu", "blockpair_tcgen05.cu", "sparse_tcgen05.cu"} <= set(FILES)
