"""The bound on how many groups of sources one list of the indexed walks serves, on the CPU."""
import pytest

import paper_1908_10583_gb300 as fora
from paper_1908_10583_gb300 import build as fbuild

CHUNK = 1024  # a node of more walks is listed, its walks in chunks of this many


@pytest.mark.parametrize("width", [1, 4])
@pytest.mark.parametrize("n", [1, 2, 255, 1 << 14, 1 << 20, 1 << 22, (1 << 22) + 1, 1 << 24,
                               (1 << 24) + 1, 1 << 25, (1 << 31) - 1])
def test_a_list_counts_its_nodes_and_chunks(n, width):
    """Nodes are counted in 28 bits, chunks in 36; the largest counts a group can bring are those
    of `width` sources of 2^32 - 1 walks each, all on nodes of 1025 walks or all on one node."""
    fbuild.build()
    groups = fora.index_list_groups(n, width)
    walks = width * ((1 << 32) - 1)
    nodes = min(n, walks // (CHUNK + 1))
    chunks = nodes + walks // CHUNK
    assert groups >= 1
    assert groups * nodes < 1 << 28
    assert groups * chunks < 1 << 36


def test_the_bound_is_reached_by_large_batches():
    """1100 sources of 2^20 nodes, most of them listed in every group, would count 275 * 2^20 nodes:
    past 28 bits, so they take more than one list; batches of the usual sizes take one."""
    fbuild.build()
    assert fora.index_list_groups(1 << 20, 4) < 1100 // 4
    assert fora.index_list_groups(1 << 20, 4) >= 256 // 4
    for n, width in ((0, 4), (1 << 31, 4), (5, 0), (5, 33)):
        with pytest.raises(fora.FORAError):
            fora.index_list_groups(n, width)
