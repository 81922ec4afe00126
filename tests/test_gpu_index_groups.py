"""Indexed walks of groups of sources (1 or 4 side by side, the last group not full): nodes of
few walks, of walks around a warp's step and a chunk of 1024, and hubs of many chunks, against the
oracle on given residues."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_index import _debug  # noqa: E402
from tests.test_gpu_parity import _built  # noqa: E402,F401

SEED, RMAX = 11, 1e-3


# node counts around the nodes of a warp (64 in groups of four, 256 alone)
@pytest.mark.parametrize("n,nsrc", [(1, 1), (63, 3), (65, 4), (255, 2), (257, 1), (300, 6), (300, 9)])
def test_indexed_walks_of_groups_are_bit_exact(n, nsrc):
    rng = np.random.default_rng(1000 * n + nsrc)
    edges = [(v, int(u)) for v in range(n) for u in rng.integers(0, n, 1 + rng.poisson(3))]
    edges += [(v, int(u)) for v in range(min(3, n)) for u in rng.integers(0, n, 700 * (v + 1))]
    rp, col = inputs.csr_from_edges(n, edges)
    deg = np.diff(rp)
    g = fora.Graph(rp, col)
    # C is about 6e4: 60 walks for an edge, up to 1e5 for a hub
    g.build_index(fora.Params.make(k=1, delta=1e-3, pf=1e-3, rmax=RMAX, seed=SEED))
    rmax, C, _ = g.index_info()
    off, dest = oracle.walk_index(rp, col, 0.2, C, rmax, SEED)
    walks = rng.choice([0.0, 0.5, 1, 7, 8, 9, 31, 32, 33, 1023, 1024, 1025, 2049, 1e9], (nsrc, n))
    r = np.minimum(walks / C, rmax * deg)
    r[0] = rmax * deg  # every stored walk
    res = rng.random((nsrc, n))
    p = fora.Params.make(k=1, delta=1e-3, pf=1e-3, rmax=RMAX, seed=1, flags=fora.FORA_USE_INDEX)
    sources = rng.integers(0, n, nsrc).astype(np.int32)
    _, _, st, out = _debug(g, sources, p, given=(res, r))
    for i in range(nsrc):
        cnt, acc, wst = oracle.walk_phase_indexed(n, C, r[i], off, dest)
        np.testing.assert_array_equal(out["count"][i], cnt)
        np.testing.assert_array_equal(out["acc"][i], acc)
        np.testing.assert_array_equal(out["estimate"][i], oracle.estimate(res[i], acc))
        assert st[i].walks == wst.walks
    g.close()


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("nsrc", [2, 9, 16])
def test_indexed_walks_in_several_lists_are_the_same(groups, nsrc):
    """Lists of one or two groups (of four groups, the last not full, or of single sources)."""
    n = 300
    rng = np.random.default_rng(nsrc)
    edges = [(v, int(u)) for v in range(n) for u in rng.integers(0, n, 1 + rng.poisson(3))]
    edges += [(v, int(u)) for v in range(3) for u in rng.integers(0, n, 700 * (v + 1))]
    rp, col = inputs.csr_from_edges(n, edges)
    deg = np.diff(rp)
    g = fora.Graph(rp, col)
    g.build_index(fora.Params.make(k=1, delta=1e-3, pf=1e-3, rmax=RMAX, seed=SEED))
    rmax, C, _ = g.index_info()
    off, dest = oracle.walk_index(rp, col, 0.2, C, rmax, SEED)
    walks = rng.choice([0.0, 1, 9, 1024, 1025, 2049, 1e9], (nsrc, n))
    r = np.minimum(walks / C, rmax * deg)
    r[0] = rmax * deg
    res = rng.random((nsrc, n))
    p = fora.Params.make(k=1, delta=1e-3, pf=1e-3, rmax=RMAX, seed=1, flags=fora.FORA_USE_INDEX)
    sources = rng.integers(0, n, nsrc).astype(np.int32)
    g.tune("index_groups", groups)
    _, _, _, out = _debug(g, sources, p, given=(res, r))
    for i in range(nsrc):
        cnt, acc, _ = oracle.walk_phase_indexed(n, C, r[i], off, dest)
        np.testing.assert_array_equal(out["count"][i], cnt)
        np.testing.assert_array_equal(out["acc"][i], acc)
    g.close()


def test_indexed_walks_of_a_node_with_almost_2_32_walks():
    """One node with a self-loop holds all walks: the last chunk of them ends at 2^32."""
    lo, hi = 1e-6, 1e-2
    for _ in range(200):  # walks fall with eps
        eps = 0.5 * (lo + hi)
        lo, hi = (eps, hi) if oracle.walk_scale(eps, 1.0, 1e-3) > 2**32 - 512 else (lo, eps)
    p = fora.Params.make(k=1, eps=hi, delta=1.0, pf=1e-3, rmax=1.0, seed=SEED)
    g = fora.Graph(np.array([0, 1]), np.array([0]))
    walks = int(np.ceil(g.resolve(p)[1]))
    assert 2**32 - 1024 < walks < 2**32 and walks % 1024
    if torch.cuda.mem_get_info()[0] < 6 * walks:
        pytest.skip("the index takes 17 GB")
    g.build_index(p)
    p.flags = fora.FORA_USE_INDEX
    _, _, st, out = _debug(g, [0], p)
    assert st[0].walks == walks
    # the residue 1 as `walks` walks of weight rint(2^63 / walks), all of them ending at the node
    weight = int(np.rint(np.float64(1.0) / np.float64(walks) * np.float64(2.0**63)))
    assert int(out["acc"][0, 0]) == walks * weight
    assert int(out["count"][0, 0]) == walks
    g.close()
