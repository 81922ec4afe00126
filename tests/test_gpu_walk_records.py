"""The walks' own numbering (records of degree class and walk id, nodes without a class, the
places of the walk ends) against the oracle, bit for bit, on graphs at its edges."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import _built, run_debug  # noqa: E402,F401


def staircase(n, rng):
    """Node v has v + 1 out-edges: n distinct degrees."""
    rp = np.concatenate([[0], np.cumsum(np.arange(1, n + 1))]).astype(np.int64)
    col = rng.integers(0, n, int(rp[-1])).astype(np.int32)
    for v in range(n):
        col[rp[v]:rp[v + 1]].sort()
    return rp, col


def regular(n, d, rng):
    rp = (np.arange(n + 1) * d).astype(np.int64)
    return rp, np.sort(rng.integers(0, n, (n, d)), axis=1).ravel().astype(np.int32)


@pytest.mark.parametrize("zero_hop", [False, True])
@pytest.mark.parametrize("shape", ["more degrees than classes", "one degree", "33 nodes", "2 nodes"])
def test_walks_bit_exact_on_graphs_at_the_edges_of_the_numbering(shape, zero_hop):
    rng = np.random.default_rng(11)
    rp, col = {"more degrees than classes": lambda: staircase(1100, rng),  # 77 nodes without
               "one degree": lambda: regular(4096, 3, rng),
               "33 nodes": lambda: staircase(33, rng),
               "2 nodes": lambda: staircase(2, rng)}[shape]()
    n = len(rp) - 1
    g = fora.Graph(rp, col)
    flags = fora.FORA_ZERO_HOP if zero_hop else 0
    # few pushes and many walks: every node is a start and an end of some
    kw = dict(delta=1e-3, pf=1e-3, rmax=2e-4)
    sources = [0, n - 1, n // 2]
    qs = [oracle.ssppr(rp, col, s, k=min(20, n), seed=23, zero_hop=zero_hop, **kw) for s in sources]
    given = (np.stack([q.reserve for q in qs]), np.stack([q.residue for q in qs]))
    p = fora.Params.make(k=min(20, n), seed=23, flags=flags, **kw)
    ids, vals, st, out = run_debug(g, sources, p, given=given)
    for i, q in enumerate(qs):
        np.testing.assert_array_equal(out["count"][i], q.count)
        np.testing.assert_array_equal(out["acc"][i], q.acc)
        np.testing.assert_array_equal(out["estimate"][i], q.est)
        np.testing.assert_array_equal(ids[i], q.ids)
        assert st[i].walk_steps == q.walk.walk_steps
    # the stored walks of an index come back as node ids
    if not zero_hop:
        ip = fora.Params.make(k=min(20, n), seed=5, **dict(kw, rmax=0.05))
        g.build_index(ip)
        off, dest = g.index_export()
        want_off, want_dest = oracle.walk_index(rp, col, 0.2, g.index_info()[1], g.index_info()[0],
                                                5)[:2]
        np.testing.assert_array_equal(off, want_off)
        np.testing.assert_array_equal(dest, want_dest)
    g.close()
