"""The push's groups of sources (1 or 4 side by side, the last group not full), its small and
large batches, and the copies of the hot nodes' residues, against the oracle."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import ATOL_PUSH, _built, run_debug  # noqa: E402,F401


def check(rp, col, g, sources, p, sample, hot):
    g.tune("spread_hot", hot)
    try:
        _, _, st, out = run_debug(g, sources, p)
    finally:
        g.tune("spread_hot", 1)
    rmax = g.resolve(p)[0]
    for i in sample:
        res, r, pst = oracle.forward_push(rp, col, int(sources[i]), 0.2, rmax)
        np.testing.assert_allclose(out["reserve"][i], res, rtol=0, atol=ATOL_PUSH)
        np.testing.assert_allclose(out["residue"][i], r, rtol=0, atol=ATOL_PUSH)
        assert (st[i].pushes, st[i].edge_pushes, st[i].push_rounds) == \
            (pst.pushes, pst.edge_pushes, pst.rounds)
        assert st[i].residual_nodes == np.count_nonzero(r)


# 2 sources: side by side 1; 3: one group that is not full; 4, 5, 7; 200: a large batch (whole
# units of the take), with rounds of more items than warps
@pytest.mark.parametrize("hot", [0, 1])
@pytest.mark.parametrize("nsrc", [1, 2, 3, 4, 5, 7, 200])
def test_push_of_every_group_width_matches_oracle(nsrc, hot):
    rp, col = inputs.rmat_csr(14, 8, 1)
    g = fora.Graph(rp, col)
    n = len(rp) - 1
    sources = inputs.uniform_sources(n, nsrc, 31 + nsrc)
    sources[-1] = int(np.argmax(np.diff(rp)))  # a hub: its edges go out in chunks
    sample = range(nsrc) if nsrc < 10 else [0, 1, 98, 197, 198, 199]
    check(rp, col, g, sources, fora.Params.make(k=10), sample, hot)
    g.close()


# node counts around the unit of the take (256 residues of a group), and below a warp's load
@pytest.mark.parametrize("n", [1, 7, 63, 65, 256, 257, 1025])
def test_push_on_small_and_ragged_graphs_matches_oracle(n):
    rng = np.random.default_rng(n)
    edges = [(v, int(u)) for v in range(n) for u in rng.integers(0, n, 1 + rng.poisson(4))]
    edges += [(v, 0) for v in range(n)] * (1 + 300 // n)  # node 0 is hot
    rp, col = inputs.csr_from_edges(n, edges)
    g = fora.Graph(rp, col)
    for nsrc in (1, 6):
        sources = rng.integers(0, n, nsrc).astype(np.int32)
        p = fora.Params.make(k=1, delta=1e-3, pf=1e-3, rmax=1e-4)
        for hot in (0, 1):
            check(rp, col, g, sources, p, range(nsrc), hot)
    g.close()
