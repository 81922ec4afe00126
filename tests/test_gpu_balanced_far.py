"""The balanced push of a batch whose scans are long enough that a warp's units come from four
places of the list (48 units of 256 residues a warp) against the same sources in batches of two."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import ATOL_PUSH, _built  # noqa: E402,F401


def test_large_balanced_batch_equals_small_ones():
    g = fora.Graph(*inputs.rmat_csr(20, 16, 2))
    sources = inputs.uniform_sources(g.n, 61, 77)
    p = fora.Params.make(eps=0.5, k=50, seed=3)
    cost = (6.6e-9, 0.0, 3.8e-8)
    ids, vals, st = g.ssppr_batch_balanced(sources, p, cost)
    for i in (0, 15, 30, 45, 59):
        _, vals2, st2 = g.ssppr_batch_balanced(sources[i:i + 2], p, cost)
        for k in range(2):
            assert (st[i + k].pushes, st[i + k].edge_pushes, st[i + k].walks) == \
                (st2[k].pushes, st2[k].edge_pushes, st2[k].walks)
            np.testing.assert_allclose(vals[i + k], vals2[k], rtol=0, atol=ATOL_PUSH)
    g.close()
