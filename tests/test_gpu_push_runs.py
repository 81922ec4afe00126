"""Copies of a multi-edge, which the balanced push of a large batch adds at once: runs within a slice
of 32 edges, across slices and across a hub's chunks of 256, against batches of two sources, which
add every copy."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import ATOL_PUSH, _built  # noqa: E402,F401


@pytest.mark.parametrize("copies", [[1], [1, 2, 3], [31, 32, 33, 70], [1, 600]])
def test_copies_of_an_edge_are_added_with_multiplicity(copies):
    rng = np.random.default_rng(len(copies))
    rp, col = inputs.rmat_csr(14, 2, 9)
    times = rng.choice(copies, len(col))
    n = len(rp) - 1
    deg = np.zeros(n, dtype=np.int64)
    np.add.at(deg, np.repeat(np.arange(n), np.diff(rp)), times)
    g = fora.Graph(np.concatenate([[0], np.cumsum(deg)]), np.repeat(col, times))
    sources = inputs.uniform_sources(n, 160, 4)  # enough for whole units of the take
    p = fora.Params.make(k=40)
    cost = (4.63e-9, 0.0, 3.82e-8)
    _, vals, st = g.ssppr_batch_balanced(sources, p, cost)
    for i in (0, 33, 80, 158):
        _, vals2, st2 = g.ssppr_batch_balanced(sources[i:i + 2], p, cost)
        for k in range(2):
            assert (st[i + k].pushes, st[i + k].edge_pushes, st[i + k].walks) == \
                (st2[k].pushes, st2[k].edge_pushes, st2[k].walks)
            np.testing.assert_allclose(vals[i + k], vals2[k], rtol=0, atol=ATOL_PUSH)
    g.close()
