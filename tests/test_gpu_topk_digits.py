"""The top-k select on rows that take each of its routes: the k-th value inside the bins of the
first digit, below them, above them, and among more equal values than the final sort holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import _built  # noqa: E402,F401


def noalloc(est, k):
    nrows, n = est.shape
    ids = torch.empty((nrows, k), dtype=torch.int32, device="cuda")
    vals = torch.empty((nrows, k), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert fora.load().fora_topk_noalloc(est.data_ptr(), n, nrows, k, ids.data_ptr(),
                                         vals.data_ptr(), None) == 0
    return ids, vals


def expect(est, k):
    order = np.lexsort((np.arange(est.shape[1])[None, :].repeat(len(est), 0), -est), axis=1)[:, :k]
    return order, np.take_along_axis(est, order, 1)


def rows(n, rng):
    spread = rng.random(n) ** 8
    tiny = rng.random(n) * 2.0 ** -70              # below the bins
    sparse = np.where(rng.random(n) < 0.003, rng.random(n), 0.0)  # zeros beyond a few
    huge = rng.random(n) * 2.0 ** 40               # above them
    equal = np.full(n, 0.125)                      # ties only
    edges = 2.0 ** rng.integers(-66, 4, n)         # the bins' edges, many equal
    close = 0.5 + rng.integers(0, 1 << 20, n) * 2.0 ** -40  # one bin of the first digit
    return np.stack([spread, tiny, sparse, huge, equal, edges, close])


# elements around a part of 4096 and a warp's load; k = 1, around the candidates the sort takes
# (8192 at most) and n
@pytest.mark.parametrize("n,k", [(1, 1), (31, 31), (1000, 17), (4095, 4095), (4097, 500),
                                 (20011, 500), (70001, 1), (70001, 4096), (1 << 20, 1000)])
def test_every_route_of_the_select(n, k):
    est = rows(n, np.random.default_rng(n + k))
    ids, vals = expect(est, k)
    d = torch.tensor(est).cuda()
    for sel in (fora.topk, noalloc):
        got_ids, got_vals = sel(d, k)
        np.testing.assert_array_equal(np.asarray(got_ids.cpu()), ids)
        np.testing.assert_array_equal(np.asarray(got_vals.cpu()), vals)


def test_more_rows_than_one_wave():
    rng = np.random.default_rng(4)
    est = np.concatenate([rows(9001, rng) for _ in range(60)])  # 420 rows
    ids, vals = expect(est, 100)
    got_ids, got_vals = fora.topk(torch.tensor(est).cuda(), 100)
    np.testing.assert_array_equal(np.asarray(got_ids.cpu()), ids)
    np.testing.assert_array_equal(np.asarray(got_vals.cpu()), vals)


# few long rows (a part of each for every block of the device), and rows of one part
@pytest.mark.parametrize("nrows,n,k", [(1, 3000001, 500), (2, 1 << 21, 4096), (3, 4096, 4096),
                                       (33, 8191, 100)])
def test_levels_over_the_whole_grid(nrows, n, k):
    rng = np.random.default_rng(nrows)
    for make in range(7):
        est = np.stack([rows(n, rng)[(make + i) % 7] for i in range(nrows)])
        ids, vals = expect(est, k)
        for _ in range(2):
            got_ids, got_vals = fora.topk(torch.tensor(est).cuda(), k)
            np.testing.assert_array_equal(np.asarray(got_ids.cpu()), ids)
            np.testing.assert_array_equal(np.asarray(got_vals.cpu()), vals)


def test_a_long_row_of_few_values_above_zero_takes_no_longer_per_level_than_a_pass():
    """The eight levels of a row whose k-th value is 0, against the two passes of a plain one: at
    most 8 + 2 passes and their hand-overs."""
    n = 1 << 25
    zeros = torch.zeros((1, n), dtype=torch.float64, device="cuda")
    zeros[0, ::n // 100] = 0.25
    plain = torch.rand((1, n), dtype=torch.float64, device="cuda") ** 8

    def ms(est):
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fora.topk(est, 500)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    ms(plain)
    assert ms(zeros) < 8 * ms(plain)
