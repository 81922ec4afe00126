"""The push as a sequence of launches, and beside other work of the device: results of a launch a
round equal the oracle's, and neither a kernel that holds an SM nor another call's long push
holds a query back."""
import threading
import time

import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import ATOL_PUSH, _built, run_debug  # noqa: E402,F401

ASYNC = 0x2
COSTS = (4.63e-9, 0.0, 3.82e-8)


# 1 and 2 sources: side by side 1; 3, 9: groups of 4; 90: whole units of the take
@pytest.mark.parametrize("nsrc", [1, 2, 3, 9, 90])
def test_a_launch_a_round_matches_oracle(nsrc):
    rp, col = inputs.rmat_csr(14, 8, 1)
    g = fora.Graph(rp, col)
    n = len(rp) - 1
    sources = inputs.uniform_sources(n, nsrc, 5 + nsrc)
    p = fora.Params.make(k=10)
    g.tune("push_slice", 0)
    assert g.tuning("push_slice") == 0
    _, _, st, out = run_debug(g, sources, p)
    rmax = g.resolve(p)[0]
    for i in sorted({0, nsrc // 2, nsrc - 1}):
        res, r, pst = oracle.forward_push(rp, col, int(sources[i]), 0.2, rmax)
        np.testing.assert_allclose(out["reserve"][i], res, rtol=0, atol=ATOL_PUSH)
        np.testing.assert_allclose(out["residue"][i], r, rtol=0, atol=ATOL_PUSH)
        assert (st[i].pushes, st[i].edge_pushes, st[i].push_rounds) == \
            (pst.pushes, pst.edge_pushes, pst.rounds)
    # without host stops: enqueued at once (64 launches of a round, then one of the rest)
    ids, vals, _ = g.ssppr_batch(sources, p)
    pa = fora.Params.make(k=10, flags=ASYNC)
    got = [torch.empty((nsrc, 10), dtype=t, device="cuda") for t in (torch.int32, torch.float64)]
    g.ssppr_batch(sources, pa, out_ids=got[0], out_vals=got[1], stats=False)
    torch.cuda.synchronize()
    np.testing.assert_allclose(got[1].cpu().numpy(), vals, rtol=0, atol=ATOL_PUSH)
    # the balanced push
    _, vals0, st0 = g.ssppr_batch_balanced(sources, p, COSTS)
    g.tune("push_slice", 1000000)
    _, vals1, st1 = g.ssppr_batch_balanced(sources, p, COSTS)
    np.testing.assert_allclose(vals0, vals1, rtol=0, atol=ATOL_PUSH)
    assert [s.push_rounds for s in st0] == [s.push_rounds for s in st1]
    for value in (-1, 1000001):
        with pytest.raises(fora.FORAError):
            g.tune("push_slice", value)
    g.close()


def test_requests_join_a_push_of_a_launch_a_round():
    g = fora.Graph(*inputs.rmat_csr(16, 16, 5))
    g.tune("push_slice", 0)
    server = fora.Server([g], lanes_per_graph=1, max_batch=16, memory_budget_bytes=2 << 30,
                         batch_window_ms=0.0, admit_during_push=True)
    try:
        p = fora.Params.make(k=50, seed=21)
        src = inputs.uniform_sources(g.n, 60, 2024)
        tickets = []
        for s in src:
            tickets.append(server.submit(0, int(s), p))
            time.sleep(0.0002)
        results = [server.wait(t, 50) for t in tickets]
        assert server.stats()["joined"] >= 1
        for s, (ids, vals, info) in zip(src, results):
            _, vals1, st1 = g.ssppr(int(s), p)
            np.testing.assert_allclose(vals, vals1, rtol=0, atol=ATOL_PUSH)
            assert info.stats.walks == st1.walks and info.stats.pushes == st1.pushes
    finally:
        server.close()
        g.close()


def test_a_kernel_that_holds_an_SM_does_not_hold_a_query():
    """A query whose push uses every SM, beside another stream's kernel of about 0.2 s (one block):
    it takes some milliseconds alone."""
    g = fora.Graph(*inputs.rmat_csr(20, 16, 2))
    p = fora.Params.make(k=50)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):
        _, alone, st0 = g.ssppr(3, p, stream=mine)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(other):
        torch.cuda._sleep(400_000_000)
        done.record()
    t0 = time.perf_counter()
    _, vals, st1 = g.ssppr(3, p, stream=mine)
    t1 = time.perf_counter()
    assert not done.query(), f"the other kernel ended first ({t1 - t0:.3f} s)"
    # a push without all its blocks
    np.testing.assert_allclose(vals, alone, rtol=0, atol=ATOL_PUSH)
    assert (st1.pushes, st1.push_rounds, st1.walks) == (st0.pushes, st0.push_rounds, st0.walks)
    torch.cuda.synchronize()
    g.close()


@pytest.mark.parametrize("nsrc,balanced", [(2, False), (64, False), (40, True)])
def test_pushes_beside_a_kernel_that_holds_an_SM(nsrc, balanced):
    """Whole and cut pushes whose blocks do not all find room: rounds as kernels of their own."""
    g = fora.Graph(*inputs.rmat_csr(18, 16, 2))
    g.tune("push_slice", 300)
    p = fora.Params.make(k=50)
    sources = inputs.uniform_sources(g.n, nsrc, 5)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()

    def run():
        if balanced:
            return g.ssppr_batch_balanced(sources, p, COSTS, stream=mine)
        return g.ssppr_batch(sources, p, stream=mine)

    _, alone, st0 = run()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(other):
        torch.cuda._sleep(800_000_000)  # about 0.4 s
        done.record()
    _, vals, st1 = run()
    held = not done.query()
    torch.cuda.synchronize()
    np.testing.assert_allclose(vals, alone, rtol=0, atol=ATOL_PUSH)
    for a, b in zip(st0, st1):
        assert (a.pushes, a.edge_pushes, a.walks) == (b.pushes, b.edge_pushes, b.walks)
        assert a.push_rounds == b.push_rounds
    assert held
    g.close()


def test_requests_beside_a_kernel_that_holds_an_SM():
    g = fora.Graph(*inputs.rmat_csr(18, 16, 2))
    server = fora.Server([g], lanes_per_graph=1, max_batch=32, memory_budget_bytes=4 << 30,
                         batch_window_ms=0.0, admit_during_push=True)
    try:
        p = fora.Params.make(k=50, seed=21)
        src = inputs.uniform_sources(g.n, 40, 2024)
        server.wait(server.submit(0, int(src[0]), p), 50)
        other = torch.cuda.Stream()
        with torch.cuda.stream(other):
            torch.cuda._sleep(800_000_000)
        tickets = []
        for s in src:
            tickets.append(server.submit(0, int(s), p))
            time.sleep(0.0002)
        results = [server.wait(t, 50) for t in tickets]
        torch.cuda.synchronize()
        for s, (ids, vals, info) in zip(src, results):
            _, vals1, st1 = g.ssppr(int(s), p)
            np.testing.assert_allclose(vals, vals1, rtol=0, atol=ATOL_PUSH)
            assert info.stats.walks == st1.walks and info.stats.pushes == st1.pushes
    finally:
        server.close()
        g.close()


def test_a_long_push_does_not_hold_queries_of_another_thread():
    """Single queries beside balanced batches, whose push is most of the call: they wait for a
    slice of it at a time, not for the whole push."""
    big, small = fora.Graph(*inputs.rmat_csr(20, 16, 2)), fora.Graph(*inputs.rmat_csr(16, 16, 5))
    p, ps = fora.Params.make(k=500), fora.Params.make(k=50)
    sources = inputs.uniform_sources(big.n, 64, 7)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = [torch.empty((64, 500), dtype=t, device="cuda") for t in (torch.int32, torch.float64)]

    def batch():
        st = big.ssppr_batch_balanced(sources, p, COSTS, out_ids=out[0], out_vals=out[1],
                                      stream=a)[2]
        return st[0].ms_push

    batch()
    push_ms = batch()
    alone = [small.ssppr(i, ps, stream=b) for i in range(40)]
    vals0 = out[1].clone()
    stop, differ = threading.Event(), []

    def load():
        while not stop.is_set():
            batch()
            differ.append(float((out[1] - vals0).abs().max()))

    th = threading.Thread(target=load)
    th.start()
    time.sleep(0.2)
    waits = []
    try:
        for i in range(40):
            t0 = time.perf_counter()
            _, vals, st = small.ssppr(i, ps, stream=b)
            waits.append((time.perf_counter() - t0) * 1e3)
            np.testing.assert_allclose(vals, alone[i][1], rtol=0, atol=ATOL_PUSH)
            assert (st.pushes, st.walks) == (alone[i][2].pushes, alone[i][2].walks)
            time.sleep(0.003)
    finally:
        stop.set()
        th.join()
    assert max(differ) <= ATOL_PUSH
    assert np.median(waits) < push_ms / 3, (np.median(waits), push_ms)
    big.close()
    small.close()
