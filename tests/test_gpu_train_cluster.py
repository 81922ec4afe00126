"""Training by an epoch per launch (one cluster, a tile of 64 samples per block) and, for batches
of more than 512 samples, step by step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1908_10583_gb300 as fora  # noqa: E402
from tests.test_gpu_parity import _built  # noqa: E402,F401

LR = 2e-3


def order(n, seed):
    """The seeded shuffle of an epoch: sample order[i] is the i-th."""
    state, perm, mask = seed, list(range(n)), 2 ** 64 - 1
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    return np.array(perm)


def data(n, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(0, 2, (n, 16)).astype(np.float32), rng.normal(0, 1, n).astype(np.float32)


# tiles of 64: one not full, full, one more sample; 8 tiles (the largest cluster), and beyond it
@pytest.mark.parametrize("n", [1, 63, 64, 65, 256, 449, 512, 513, 700])
def test_one_step_is_adam_on_the_gradient(n):
    x, t = data(n, n)
    m, h = fora.Model(5), fora.Model(5)
    p0, _ = m.get()
    m.train(x, t, epochs=1, batch=n, lr=LR, seed=9)
    p1, norm = m.get()
    h.set(p0, norm)
    at = order(n, 9)
    g, _ = h.gradient(x[at], t[at])
    g = g.astype(np.float64)
    b1, b2 = np.float64(np.float32(0.9)), np.float64(np.float32(0.999))
    # step 1: m / c1 = g and v / c2 = g^2 up to the roundings of the moments, the corrections
    # (1 - b2 keeps 14 of its 24 bits, in both places the same value) and the quotient: each of
    # about ten operations by 2^-24, then the subtraction from the master by 2^-24 of it
    mh = (1 - b1) * g / (1 - b1)
    vh = (1 - b2) * g * g / (1 - b2)
    want = p0 - np.float32(LR) * mh / (np.sqrt(vh) + 1e-8)
    assert np.all(np.abs(p1 - want) <= 2.0 ** -24 * (16 * LR + np.abs(p0)))


# steps of an epoch in one call against a call each: the moments, the next step's inputs and the
# parameters that the blocks exchange, with a last batch of half the size
@pytest.mark.parametrize("batch", [2, 62, 128, 130, 320, 512])
def test_an_epoch_equals_its_steps(batch):
    rng = np.random.default_rng(batch)
    half = rng.integers(-8, 9, (batch // 2, 16)).astype(np.float32)

    def part(copies):  # column-wise shuffles: the same mean and variance, exactly
        rows = np.concatenate([half] * copies)
        return np.stack([rng.permutation(rows[:, i]) for i in range(16)], axis=1)

    parts = [part(2), part(2), part(2), part(1)]
    targets = [rng.normal(0, 1, len(q)).astype(np.float32) for q in parts]
    one, steps = fora.Model(3), fora.Model(3)
    x, t = np.concatenate(parts), np.concatenate(targets)
    at = order(len(x), 4)
    xs, ts = np.empty_like(x), np.empty_like(t)
    xs[at], ts[at] = x, t  # so that the shuffle gives the parts one after the other
    one.train(xs, ts, epochs=1, batch=batch, lr=LR, seed=4)
    for q, u in zip(parts, targets):
        at = order(len(q), 4)
        qs, us = np.empty_like(q), np.empty_like(u)
        qs[at], us[at] = q, u
        steps.train(qs, us, epochs=1, batch=batch, lr=LR, seed=4)
    (pa, na), (pb, nb) = one.get(), steps.get()
    np.testing.assert_array_equal(na, nb)
    np.testing.assert_array_equal(pa, pb)
