"""The work that a user has this library do, as cases with their inputs.

A case is a query of one kind (one source, a batch, top-k FORA, a walk index, a server),
the top-k select on its own, or the training of the r_max network, each through the entry
points of ``paper_1908_10583_gb300``.  Graphs are seeded R-MAT graphs with the quadrant
probabilities of ``inputs`` (0.57, 0.19, 0.19, 0.05), or graphs of Poisson out-degrees and
uniform targets, which have no node of high in-degree; they are generated on the GPU.
``exact`` evaluates the same query in plain torch: the push and the estimate in FP64, the
walks on the same Philox4x32-10 words.
"""
import math
import os

import numpy as np
import torch

import paper_1908_10583_gb300 as fora

ALPHA = 0.2
MODEL = os.path.join(os.path.dirname(fora.__file__), "models", "rmax_rmat20_deg16.npz")
COUNTERS = ("pushes", "edge_pushes", "residual_nodes", "walks", "walk_steps", "push_rounds")
# Costs of one edge push, one node push and one walk for the balanced push of Alg. 3 (ms, as
# the training report of the committed model gives them).
BALANCE = (4.63e-9, 0.0, 3.82e-8)


def listed():
    return [
        # One query on the small test graph: a caller who waits for each answer; host and
        # launch latency dominate.
        dict(name="one, 2^14 nodes", kind="one", graph="rmat", n=1 << 14, deg=8.0, k=50, eps=0.5),
        # One query at a time on the benchmark's graph (plain FORA).
        dict(name="one, 2^20 nodes", kind="one", graph="rmat", n=1 << 20, deg=16.0, k=500, eps=0.5),
        # The benchmark: 256 queries in one launch, r_max from the committed network.
        dict(name="learned batch, 256 x 2^20", kind="batch", mode="learned", graph="rmat", n=1 << 20,
             deg=16.0, nsrc=256, k=500, eps=0.5),
        # A batch with the rule's r_max on a mid-size graph (the serving graph of 2^18 nodes).
        dict(name="rule batch, 64 x 2^18", kind="batch", mode="rule", graph="rmat", n=1 << 18, deg=16.0,
             nsrc=64, k=500, eps=0.5),
        # Ragged sizes, a tighter error bound, and the zero-hop pruning of Section 4.1.
        dict(name="zero-hop batch, 37 x 100003", kind="batch", mode="zero_hop", graph="rmat", n=100003,
             deg=11.0, nsrc=37, k=100, eps=0.3),
        # A graph without hubs (no in-degree far above the mean), an odd batch.
        dict(name="uniform batch, 100 x 200003", kind="batch", mode="rule", graph="uniform", n=200003,
             deg=10.0, nsrc=100, k=200, eps=0.5),
        # FORA+ (Section 3.3): walks taken from a stored index.
        dict(name="index batch, 64 x 2^20", kind="batch", mode="index", graph="rmat", n=1 << 20,
             deg=16.0, nsrc=64, k=500, eps=0.5),
        # The balanced push of Section 4.2, whose threshold falls until its cost rule stops it.
        dict(name="balanced batch, 32 x 2^18", kind="batch", mode="balanced", graph="rmat", n=1 << 18,
             deg=16.0, nsrc=32, k=500, eps=0.5),
        # Top-k FORA (Alg. 5): rounds of queries with falling delta.
        dict(name="top-k FORA, 32 x 2^16", kind="topk_fora", graph="rmat", n=1 << 16, deg=16.0, nsrc=32,
             k=100, eps=0.5),
        # The select alone, on score rows that a caller holds.
        dict(name="select, 24 x 1000003", kind="select", n=1000003, nsrc=24, k=500),
        # A burst of requests to the server, waited for in order.
        dict(name="serve, 24 requests, 2^16", kind="serve", graph="rmat", n=1 << 16, deg=16.0, nsrc=24,
             k=50, eps=0.5),
        # Training the r_max network (forward, backward and Adam on the device).
        dict(name="train r_max, 10000 samples", kind="train", nsrc=10000, batch=256, epochs=2),
    ]


def draw(rng):
    kind = rng.choice(["one", "batch", "batch", "batch", "batch", "topk_fora", "select", "serve", "train"])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "train":
        return dict(kind=kind, nsrc=spread(300, 20000), batch=rng.choice([64, 100, 256, 512]),
                    epochs=rng.randint(1, 3))
    if kind == "select":
        n = spread(5000, 2000000)
        return dict(kind=kind, n=n, nsrc=max(1, min(spread(1, 64), (1 << 26) // n)),
                    k=min(spread(1, 2000), n))
    case = dict(kind=kind, graph=rng.choice(["rmat", "rmat", "uniform"]))
    deg = rng.uniform(4.0, 24.0)
    n = spread(4000, min(1 << 20, int((1 << 24) / deg)))
    case.update(n=n | rng.randint(0, 1), deg=round(deg, 1), k=spread(1, 800), eps=rng.choice([0.5, 0.5, 0.3]))
    if kind == "batch":
        case.update(mode=rng.choice(["rule", "rule", "learned", "constant", "zero_hop", "index", "balanced"]),
                    nsrc=spread(2, 256))
    elif kind != "one":
        case["nsrc"] = spread(4, 48)
        case["k"] = min(case["k"], 200)
    most = work(listed()[2])["bytes"] / 4
    while case.get("nsrc", 1) > 1 and work(case)["bytes"] > most:
        case["nsrc"] = (case["nsrc"] + 1) // 2
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _csr(n, src, dst, gen):
    """CSR with sorted rows; a node without out-edges gets one edge to a uniform node."""
    none = torch.nonzero(torch.bincount(src, minlength=n) == 0).flatten()
    src = torch.cat([src, none])
    dst = torch.cat([dst, torch.randint(0, n, (len(none),), generator=gen, device="cuda")])
    key = torch.sort(src * n + dst).values
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return row, (key % n).to(torch.int32)


def _graph(case, seed):
    """(row_ptr, col) on the GPU: row_ptr int64 [n + 1], col int32 [m]."""
    n, gen = case["n"], _gen(seed, 0)
    if case["graph"] == "uniform":
        deg = 1 + torch.poisson(torch.full((n,), case["deg"] - 1, device="cuda"), generator=gen).long()
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
        return _csr(n, src, torch.randint(0, n, (len(src),), generator=gen, device="cuda"), gen)
    a, b, c = 0.57, 0.19, 0.19
    scale, m = max(1, (n - 1).bit_length()), int(n * case["deg"])
    src = torch.zeros(m, dtype=torch.int64, device="cuda")
    dst = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        u = torch.rand(m, generator=gen, device="cuda")
        src = src * 2 + (u >= a + b)
        dst = dst * 2 + (((u >= a) & (u < a + b)) | (u >= a + b + c))
    label = torch.randperm(n, generator=gen, device="cuda")
    return _csr(n, label[(src * n) >> scale], label[(dst * n) >> scale], gen)


def _sources(case, seed):
    return np.random.RandomState(seed % (1 << 31)).randint(0, case["n"], case.get("nsrc", 1)).astype(np.int32)


def _params(case, seed):
    mode = case.get("mode")
    flags = {"zero_hop": fora.FORA_ZERO_HOP, "index": fora.FORA_USE_INDEX}.get(mode, 0)
    return fora.Params.make(alpha=ALPHA, eps=case["eps"], k=min(case["k"], case["n"]), flags=flags,
                            seed=0x5EED + int(seed))


def _scores(case, seed):
    """Score rows as estimates are: many zeros and equal values, the others over many binades."""
    gen = _gen(seed, 1)
    u = torch.rand((case["nsrc"], case["n"]), generator=gen, device="cuda", dtype=torch.float64)
    v = 1e-9 / (u + 1e-7)
    v = torch.where(u > 0.6, torch.floor(v * 2.0 ** 31) * 2.0 ** -31, v)
    return torch.where(u > 0.9, torch.zeros_like(v), v)


def _samples(case, seed):
    """Features and log2 multipliers of the r_max network's training set."""
    r = np.random.RandomState(seed % (1 << 31))
    x = np.zeros((case["nsrc"], 16), dtype=np.float32)
    base = r.exponential(1.5, case["nsrc"])
    for i in range(6):
        x[:, i] = np.log1p(base * (3.0 + 2.0 * i)) + 0.3 * r.standard_normal(case["nsrc"])
    x[:, 6], x[:, 7] = -1.06, 2.8
    t = -1.44 + 0.2 * np.tanh(x[:, 0] - x[:, 2]) + 0.05 * r.standard_normal(case["nsrc"])
    return x, t.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "select":
        return dict(case=case, est=_scores(case, seed))
    if kind == "train":
        x, t = _samples(case, seed)
        return dict(case=case, x=x, t=t, seed=int(seed) % 1000)
    row, col = _graph(case, seed)
    graph = fora.Graph(row.cpu().numpy(), col.cpu().numpy())
    params = _params(case, seed)
    state = dict(case=case, graph=graph, params=params, sources=_sources(case, seed))
    if kind == "batch":
        k = params.k
        state["ids"] = torch.empty((case["nsrc"], k), dtype=torch.int32, device="cuda")
        state["vals"] = torch.empty((case["nsrc"], k), dtype=torch.float64, device="cuda")
        if case["mode"] == "learned":
            state["model"] = fora.Model.load_file(MODEL)
        elif case["mode"] == "constant":
            state["rmax"] = np.full(case["nsrc"], 0.354 * graph.resolve(params)[0])
        elif case["mode"] == "index":
            graph.build_index(params)
    elif kind == "serve":
        state["server"] = fora.Server([graph], lanes_per_graph=2, max_batch=32,
                                      memory_budget_bytes=20 << 30, batch_window_ms=0.5)
    return state


# ---------------------------------------------------------------- one pass

def _counters(stats):
    return np.array([[getattr(s, f) for f in COUNTERS] for s in stats], dtype=np.int64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "select":
        ids, vals = fora.topk(state["est"], case["k"])
        return dict(ids=ids, vals=vals)
    if kind == "train":
        model = fora.Model(state["seed"])
        loss = model.train(state["x"], state["t"], epochs=case["epochs"], batch=case["batch"], lr=2e-3,
                           seed=state["seed"])
        weights, norm = model.get()
        return dict(weights=weights, norm=norm, loss=loss)
    g, p, src = state["graph"], state["params"], state["sources"]
    if kind == "one":
        ids, vals, stats = g.ssppr(int(src[0]), p)
        return dict(ids=ids, vals=vals, counters=_counters([stats]))
    if kind == "topk_fora":
        ids, vals, stats, rounds = g.topk_fora(src, p)
        return dict(ids=ids, vals=vals, rounds=rounds.astype(np.int64), counters=_counters(stats))
    if kind == "serve":
        tickets = [state["server"].submit(0, int(s), p) for s in src]
        got = [state["server"].wait(t, p.k) for t in tickets]
        return dict(ids=np.stack([x[0] for x in got]), vals=np.stack([x[1] for x in got]),
                    counters=_counters([x[2].stats for x in got]))
    mode, out = case["mode"], dict(out_ids=state["ids"], out_vals=state["vals"])
    if mode == "learned":
        ids, vals, stats = g.ssppr_batch_learned(src, p, state["model"], **out)
    elif mode == "constant":
        ids, vals, stats = g.ssppr_batch_rmax(src, state["rmax"], p, **out)
    elif mode == "balanced":
        ids, vals, stats = g.ssppr_batch_balanced(src, p, BALANCE, **out)
    else:
        ids, vals, stats = g.ssppr_batch(src, p, **out)
    return dict(ids=ids, vals=vals, counters=_counters(stats))


def work(case):
    """What a pass cannot do without.

    Queries, by the cost model of Section 3.2: 1 / r_max edge pushes per source (a target of
    4 bytes, a read-modify-write of an FP64 residue, one multiply-add) and half of
    m r_max C walks (the bound counts a full residue at every node) of (1 - alpha) / alpha
    moves (a target of 4 bytes) with a read-modify-write of 8 bytes at the end; the graph
    read once; the estimate of every node written once."""
    if case["kind"] == "select":
        return dict(bytes=8.0 * case["nsrc"] * case["n"] + 12.0 * case["nsrc"] * case["k"], flops=0.0)
    if case["kind"] == "train":
        samples = case["nsrc"] * case["epochs"]
        return dict(bytes=68.0 * samples + 4.0 * 5313 * 7, flops=3 * 2 * 5200.0 * samples)
    n, m, nsrc, eps = case["n"], case["n"] * case["deg"], case.get("nsrc", 1), case["eps"]
    c = (2 * eps / 3 + 2) * math.log(2 * n) * n / (eps * eps)
    rmax = min(eps / math.sqrt(m) * math.sqrt(1 / n / ((2 * eps / 3 + 2) * math.log(2 * n))), 1.0)
    if m * rmax > 1:
        rmax = 1 / c
    if case.get("mode") in ("learned", "constant", "balanced"):
        rmax *= 0.354
    walks = 0.5 * m * rmax * c
    moves = 0.0 if case.get("mode") == "index" else walks * (1 - ALPHA) / ALPHA
    per_source = 20 / rmax + 4 * moves + 20 * walks + 8 * n + 12 * case["k"]
    return dict(bytes=4.0 * (m + n) + nsrc * per_source, flops=nsrc * (2 / rmax + walks))


# ---------------------------------------------------------------- the same in plain torch

M32 = 0xFFFFFFFF


def _mulhilo(a, b):
    """High and low words of the product of 32-bit words held in int64 tensors."""
    hi = (((a >> 16) * b) + (((a & 0xFFFF) * b) >> 16)) >> 16
    return hi & M32, (a * b) & M32


def _philox(c, key):
    k0, k1 = key & M32, (key >> 32) & M32
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _walk_ends(row, deg, col, v, j, source, key, zero_hop):
    """Ends of walks j from nodes v, whose words are the Philox blocks (c, j, v, source)."""
    stop_below = int(math.floor(ALPHA * 4294967296.0))
    end = torch.empty_like(v)
    at, x = torch.arange(len(v), device="cuda"), v.clone()
    moving = torch.full_like(v, 1 if zero_hop else 0, dtype=torch.bool)
    block = 0
    while len(at):
        words = _philox((torch.full_like(v, block), j, v, torch.full_like(v, source)), key)
        live = torch.ones_like(moving)
        for w in words:
            stop = live & ~moving & (w < stop_below)
            d = deg[x]
            hi, lo = _mulhilo(w, d)
            step = live & moving & ((lo >= d) | (lo >= (4294967296 - d) % d))
            to = col[torch.clamp(row[x] + hi, max=len(col) - 1)].long()
            moving = torch.where(live, torch.where(moving, ~step, ~stop), moving)
            x = torch.where(step, to, x)
            live = live & ~stop
        end[at[~live]] = x[~live]
        at, x, moving, v, j = at[live], x[live], moving[live], v[live], j[live]
        block += 1
    return end


def _push(row, deg, col, src_of, s, rmax, scale, balanced):
    """Reserve and residue of Alg. 1 in synchronous rounds, or of Alg. 3."""
    n = len(deg)
    res, r = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    r[s] = 1.0
    d = deg.double()
    theta, edges, pushes, moved = 1.0 if balanced else rmax, 0.0, 0.0, 0.0
    while True:
        if balanced and BALANCE[0] * edges + BALANCE[1] * pushes >= (1.0 - moved) * scale * BALANCE[2]:
            return res, r
        front = r > theta * d
        if not bool(front.any()):
            if not balanced:
                return res, r
            theta *= 0.5
            continue
        a = torch.where(front, r, torch.zeros_like(r))
        res += ALPHA * a
        r = torch.where(front, torch.zeros_like(r), r)
        r.index_add_(0, col, ((1.0 - ALPHA) * a / d)[src_of])
        if balanced:
            edges += float(d[front].sum())
            pushes += float(front.sum())
            moved += float((ALPHA * a).sum())


def _estimate(graph, s, eps, delta, pf, key, mode, rmax=None, stream=None):
    """The estimate of every node for source s, and the walks it took."""
    row, col, deg, src_of = graph
    m = len(col)
    c = ((2 * eps / 3 + 2) * math.log(2 / pf)) / (eps * eps * delta)
    if rmax is None:
        rmax = eps / math.sqrt(m) * math.sqrt(delta / ((2 * eps / 3 + 2) * math.log(2 / pf)))
        if m * rmax > 1:
            rmax = 1 / c
    if mode == "constant":
        rmax *= 0.354
    res, r = _push(row, deg, col, src_of, s, rmax, c, mode == "balanced")
    zero_hop = mode == "zero_hop"
    est = res + ALPHA * r if zero_hop else res.clone()
    r = (1.0 - ALPHA) * r if zero_hop else r
    nodes = torch.nonzero(r > 0).flatten()
    omega = torch.ceil(r[nodes] * c).long()
    weight = r[nodes] / omega
    first = torch.cumsum(omega, 0) - omega
    total = int(omega.sum())
    for lo in range(0, total, 1 << 23):
        i = torch.arange(lo, min(lo + (1 << 23), total), device="cuda")
        e = torch.searchsorted(first, i, right=True) - 1
        v = nodes[e]
        end = _walk_ends(row, deg, col, v, i - first[e], s if stream is None else stream, key, zero_hop)
        est.index_add_(0, end, weight[e])
    return est


def _top(est, k):
    return torch.sort(est, descending=True, stable=True).values[:k].cpu().numpy()


def _exact_train(case, seed):
    """The training loop with FP64 sums; parameters and activations rounded to BF16 where the
    network's definition rounds them."""
    x, t = _samples(case, seed)
    seed = int(seed) % 1000
    state = [seed]

    def mix():
        state[0] = (state[0] + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
        z = state[0]
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
        return z ^ (z >> 31)

    def uniform(bound):
        return np.float32(((mix() >> 11) * 2.0 ** -53 * 2.0 - 1.0) * np.float64(np.float32(bound)))

    def bf(v):
        return v.to(torch.bfloat16).double()

    sizes = [(64, 16), (64,), (64, 64), (64,), (64,), (1,)]
    bounds = [math.sqrt(6 / 16), 0, math.sqrt(6 / 64), 0, math.sqrt(6 / 64), 0]
    p = []
    for size, bound in zip(sizes, bounds):
        cnt = int(np.prod(size))
        v = np.array([uniform(bound) for _ in range(cnt)]) if bound else np.zeros(cnt)
        p.append(torch.tensor(v, dtype=torch.float64).reshape(size).cuda())
    x64 = x.astype(np.float64)
    mean = x64.mean(0)
    var = (x64 * x64).mean(0) - mean * mean
    sigma = np.where(var > 1e-12, np.sqrt(np.maximum(var, 0)), 1.0)
    norm = np.concatenate([mean, sigma]).astype(np.float32)
    nt = torch.tensor(norm).cuda()
    xs = bf((torch.tensor(x).cuda() - nt[:16]) / nt[16:])
    ts = torch.tensor(t).cuda().double()
    m1, m2 = [torch.zeros_like(q) for q in p], [torch.zeros_like(q) for q in p]
    state[0], step, losses, n = seed, 0, [], case["nsrc"]
    for _ in range(case["epochs"]):
        perm = np.arange(n)
        for i in range(n - 1, 0, -1):
            j = mix() % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        perm, loss = torch.tensor(perm).cuda(), 0.0
        batch = min(case["batch"], n)
        for lo in range(0, n, batch):
            at = perm[lo:lo + batch]
            w1, b1, w2, b2, w3, b3 = [bf(q.float()) for q in p]
            h0 = xs[at]
            z1 = h0 @ w1.T + b1
            h1 = bf(torch.relu(z1).float())
            z2 = h1 @ w2.T + b2
            h2 = bf(torch.relu(z2).float())
            err = h2 @ w3 + b3 - ts[at]
            loss += float((0.5 * err * err).sum())
            dy = err / len(at)
            d2 = dy[:, None] * w3 * (z2 > 0)
            d1 = (d2 @ w2) * (z1 > 0)
            grads = [d1.T @ h0, d1.sum(0), d2.T @ h1, d2.sum(0), h2.T @ dy, dy.sum().reshape(1)]
            step += 1
            for q, g, u, v in zip(p, grads, m1, m2):
                u.mul_(0.9).add_(0.1 * g)
                v.mul_(0.999).add_(0.001 * g * g)
                q -= 2e-3 * (u / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
        losses.append(loss / n)
    weights = torch.cat([q.flatten() for q in p]).cpu().numpy()
    return dict(weights=weights, norm=norm.astype(np.float64), loss=np.array(losses))


def exact(case, seed):
    kind = case["kind"]
    if kind == "select":
        vals = torch.topk(_scores(case, seed), case["k"], dim=1).values
        return dict(ids=None, vals=vals)
    if kind == "train":
        return _exact_train(case, seed)
    mode = case.get("mode")
    # a query takes about a second per 10^9 bytes of work here; the network's r_max is FP32
    if mode == "learned" or work(case)["bytes"] > 3e10 or case.get("nsrc", 1) * case["n"] * case["deg"] > 3e8:
        return None
    row, col = _graph(case, seed)
    deg = row[1:] - row[:-1]
    col = col.long()
    graph = (row, col, deg, torch.repeat_interleave(torch.arange(case["n"], device="cuda"), deg))
    params, eps, n = _params(case, seed), case["eps"], case["n"]
    key, k, vals = params.seed, params.k, []
    for s in _sources(case, seed):
        if kind != "topk_fora":
            est = _estimate(graph, int(s), eps, 1 / n, 1 / n, key, mode,
                            stream=M32 if mode == "index" else None)
            vals.append(_top(est, k))
            continue
        last = max(0, math.ceil(math.log2(n / k)))
        pf = 1 / n / (n * max(1.0, math.log2(n / k)))
        for i in range(last + 1):
            delta = 1.0 / (k * 2.0 ** i) if i < last else 1.0 / n
            top = _top(_estimate(graph, int(s), eps / 2, delta, pf, key + i, None), k)
            if top[k - 1] >= (1 + eps) * delta:
                break
        vals.append(top)
    vals = np.stack(vals)
    return dict(ids=None, vals=vals[0] if kind == "one" else vals)
