"""Workloads by which the speed of the library is judged: whole solves, batches,
the single steps of a solve, the candidate graph and the warm-start network,
each through the entry points of paper_2011_08170_gb300 that a program calls.

``listed()`` are the fixed cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare`` makes what a program has in hand before the call, ``run``
makes one pass and returns its outputs, ``work`` counts what a pass cannot do
without, and ``exact`` computes the outputs in 64 bits with plain torch.

Points are integers in [0, 10^6]^2, uniform, or 70 % from 100 Gaussian clusters
(sigma 5,000) and 30 % uniform; candidate graphs are symmetrised k-nearest-
neighbour graphs with k = 8 ... 12.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300.warm_start import load_weights

SIDE = 1_000_000
F = 8          # fractional bits of lambda, the library's default
SWEEPS = 128   # sweeps per GDP phase, the library's default


def listed():
    return [
        # One small instance from host arrays to host results in one call: what a
        # program that solves instances as they arrive waits for.
        dict(name="solve_1k", kind="solve", n=1000, k=10, points="uniform", pricing=1, io="host"),
        # The headline size: points and graph on the device, results left there.
        dict(name="solve_100k", kind="solve", n=100_000, k=10, points="uniform", pricing=1, io="device"),
        # The largest single instance: clustered points, denser candidate graph.
        dict(name="solve_200k_clustered", kind="solve", n=200_000, k=12, points="clustered", pricing=1,
             io="device"),
        # A ragged mid-size instance with the culled pricing scan.
        dict(name="solve_37k_culled", kind="solve", n=37_511, k=9, points="clustered", pricing=2,
             io="device"),
        # Many instances of mixed size at once (training data, replicas): 256 of
        # 1,000 to 20,000 points, half of them clustered.
        dict(name="batch_256", kind="batch", count=256, lo=1000, hi=20_000, k=10),
        # Degree requirements b_v in 1 ... 4 (fractional b-matching), host arrays.
        dict(name="bmatching_30k", kind="bmatching", n=30_011, k=10, points="uniform", bmax=4),
        # The bound with subtour-elimination cuts, two rounds of separation.
        dict(name="subtour_20k", kind="subtour", n=20_000, k=10, points="uniform", rounds=2),
        # One GDP phase to its fixed point (max_iters lifted), the paper's own stop.
        dict(name="gdp_20k_fixpoint", kind="gdp", n=20_011, k=10, points="uniform", sweeps=20_000),
        # One all-pairs pricing scan at the lambda of a GDP phase, pairs to the host.
        dict(name="price_60k", kind="price", n=60_013, k=10, points="uniform", pricing=1),
        # The candidate graph of a large instance, host points to host CSR: what
        # every program calls before f2m_create.
        dict(name="knn_100k", kind="knn", n=100_000, k=10, points="uniform"),
        # Warm-start inference: features of the points on the device, then the network.
        dict(name="warm_start_200k", kind="infer", n=200_000, points="clustered"),
        # Forward and backward of the network on one training step's samples.
        dict(name="mlp_grad_39k", kind="mlp_grad", count=38_912),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "bmatching", "subtour", "gdp", "price",
                       "knn", "infer", "mlp_grad"])
    points = rng.choice(["uniform", "clustered"])
    k = rng.randint(8, 12)
    if kind == "solve":
        return dict(kind=kind, n=_log_int(rng, 1000, 200_000), k=k, points=points,
                    pricing=rng.choice([1, 2]), io=rng.choice(["host", "device"]))
    if kind == "batch":
        lo = _log_int(rng, 1000, 8000)
        return dict(kind=kind, count=_log_int(rng, 4, 200), lo=lo, hi=_log_int(rng, lo, 16_000),
                    k=rng.randint(8, 10))
    if kind == "bmatching":
        return dict(kind=kind, n=_log_int(rng, 2000, 60_000), k=rng.randint(10, 12), points="uniform",
                    bmax=rng.randint(3, 4))
    if kind == "subtour":
        return dict(kind=kind, n=_log_int(rng, 2000, 40_000), k=rng.randint(9, 12), points=points,
                    rounds=rng.randint(1, 2))
    if kind == "gdp":
        n = _log_int(rng, 1000, 200_000)
        return dict(kind=kind, n=n, k=k, points=points,
                    sweeps=_log_int(rng, 64, max(65, min(20_000, 60_000_000 // n))))
    if kind == "price":
        return dict(kind=kind, n=_log_int(rng, 4000, 100_000), k=k, points=points,
                    pricing=rng.choice([1, 2]))
    if kind == "knn":
        return dict(kind=kind, n=_log_int(rng, 1000, 200_000), k=k, points=points)
    if kind == "infer":
        return dict(kind=kind, n=_log_int(rng, 1000, 200_000), points=points)
    return dict(kind=kind, count=_log_int(rng, 1000, 160_000))


# ---- inputs -----------------------------------------------------------------------------


def _points(n, points, gen):
    """int32 [n, 2] host points."""
    uni = n if points == "uniform" else n - int(round(0.7 * n))
    parts = []
    need = n - uni
    centres = gen.integers(0, SIDE + 1, size=(100, 2))
    while need:
        c = centres[gen.integers(0, 100, size=2 * need + 16)]
        p = np.floor(c + gen.normal(0.0, 5000.0, size=c.shape) + 0.5)
        p = p[((p >= 0) & (p <= SIDE)).all(axis=1)][:need]
        parts.append(p.astype(np.int32))
        need -= len(p)
    parts.append(gen.integers(0, SIDE + 1, size=(uni, 2)).astype(np.int32))
    return np.ascontiguousarray(np.concatenate(parts))


def _gen(seed, tag=0):
    return np.random.default_rng([seed, tag])


def _sizes(case):
    """Sizes of a batch's instances, log-uniform in [lo, hi], the same for every seed."""
    gen = np.random.default_rng([case["count"], case["lo"], case["hi"]])
    return np.round(np.exp(gen.uniform(math.log(case["lo"]), math.log(case["hi"]),
                                       size=case["count"]))).astype(int)


def _room(n, k):
    """Entries a result's arrays have room for: a k-NN graph's 2 n k at most, and
    those that pricing adds."""
    return 2 * n * k + 2 * n


def _out(n, k, device):
    """Result arrays that a program keeps from one solve to the next: row_ptr, col,
    x2, cost, lambda.  The entries in use lead; what follows them stays zero."""
    make = (lambda c, t: torch.zeros(c, dtype=t, device="cuda")) if device else \
        (lambda c, t: torch.zeros(c, dtype=t).numpy())
    m = _room(n, k)
    return (make(n + 1, torch.int32), make(m, torch.int32), make(m, torch.uint8), make(m, torch.int32),
            make(n, torch.int32))


def _samples(case, seed):
    """Features and targets of training samples: ascending distances over their
    mean, targets of the order of the solved lambda over the mean distance."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.rand(case["count"], 16, generator=g, device="cuda").add_(0.05).cumsum(1).sqrt_()
    feat = d / d.mean(1, keepdim=True)
    target = 0.45 + 0.12 * torch.randn(case["count"], generator=g, device="cuda") + 0.2 * (feat[:, 0] - 0.4)
    return feat.contiguous(), target.contiguous()


def _dev(a):
    return torch.from_numpy(a).cuda()


def prepare(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    st = dict(case=case)
    if kind == "mlp_grad":
        st["mlp"] = f2m.f2m_mlp_create(load_weights())
        st["feat"], st["target"] = _samples(case, seed)
        return st
    if kind == "batch":
        insts = []
        sizes = [int(n) for n in _sizes(case)]
        for i, n in enumerate(sizes):
            xy = _points(n, "clustered" if i % 2 else "uniform", _gen(seed, 1 + i))
            insts.append((xy,) + f2m.f2m_knn_csr(xy, case["k"]))
        st["instances"] = insts
        # where the results go: one device array of each kind, an instance's part of each
        rooms = [_room(n, case["k"]) for n in sizes]
        st["out"] = [torch.zeros(c, dtype=t, device="cuda")
                     for c, t in ((sum(sizes), torch.int32), (sum(sizes) + len(sizes), torch.int32),
                                  (sum(rooms), torch.int32), (sum(rooms), torch.uint8))]
        st["parts"] = list(zip(*[a.split(c) for a, c in
                                 zip(st["out"], (sizes, [n + 1 for n in sizes], rooms, rooms))]))
        return st
    xy = _points(case["n"], case["points"], gen)
    if kind == "knn":
        st["xy"] = xy
        st["col"] = np.zeros(_room(case["n"], case["k"]), np.int32)
        return st
    if kind == "infer":
        st["xy"] = _dev(xy)
        st["mlp"] = f2m.f2m_mlp_create(load_weights())
        return st
    rp, col = f2m.f2m_knn_csr(xy, case["k"])
    if kind == "bmatching":
        st["graph"] = (xy, rp, col)
        st["b"] = gen.integers(1, case["bmax"] + 1, size=case["n"]).astype(np.int32)
        st["out"] = _out(case["n"], case["k"], False)
        return st
    if kind == "solve" and case["io"] == "host":
        st["graph"] = (xy, rp, col)
    else:
        st["graph"] = (_dev(xy), _dev(rp), _dev(col))
    if kind in ("solve", "subtour"):
        st["out"] = _out(case["n"], case["k"], case.get("io") != "host")
    if kind == "subtour":
        st["mu"] = np.zeros(case["n"], np.int32)
    if kind in ("solve", "price"):
        st["params"] = f2m.f2m_default_params(pricing=case["pricing"])
    if kind in ("gdp", "price"):
        st["ctx"] = f2m.f2m_create(*st["graph"], params=st.get("params"))
        st["lam0"] = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
    if kind == "price":
        f2m.f2m_gdp(st["ctx"], SWEEPS)
        st["pairs"] = np.zeros((4 * case["n"], 2), np.int32)
    return st


# ---- one pass ---------------------------------------------------------------------------


def _results(ctx, out):
    f2m.f2m_get_x(ctx, out=out[:4])
    _, fb = f2m.f2m_get_lambda(ctx, out=out[4])
    return [*out, fb]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("solve", "bmatching", "subtour"):
        ctx = f2m.f2m_create(*st["graph"], params=st.get("params"))
        if kind == "bmatching":
            f2m.f2m_set_degrees(ctx, st["b"])
        if kind == "subtour":
            bound2 = f2m.f2m_solve_subtour(ctx, case["rounds"])["bound2"]
            mu, layers = f2m.f2m_get_cut_duals(ctx)
            st["mu"][:len(mu)] = mu
            extra = [bound2, st["mu"], layers]
        else:
            extra = [f2m.f2m_solve(ctx).bound2]
        out = _results(ctx, st["out"]) + extra
        f2m.f2m_destroy(ctx)
        return out
    if kind == "batch":
        b = f2m.f2m_create_batch(st["instances"])
        infos, _ = f2m.f2m_solve_batch(b)
        for i, (lam, rp, col, x2) in enumerate(st["parts"]):
            f2m.f2m_batch_get_lambda(b, i, out=lam)
            f2m.f2m_batch_get_x(b, i, out=(rp, col, x2))
        f2m.f2m_destroy_batch(b)
        return [*st["out"], np.array([[i.bound2, i.frac_bits] for i in infos])]
    if kind == "gdp":
        f2m.f2m_set_lambda(st["ctx"], st["lam0"], F)
        status, sweeps, _, _ = f2m.f2m_gdp(st["ctx"], case["sweeps"])
        lam, _ = f2m.f2m_get_lambda(st["ctx"], device="cuda")
        return [lam, sweeps, status]
    if kind == "price":
        count, pairs = f2m.f2m_price(st["ctx"])
        # they come in no stated order
        st["pairs"][:count] = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
        return [count, st["pairs"]]
    if kind == "knn":
        rp, col = f2m.f2m_knn_csr(st["xy"], case["k"])
        st["col"][:len(col)] = col
        return [rp, st["col"]]
    if kind == "infer":
        feat, scale = f2m.f2m_features(st["xy"], device="cuda")
        return [feat, scale, f2m.f2m_mlp_forward(st["mlp"], feat)]
    loss, grad = f2m.f2m_mlp_grad(st["mlp"], st["feat"], st["target"])
    return [loss, grad]


# ---- what a pass cannot do without ----------------------------------------------------------


def _nnz(n, k):
    """Entries of a symmetrised k-NN graph: about 1.14 n k on these points."""
    return int(1.14 * n * k)


def _solve_work(n, nnz):
    """Points and graph in; graph, costs, x and lambda out; 128 sweeps of about
    10 integer operations an entry; 7 operations a pair, all pairs once."""
    return dict(bytes=8 * n + 4 * n + 4 * nnz + 4 * n + 9 * nnz + 4 * n,
                flops=10 * SWEEPS * nnz + 7 * n * (n - 1) // 2)


def work(case):
    kind = case["kind"]
    if kind == "mlp_grad":
        c = case["count"]
        return dict(bytes=c * 17 * 4 + 2 * 4 * f2m.F2M_MLP_NPARAMS,
                    flops=c * 2 * (3 * 128 * 128 + 2 * 16 * 128 + 2 * 128))
    if kind == "batch":
        mean = (case["hi"] - case["lo"]) / max(math.log(case["hi"] / case["lo"]), 1e-9) \
            if case["hi"] > case["lo"] else case["lo"]
        w = _solve_work(int(mean), _nnz(mean, case["k"]))
        return {key: case["count"] * v for key, v in w.items()}
    n = case["n"]
    if kind == "infer":
        # points in, features, scale and y out; the network's two products
        return dict(bytes=8 * n + 64 * n + 4 * n + 4 * n, flops=n * 2 * (16 * 128 + 128 * 128 + 128))
    nnz = _nnz(n, case["k"])
    if kind == "knn":
        return dict(bytes=8 * n + 4 * n + 4 * nnz, flops=5 * nnz)
    if kind == "gdp":
        # phases that reach their fixed point end before the cap (about 5,000
        # sweeps at 20,000 points)
        return dict(bytes=8 * nnz + 12 * n, flops=10 * nnz * min(case["sweeps"], 5000))
    if kind == "price":
        return dict(bytes=8 * n + 4 * n + 4 * nnz, flops=7 * n * (n - 1) // 2)
    w = _solve_work(n, nnz)
    if kind == "bmatching":
        w["bytes"] += 4 * n
    if kind == "subtour":
        w = {key: (1 + case["rounds"]) * v for key, v in w.items()}
    return w


# ---- the same in 64 bits -----------------------------------------------------------------


def _knn_exact(xy, k):
    """(index [n, k], d2 [n, k]) int64: nearest other points, ties by index."""
    p = _dev(xy).long()
    n = len(p)
    ids = torch.arange(n, device="cuda")
    idx, dist = [], []
    step = max(1, 100_000_000 // n)
    for a in range(0, n, step):
        q = p[a:a + step]
        key = (q[:, None, 0] - p[None, :, 0]) ** 2 + (q[:, None, 1] - p[None, :, 1]) ** 2
        key.mul_(1 << 18).add_(ids)
        key[torch.arange(len(q), device="cuda"), ids[a:a + step]] = 1 << 62
        top = key.topk(k, dim=1, largest=False).values
        idx.append(top & ((1 << 18) - 1))
        dist.append(top >> 18)
    return torch.cat(idx), torch.cat(dist)


def _csr_exact(xy, k):
    """(row_ptr, col) int64 of the symmetrised graph, rows ascending."""
    n = len(xy)
    idx, _ = _knn_exact(xy, k)
    u = torch.arange(n, device="cuda")[:, None].expand(n, k).reshape(-1)
    v = idx.reshape(-1)
    key = torch.cat([u * n + v, v * n + u]).unique()
    rp = torch.zeros(n + 1, dtype=torch.long, device="cuda")
    rp[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return rp, key % n


def _cost(d2):
    """nint(sqrt(d2)), exactly: r = floor(sqrt), one more beyond r (r + 1)."""
    r = d2.double().sqrt().long()
    r = torch.where(r * r > d2, r - 1, r)
    return r + (d2 > r * r + r)


def _gdp_exact(xy, rp, col, sweeps):
    """(lambda, sweeps run, status) of a GDP phase from 0."""
    n = len(xy)
    p = _dev(xy).long()
    deg = rp[1:] - rp[:-1]
    width = int(deg.max())
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    at = torch.arange(len(col), device="cuda") - rp[row]
    cost = torch.full((n, width), 1 << 45, dtype=torch.long, device="cuda")
    nbr = torch.zeros((n, width), dtype=torch.long, device="cuda")
    cost[row, at] = _cost(((p[row] - p[col]) ** 2).sum(1)) << F
    nbr[row, at] = col
    lam = torch.zeros(n, dtype=torch.long, device="cuda")
    for t in range(1, sweeps + 1):
        z = cost - lam[:, None] - lam[nbr]
        top = z.topk(3, dim=1, largest=False).values
        d = torch.div(top[:, 1] + top[:, 2], 4, rounding_mode="trunc")
        lam = lam + d
        if not bool(d.any()):
            return lam, t, 0
    return lam, sweeps, f2m.F2M_ERR_NOT_CONVERGED


def _price_exact(xy, rp, col, lam):
    """Pairs u < v outside the graph with c_uv 2^F < lambda_u + lambda_v, ascending."""
    p = _dev(xy).long()
    n = len(p)
    ids = torch.arange(n, device="cuda")
    row = torch.repeat_interleave(ids, rp[1:] - rp[:-1])
    found = []
    step = max(1, 50_000_000 // n)
    for a in range(0, n, step):
        q = p[a:a + step]
        d2 = (q[:, None, 0] - p[None, :, 0]) ** 2 + (q[:, None, 1] - p[None, :, 1]) ** 2
        neg = (_cost(d2) << F) < lam[a:a + step, None] + lam[None, :]
        neg &= ids[None, :] > ids[a:a + step, None]
        here = (row >= a) & (row < a + step)
        neg[row[here] - a, col[here]] = False
        found.append(neg.nonzero() + torch.tensor([a, 0], device="cuda"))
    return torch.cat(found)


def _mlp_forward_exact(w, feat):
    W1, b1, W2 = w[:2048].view(128, 16), w[2048:2176], w[2176:18560].view(128, 128)
    b2, w3, b3 = w[18560:18688], w[18688:18816], w[18816]
    h = torch.relu(feat @ W1.T + b1)
    return torch.relu(h @ W2.T + b2) @ w3 + b3


def exact(case, seed):
    """The integer results of whole solves are optima among several, chosen by the
    library's own search order: they have no independent value here."""
    kind = case["kind"]
    w = torch.from_numpy(load_weights()).cuda().double()
    if kind == "mlp_grad":
        feat, target = _samples(case, seed)
        w.requires_grad_(True)
        loss = ((_mlp_forward_exact(w, feat.double()) - target.double()) ** 2).mean()
        loss.backward()
        return [float(loss.detach()), w.grad.cpu().numpy()]
    if kind not in ("knn", "infer", "gdp", "price"):
        return None
    xy = _points(case["n"], case["points"], _gen(seed))
    if kind == "infer":
        _, d2 = _knn_exact(xy, 16)
        d = d2.double().sqrt()
        scale = d.mean(1).clamp(min=1.0)
        feat = d / scale[:, None]
        return [feat, scale, _mlp_forward_exact(w, feat)]
    rp, col = _csr_exact(xy, case["k"])
    if kind == "knn":
        full = np.zeros(_room(case["n"], case["k"]), np.int32)
        full[:len(col)] = col.cpu().numpy()
        return [rp.cpu().numpy(), full]
    lam, sweeps, status = _gdp_exact(xy, rp, col, case["sweeps"] if kind == "gdp" else SWEEPS)
    if kind == "gdp":
        return [lam, sweeps, status]
    pairs = _price_exact(xy, rp, col, lam)
    full = np.zeros((4 * case["n"], 2), np.int32)
    full[:len(pairs)] = pairs.cpu().numpy()
    return [len(pairs), full]
