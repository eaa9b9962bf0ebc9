"""What the performance of this repository is measured on: its public calls over the sizes a user asks.

The graphs are the families of graphgen/workloads.py and bench.py (grids, road-like grids,
Chung-Lu, R-MAT, Erdos-Renyi with n ln n edges), drawn here on the GPU, the largest component
kept. ``prepare`` builds the graph handle and warms it up with a one-step query
(on which the library tunes itself for the batch width), as a service does before it answers;
``run`` is one public call (one training step where the case is training).

Every call returns its outputs whole. Distances come back as float64; with FP32 vectors
(mode "fp32") they hold FP32 precision -- the library picks its kernels by timing, so already two
processes differ in the last FP32 digits -- and a program that asks for that mode keeps them as
float32 features, as ``run`` does here. The FP64-class modes keep float64.
"""
import math

import numpy as np
import torch

import paper_2601_11159_gb300 as rd

# Stop rules in use: the benchmark's (relative error 1e-6), the paper's fixed k, a residual.
FIELDS = ("k_max", "rel_tol", "resid_tol", "fixed_k")


def _case(name, call, graph, size, pairs, mode, k_max, rel_tol=0.0, resid_tol=0.0, fixed_k=False, deg=20.0,
          gamma=2.1, weighted=False, host=False, steps=0):
    """``size``: vertices (grids: vertices a side; R-MAT: scale). ``steps``: Lanczos steps a pass
    runs, for ``work`` (typical where a tolerance decides)."""
    c = dict(call=call, graph=graph, size=size, pairs=pairs, mode=mode, k_max=k_max, rel_tol=rel_tol,
             resid_tol=resid_tol, fixed_k=fixed_k, deg=deg, gamma=gamma, weighted=weighted, host=host,
             steps=steps or k_max)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one interactive question on a small road map, to residual 1e-10 in FP64 (ids and result on the host)
        _case("pair_grid64_fp64", "query", "grid", 64, 1, "fp64", 500, resid_tol=1e-10, host=True, steps=190),
        # the paper's scalability experiment at its small end: 64 pairs, k = 20 steps, a 1,000-vertex graph
        _case("batch_er1000_fp32", "query", "er", 1000, 64, "fp32", 20, fixed_k=True),
        # a mid-size network, an odd number of pairs, FP64 throughout
        _case("batch_cl20k_fp64", "query", "cl", 20_000, 70, "fp64", 200, rel_tol=1e-9, steps=10),
        # one question on the benchmark's graph: the single-vector path
        _case("pair_cl1m_fp32", "query", "cl", 1_000_000, 1, "fp32", 200, rel_tol=1e-6, steps=6),
        # the benchmark itself: 256 pairs at once on a million vertices
        _case("batch_cl1m_fp32", "query", "cl", 1_000_000, 256, "fp32", 200, rel_tol=1e-6, steps=7),
        # throughput on a skewed graph (R-MAT, edge factor 16), 128 pairs
        _case("batch_rmat20_fp32", "query", "rmat", 20, 128, "fp32", 200, rel_tol=1e-6, deg=30.0, steps=6),
        # a stretch of a long road-network run (large condition number) in double-float, 64 pairs
        _case("batch_road1024_df64", "query", "road", 1024, 64, "df64", 200, fixed_k=True, weighted=True),
        # gradient of 32 distances over all edges of a large weighted network
        _case("grad_cl4m_fp32", "grad", "cl", 4_000_000, 32, "fp32", 200, rel_tol=1e-6, gamma=2.3, weighted=True,
              steps=8),
        # a training step on edge weights: new weights in, distances, loss, gradient back
        _case("train_cl100k_fp32", "train", "cl", 100_000, 64, "fp32", 200, rel_tol=1e-6, gamma=2.3, weighted=True,
              steps=8),
        # electric potentials on a road map (what route search starts from)
        _case("potential_road500_fp64", "potential", "road", 500, 16, "fp64", 100, fixed_k=True, weighted=True),
        # electric flows of a few pairs over every edge of a social network
        _case("flow_cl200k_fp32", "flow", "cl", 200_000, 16, "fp32", 200, rel_tol=1e-6, steps=7),
        # the Power Method baseline, with the estimate after each term
        _case("power_er100k_fp64", "power", "er", 100_000, 16, "fp64", 50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair_grid", "batch_er", "batch_cl_mid", "pair_cl", "batch_cl", "batch_rmat", "batch_road",
                       "grad", "train", "potential", "flow", "power"])
    mode = rng.choice(["fp32", "fp64"])
    if kind == "pair_grid":
        g = rng.choice(["grid", "road"])
        return _case(None, "query", g, rng.randint(20, 90), rng.choice([1, 1, 2, 3]), "fp64", 1000, resid_tol=1e-10,
                     weighted=g == "road", host=True, steps=200)
    if kind == "batch_er":
        return _case(None, "query", "er", _log(rng, 100, 2500), _log(rng, 20, 300), mode, rng.randint(10, 25),
                     fixed_k=True)
    if kind == "batch_cl_mid":
        m = rng.choice(["fp32", "fp64", "df64"])
        return _case(None, "query", "cl", _log(rng, 12_000, 100_000), _log(rng, 5, 250), m, 200,
                     rel_tol=1e-6 if m == "fp32" else 1e-9, weighted=rng.random() < 0.5, steps=8)
    if kind == "pair_cl":
        return _case(None, "query", "cl", _log(rng, 50_000, 1_000_000), 1, mode, 200, rel_tol=1e-6,
                     weighted=rng.random() < 0.3, host=rng.random() < 0.5, steps=6)
    if kind == "batch_cl":
        return _case(None, "query", "cl", _log(rng, 200_000, 1_000_000), rng.randint(33, 256), "fp32", 200,
                     rel_tol=1e-6, deg=rng.choice([10.0, 20.0]), weighted=rng.random() < 0.3, steps=7)
    if kind == "batch_rmat":
        return _case(None, "query", "rmat", rng.randint(15, 19), rng.randint(17, 128), "fp32", 200, rel_tol=1e-6,
                     deg=30.0, steps=6)
    if kind == "batch_road":
        return _case(None, "query", "road", _log(rng, 150, 1000), _log(rng, 3, 64), rng.choice(["df64", "fp64"]),
                     rng.randint(30, 120), fixed_k=True, weighted=True)
    if kind == "grad":
        return _case(None, "grad", "cl", _log(rng, 200_000, 2_000_000), _log(rng, 5, 32), "fp32", 200, rel_tol=1e-6,
                     gamma=2.3, weighted=True, steps=8)
    if kind == "train":
        return _case(None, "train", "cl", _log(rng, 10_000, 200_000), _log(rng, 10, 100), mode, 200, rel_tol=1e-6,
                     gamma=2.3, weighted=True, steps=8)
    if kind == "potential":
        return _case(None, "potential", "road", _log(rng, 100, 600), _log(rng, 2, 40), "fp64", rng.randint(50, 120),
                     fixed_k=True, weighted=True)
    if kind == "flow":
        return _case(None, "flow", "cl", _log(rng, 20_000, 300_000), _log(rng, 2, 40), mode, 200,
                     rel_tol=1e-6 if mode == "fp32" else 1e-8, steps=8)
    return _case(None, "power", "er", _log(rng, 10_000, 200_000), _log(rng, 2, 60), mode, rng.randint(20, 60))


# ------------------------------------------------------------------ inputs
def _rand(gen, n):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)


def _largest_component(n, a, b):
    """Vertices of the largest component (bool[n]): labels hooked to the smaller root, then flattened."""
    lab = torch.arange(n, device="cuda")
    ea, eb = a, b
    while True:
        la, lb = lab[ea], lab[eb]
        m = la != lb
        if not bool(m.any()):
            break
        ea, eb, la, lb = ea[m], eb[m], la[m], lb[m]
        lab.scatter_reduce_(0, torch.maximum(la, lb), torch.minimum(la, lb), "amin")
        while True:
            up = lab[lab]
            if torch.equal(up, lab):
                break
            lab = up
    return lab == torch.bincount(lab).argmax()


def _edges(case, gen):
    """(n, a, b): endpoints before self-loops, duplicates and small components are dropped."""
    kind, size = case["graph"], case["size"]
    if kind in ("grid", "road"):
        ids = torch.arange(size * size, device="cuda").view(size, size)
        a = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
        b = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
        if kind == "road":  # 5% of the edges deleted
            keep = _rand(gen, a.numel()) >= 0.05
            a, b = a[keep], b[keep]
        return size * size, a, b
    if kind == "er":
        m = int(size * math.log(size))
        ends = torch.randint(0, size, (2, m), device="cuda", generator=gen)
        return size, ends[0], ends[1]
    if kind == "rmat":  # quadrant probabilities 0.57, 0.19, 0.19, 0.05 at every level
        u = torch.zeros(16 << size, dtype=torch.int64, device="cuda")
        v = torch.zeros_like(u)
        for _ in range(size):
            r = torch.rand(u.numel(), device="cuda", generator=gen)
            u = (u << 1) | (r >= 0.76)
            v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        return 1 << size, u, v
    # Chung-Lu: expected degrees ~ (i+1)^(-1/(gamma-1)), scaled to the mean, capped at sqrt of their sum
    w = torch.arange(1, size + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (case["gamma"] - 1.0))
    total = case["deg"] * size
    for _ in range(50):
        w = torch.clamp(w * (total / w.sum()), max=math.sqrt(total))
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    m = int(total / 2)
    a, b = (torch.searchsorted(cdf, _rand(gen, m), right=True).clamp_(max=size - 1) for _ in range(2))
    return size, a, b


def _graph(case, fixed, gen):
    """Symmetric CSR on the GPU: row_ptr int64, col int32, w float32 or None, old id of each vertex."""
    n, a, b = _edges(case, fixed)
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    key = torch.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    keep = _largest_component(n, lo, hi)
    old = torch.nonzero(keep).view(-1)
    new = torch.cumsum(keep, 0) - 1
    m = keep[lo]
    lo, hi = new[lo[m]], new[hi[m]]
    n = old.numel()
    key, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    row, col = key // n, key % n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    w = None
    if case["weighted"]:  # roads: uniform in [0.5, 2]; networks: lognormal(0, 0.5)
        m = lo.numel()
        if case["graph"] == "road":
            x = 0.5 + 1.5 * _rand(gen, m)
        else:
            x = torch.exp(0.5 * torch.randn(m, dtype=torch.float64, device="cuda", generator=gen))
        w = x.float().repeat(2)[order].contiguous()
    return row_ptr, col.int().contiguous(), w, old


def _pairs(case, gen, n, old):
    """Pair ids: uniform, or on grids at a Manhattan distance of a quarter of the side."""
    P = case["pairs"]
    if case["graph"] in ("grid", "road"):
        side = case["size"]
        dist = max(1, side // 4)
        pick = torch.randint(0, n, (400 * P,), device="cuda", generator=gen)
        dx = torch.randint(0, dist + 1, (400 * P,), device="cuda", generator=gen)
        sign = torch.randint(0, 2, (2, 400 * P), device="cuda", generator=gen) * 2 - 1
        x, y = old[pick] % side + sign[0] * dx, old[pick] // side + sign[1] * (dist - dx)
        new = torch.full((side * side,), -1, dtype=torch.int64, device="cuda")
        new[old] = torch.arange(n, device="cuda")
        ok = (x >= 0) & (x < side) & (y >= 0) & (y < side)
        other = torch.where(ok, new[torch.where(ok, y * side + x, 0)], -1)
        at = torch.nonzero(other >= 0).view(-1)[:P]
        return pick[at].int(), other[at].int()
    s = torch.randint(0, n, (P,), device="cuda", generator=gen)
    t = torch.randint(0, n - 1, (P,), device="cuda", generator=gen)
    return s.int(), (t + (t >= s)).int()


def _inputs(case, seed):
    # the network of a case is fixed, as a service's is; the questions, the weights and the targets are the seed's
    fixed, gen = torch.Generator(device="cuda"), torch.Generator(device="cuda")
    fixed.manual_seed(20260101)
    gen.manual_seed(seed)
    row_ptr, col, w, old = _graph(case, fixed, gen)
    s, t = _pairs(case, gen, old.numel(), old)
    # what a training loop wants the distances to be
    target = 0.5 * torch.rand(case["pairs"], dtype=torch.float64, device="cuda", generator=gen)
    return row_ptr, col, w, s, t, target


def prepare(case, seed):
    row_ptr, col, w, s, t, target = _inputs(case, seed)
    G = rd.Graph(row_ptr, col, w)
    opts = dict(mode=case["mode"], **{k: case[k] for k in FIELDS})
    if case["call"] != "power":
        G.query(s, t, mode=case["mode"], k_max=1, fixed_k=True)
    if case["host"]:
        s, t = s.cpu().numpy(), t.cpu().numpy()
    return dict(call=case["call"], G=G, s=s, t=t, w=w, target=target, opts=opts, single=case["mode"] == "fp32",
                steps=case["k_max"], ones=torch.ones(case["pairs"], dtype=torch.float64, device="cuda"))


# -------------------------------------------------------------------- calls
def _r(r, single):
    if not single:
        return r
    return r.float() if isinstance(r, torch.Tensor) else r.astype(np.float32)


def run(state):
    G, s, t, opts, single = state["G"], state["s"], state["t"], state["opts"], state["single"]
    call = state["call"]
    if call == "query":
        res = G.query(s, t, **opts)
        out = {"r": _r(res.r, single), "iters": res.iters, "status": res.status}
        if not opts["fixed_k"]:  # a program that names a tolerance looks at the estimate it stopped on
            out["err"] = _r(res.err, single)
        return out
    if call == "grad":
        gw, r = G.edge_grad(s, t, state["ones"], **opts)
        return {"grad_w": gw, "r": _r(r, single)}
    if call == "train":
        w = state["w"].detach().requires_grad_()
        r = rd.ResistanceDistance.apply(w, G, s, t, opts)
        loss = ((r - state["target"]) ** 2).mean()
        loss.backward()
        return {"r": _r(r.detach(), single), "grad_w": w.grad}
    if call == "potential":
        phi, r = G.potential(s, t, **opts)
        return {"phi": phi, "r": _r(r, single)}
    if call == "flow":
        f, r = G.flow(s, t, **opts)
        return {"flow": f, "r": _r(r, single)}
    r, hist = G.power_method(s, t, state["steps"], mode=opts["mode"], history=True)
    return {"r": _r(r, single), "hist": _r(hist, single)}


# --------------------------------------------------------------------- work
def _sizes(case):
    """Vertices and stored entries (after the small components are gone), as the families have them."""
    size = case["size"]
    if case["graph"] == "grid":
        return size * size, 4 * size * (size - 1)
    if case["graph"] == "road":
        return size * size, int(0.95 * 4 * size * (size - 1))
    if case["graph"] == "er":
        return size, int(2 * size * math.log(size))
    if case["graph"] == "rmat":
        return int(0.6 * (1 << size)), int(30.0 * (1 << size))
    return size, int(0.985 * case["deg"] * size)


def work(case):
    """Bytes: per step the CSR once and, per pair column, q_i and q_{i-1} in and q_{i+1} out; where all
    of that stays on the chip between steps (under 100 MB) it is counted once for the call. Then the
    call's own outputs. Flops: a multiply-add per entry and column (an add, unweighted) and about ten
    operations per vector element and step."""
    n, nnz = _sizes(case)
    P, steps = case["pairs"], case["steps"]
    elem = 4 if case["mode"] == "fp32" else 8
    csr = nnz * (8 if case["weighted"] else 4) + 8 * n
    vec = 3 * n * P * elem
    once = csr + vec < 100e6
    total = csr + (0 if once else steps * vec + (steps - 1) * csr)
    flops = steps * P * ((2 if case["weighted"] else 1) * nnz + 10.0 * n)
    if case["call"] in ("grad", "train"):
        total += n * P * elem + 8 * nnz  # the potentials, the entries and the gradient
        flops += 3.0 * nnz * P
    if case["call"] == "train":
        total += 4 * nnz  # the new weights
    if case["call"] == "potential":
        total += 4 * n * P
    if case["call"] == "flow":
        total += n * P * elem + 4 * nnz * P
    return {"bytes": float(total), "flops": float(flops)}


# -------------------------------------------------------------------- exact
def _operator(row_ptr, col, w):
    """D^{-1/2} W D^{-1/2} in 64 bits, the degrees, the row of each entry."""
    n = row_ptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    val = torch.ones(col.numel(), dtype=torch.float64, device="cuda") if w is None else w.double()
    deg = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, val)
    val = val / torch.sqrt(deg[row] * deg[col.long()])
    return torch.sparse_csr_tensor(row_ptr, col.long(), val, size=(n, n)), deg, row


def _lanczos(A, deg, s, t, case, want_x):
    """Lanczos iteration (the paper's Algorithm 3) from b = e_s/sqrt(d_s) - e_t/sqrt(d_t), all columns at once,
    each until the case's stop rule; r = |b|^2 e_1' (I - T)^-1 e_1 and, asked for, D^{-1/2} x with (I - A) x = b."""
    n, P = deg.numel(), s.numel()
    s, t, cols = s.long(), t.long(), torch.arange(P, device="cuda")
    dh = torch.sqrt(deg)
    top = (dh / torch.linalg.vector_norm(dh))[:, None]
    b2 = 1.0 / deg[s] + 1.0 / deg[t]
    v = torch.zeros(n, P, dtype=torch.float64, device="cuda")
    v[s, cols] = 1.0 / (dh[s] * b2.sqrt())
    v[t, cols] = -1.0 / (dh[t] * b2.sqrt())
    prev = torch.zeros_like(v)
    x, d = (torch.zeros_like(v), torch.zeros_like(v)) if want_x else (None, None)
    zero = torch.zeros(P, dtype=torch.float64, device="cuda")
    beta, delta, g, S = zero.clone(), zero + 1.0, zero + 1.0, zero.clone()
    active = torch.ones(P, dtype=torch.bool, device="cuda")
    iters = torch.zeros(P, dtype=torch.int32, device="cuda")
    inc = []
    for k in range(1, case["k_max"] + 1):
        w = A @ v - beta * prev
        alpha = (w * v).sum(0)
        w = w - alpha * v
        w = w - top * (top * w).sum(0)
        nb = torch.linalg.vector_norm(w, dim=0)
        lam = beta / delta if k > 1 else zero
        delta = 1.0 - alpha - (beta * lam if k > 1 else 0.0)
        g = g * lam if k > 1 else g
        inc.append(g * g / delta)
        S = torch.where(active, S + inc[-1], S)
        iters += active
        if want_x:
            d = v + lam * d
            x = x + torch.where(active, b2.sqrt() * g / delta, zero) * d
        stop = nb <= 1e-12 * (alpha.abs() + beta)
        if not case["fixed_k"]:
            if case["resid_tol"] > 0:
                stop |= nb * (g / delta).abs() <= case["resid_tol"]
            if case["rel_tol"] > 0 and k >= 4:
                rho = torch.stack([inc[-j] / inc[-j - 1] for j in (1, 2, 3)]).amax(0).clamp(min=0.5)
                stop |= (rho < 1) & (inc[-1] * rho / ((1 - rho) ** 2 * S) <= case["rel_tol"])
        active &= ~stop
        if not bool(active.any()):
            break
        nb = torch.where(active, nb, zero + 1.0)
        prev, v, beta = v, torch.where(active, w / nb, zero), torch.where(active, nb, zero)
        delta, g = torch.where(active, delta, zero + 1.0), torch.where(active, g, zero)
    return b2 * S, iters, (x / dh[:, None] if want_x else None)


def exact(case, seed):
    row_ptr, col, w, s, t, target = _inputs(case, seed)
    A, deg, row = _operator(row_ptr, col, w)
    call = case["call"]
    if call == "power":  # the lazy walk's series: rbar_l = 1/2 sum_i (e_s-e_t)' D^-1 (I/2 + P/2)^i (e_s-e_t)
        s, t, cols = s.long(), t.long(), torch.arange(s.numel(), device="cuda")
        dh = torch.sqrt(deg)
        y = torch.zeros(deg.numel(), s.numel(), dtype=torch.float64, device="cuda")
        y[s, cols] = 1.0 / dh[s]
        y[t, cols] = -1.0 / dh[t]
        hist = []
        for i in range(case["k_max"] + 1):
            term = 0.5 * (y[s, cols] / dh[s] - y[t, cols] / dh[t])
            hist.append(term if not hist else hist[-1] + term)
            y = 0.5 * y + 0.5 * (A @ y)
        return {"r": hist[-1], "hist": torch.stack(hist)}
    r, iters, phi = _lanczos(A, deg, s, t, case, call != "query")
    if call == "query":
        return {"r": r, "iters": None, "status": None, "err": None}
    if call == "potential":
        return {"phi": phi.T.contiguous(), "r": r}
    col = col.long()
    if call == "flow":
        return {"flow": (phi[row] - phi[col]).T.contiguous(), "r": r}
    gr = 2.0 * (r - target) / r.numel() if call == "train" else torch.ones_like(r)
    gw = torch.empty(col.numel(), dtype=torch.float64, device="cuda")
    step = 1 << 22
    for e in range(0, col.numel(), step):
        gw[e:e + step] = -0.5 * ((phi[row[e:e + step]] - phi[col[e:e + step]]) ** 2 * gr).sum(1)
    return {"grad_w": gw, "r": r}
