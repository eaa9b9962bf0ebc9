"""GPU parity: the CUDA path (called through the C ABI via the thin binding) against
the CPU oracle on the same seeded inputs.

Tolerances: FP64 mode within 1e-9 relative of the oracle, FP32-vector mode within
1e-5 relative (the bars fixed for this method's two precision modes).
"""
import numpy as np
import pytest

from graphgen import families as F
from graphgen import workloads as W
from graphgen.graph import to_csr
from oracle import dense, lanczos, power
from tests import closed_forms as CF

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-9
FP32_TOL = 1e-5


@pytest.fixture(scope="module")
def rd():
    import torch

    assert torch.cuda.is_available()
    import paper_2601_11159_gb300 as rd

    rd.lib()  # fails loudly if the library is not built
    return rd


def rel(a, b):
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    return np.abs(a - b) / np.abs(b)


SMALL = [
    ("K7", lambda: F.complete(7)),
    ("C11", lambda: F.cycle(11)),
    ("P9", lambda: F.path(9)),
    ("toy", lambda: F.toy_graph()),
    ("grid8", lambda: F.grid(8)),
    ("grid5x7", lambda: F.grid(5, 7)),
    ("rc60u", lambda: F.random_connected(60, 100, 3, None)),
    ("rc70w", lambda: F.random_connected(70, 140, 5, "uniform")),
    ("rc80ln", lambda: F.random_connected(80, 200, 7, "lognormal")),
]


@pytest.mark.parametrize("name,make", SMALL)
@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("kernel", ["group", "group_sorted", "stream", "async", "onchip"])
def test_small_graphs_vs_dense(rd, name, make, mode, kernel):
    g = make()
    s, t = F.random_pairs(g.n, 9, 17)
    ref = dense.DenseRD.of(g).r(s, t)
    G = rd.Graph.from_csr(g)
    tol = FP64_TOL if mode == "fp64" else FP32_TOL
    kw = dict(onchip=True) if kernel == "onchip" else dict(kernel=kernel, onchip=False)
    res = G.query(s, t, mode=mode, k_max=400, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-6, **kw)
    assert np.all(res.status >= 0), res.status
    assert rel(res.r, ref).max() < tol, (name, mode, rel(res.r, ref).max())


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-11), ("fp32", 2e-5)])
def test_fixed_k_matches_oracle_history(rd, mode, tol):
    """Same k, same recurrence: the GPU estimate after k steps equals the oracle's rhat_k."""
    g = F.grid_deleted(24, 0.05, 9)
    s, t = F.random_pairs(g.n, 5, 2)
    G = rd.Graph.from_csr(g)
    for k in [1, 2, 5, 12, 30]:
        ref = np.array([lanczos.lanczos_pair(g, int(a), int(b), k_max=k)["r"] for a, b in zip(s, t)])
        for onchip in (False, True):
            res = G.query(s, t, mode=mode, k_max=k, fixed_k=True, onchip=onchip)
            assert np.all(res.iters == k)
            assert rel(res.r, ref).max() < tol, (k, onchip, rel(res.r, ref).max())


def test_grid64_corner_fp64_closed_form(rd):
    """64x64 grid, s = 0, t = 4095, FP64, k <= 500 or relative residual 1e-10."""
    g, s, t = W.grid64()
    ref = CF.grid_r(64, 64, 0, 4095)
    G = rd.Graph.from_csr(g)
    res = G.query(s, t, mode="fp64", k_max=500, rel_tol=0.0, resid_tol=1e-10)
    assert res.status[0] == 0 and res.iters[0] < 500
    assert rel(res.r, [ref]).max() < FP64_TOL
    # the same with the single-vector SpMV paths (row-group and row-stream kernels)
    for kernel in ["group", "group_sorted", "stream"]:
        res1 = G.query(s, t, mode="fp64", k_max=500, rel_tol=0.0, resid_tol=1e-10, plain=True, kernel=kernel)
        assert rel(res1.r, [ref]).max() < FP64_TOL


def test_ragged_batch_edge_cases(rd):
    g = F.random_connected(300, 500, 4, "uniform")
    n = g.n
    s, t = F.random_pairs(n, 37, 8)          # 37 pairs: not a multiple of any tile
    s[3] = t[3]                              # s == t
    s[10], t[10] = 0, n - 1                  # extreme ids
    ref = dense.DenseRD.of(g).r(s, t)
    G = rd.Graph.from_csr(g)
    for mode, tol in [("fp64", FP64_TOL), ("fp32", FP32_TOL)]:
        for onchip in (False, True):
            res = G.query(s, t, mode=mode, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-6, onchip=onchip)
            assert res.r[3] == 0.0 and res.iters[3] == 0 and res.status[3] == 0
            m = np.arange(37) != 3
            assert rel(res.r[m], ref[m]).max() < tol
    empty = G.query(np.zeros(0, np.int32), np.zeros(0, np.int32))
    assert empty.r.size == 0


def test_disconnected_and_invalid(rd):
    a = F.cycle(6)
    b = F.path(5)
    ea, eb, _ = a.undirected_edges()
    fa, fb, _ = b.undirected_edges()
    g = to_csr(11, np.concatenate([ea, fa + 6]), np.concatenate([eb, fb + 6]))
    G = rd.Graph.from_csr(g)
    assert G.ncomponents == 2
    res = G.query(np.array([0, 6, 1], np.int32), np.array([3, 10, 8], np.int32), mode="fp64", rel_tol=1e-12)
    assert res.r[0] == pytest.approx(CF.cycle_r(6, 3), rel=1e-9)
    assert res.r[1] == pytest.approx(4.0, rel=1e-9)
    assert np.isinf(res.r[2]) and res.status[2] == rd.RD_ERR_DISCONNECTED
    with pytest.raises(rd.RDError):
        G.query(np.array([0], np.int32), np.array([11], np.int32))
    with pytest.raises(rd.RDError):
        G.query(np.array([-1], np.int32), np.array([2], np.int32))


def test_bad_graphs_rejected(rd):
    g = F.path(4)
    with pytest.raises(rd.RDError):
        rd.Graph(g.row_ptr, np.array([1, 0, 2, 1, 3, 9], np.int32))           # column out of range
    with pytest.raises(rd.RDError):
        rd.Graph(g.row_ptr, g.col, np.array([1, 1, -1, 1, 1, 1], np.float32))  # negative weight
    with pytest.raises(rd.RDError):
        rd.Graph(np.array([0, 1, 2, 2], np.int64), np.array([1, 0], np.int32))  # isolated vertex 2
    asym = to_csr(3, np.array([0, 1]), np.array([1, 2]), np.array([1.0, 2.0], np.float32))
    w = asym.w.copy()
    w[0] = 5.0
    with pytest.raises(rd.RDError):
        rd.Graph(asym.row_ptr, asym.col, w, check_symmetry=True)


def test_self_loops_dropped(rd):
    g = F.random_connected(40, 60, 2, "uniform")
    rows = g.rows()
    # insert a self-loop at every vertex
    ra = np.concatenate([rows, np.arange(g.n)])
    ca = np.concatenate([g.col.astype(np.int64), np.arange(g.n)])
    wa = np.concatenate([g.w, np.full(g.n, 3.0, np.float32)])
    order = np.lexsort((ca, ra))
    rp = np.zeros(g.n + 1, np.int64)
    np.cumsum(np.bincount(ra, minlength=g.n), out=rp[1:])
    G = rd.Graph(rp, ca[order].astype(np.int32), wa[order])
    assert G.nnz == g.nnz
    s, t = F.random_pairs(g.n, 5, 1)
    res = G.query(s, t, mode="fp64", rel_tol=0.0, resid_tol=1e-12)
    assert rel(res.r, dense.DenseRD.of(g).r(s, t)).max() < FP64_TOL


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("kernel", ["group", "group_sorted", "stream"])
def test_batched_vs_plain_and_order(rd, mode, tol, kernel):
    g, s, t = W.chunglu(20000, 2.1, 20.0, 200000, 40, 77)
    G = rd.Graph.from_csr(g)
    kw = dict(mode=mode, k_max=60, fixed_k=True, kernel=kernel)
    b = G.query(s, t, **kw)
    p = G.query(s, t, plain=True, **kw)
    assert rel(b.r, p.r).max() < tol
    for tile in [16, 32, 64, 128, 256]:
        if mode == "fp64" and tile == 256:
            continue
        bt = G.query(s, t, rhs_tile=tile, **kw)
        assert rel(bt.r, p.r).max() < tol, tile
    perm = np.random.default_rng(0).permutation(len(s))
    bp = G.query(s[perm], t[perm], **kw)
    assert np.array_equal(bp.r, b.r[perm])      # same batch size: bitwise equal per pair
    again = G.query(s, t, **kw)
    assert np.array_equal(again.r, b.r)          # deterministic


@pytest.mark.parametrize("weighted", [False, True])
def test_async_kernel_vs_oracle_and_row_stream(rd, weighted):
    """The row-stream SpMM with asynchronous gathers into a shared-memory ring (FP32 vectors):
    on a power-law graph with heavy rows (split into chunks by the pre-pass) and a ragged pair
    count, every column slab width agrees with the oracle at convergence, with the row-stream
    kernel at fixed k, and with itself bitwise on a repeat and under a permutation; new
    weights are followed."""
    kernel = "async"
    g, s, t = W.chunglu(20000, 2.1, 20.0, 200000, 37, 77, weights="lognormal" if weighted else None)
    assert np.diff(g.row_ptr).max() > 256  # heavy rows present
    G = rd.Graph.from_csr(g)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=300, stop_tol=1e-14, threads=0)
    code = 5
    for tile in [16, 32, 64, 128]:
        kw = dict(mode="fp32", kernel=kernel, rhs_tile=tile, compact=False)
        res = G.query(s, t, k_max=300, rel_tol=0.0, resid_tol=1e-7, **kw)
        st = G.last_stats()
        assert st["kernel"] == code and st["rhs_tile"] == tile
        assert np.all(res.status >= 0)
        assert rel(res.r, ref).max() < FP32_TOL, (tile, rel(res.r, ref).max())
        fa = G.query(s, t, k_max=25, fixed_k=True, **kw)
        fs = G.query(s, t, mode="fp32", kernel="stream", rhs_tile=tile, compact=False, k_max=25, fixed_k=True)
        assert rel(fa.r, fs.r).max() < 2e-6, (tile, rel(fa.r, fs.r).max())
        assert np.array_equal(G.query(s, t, k_max=25, fixed_k=True, **kw).r, fa.r)
        perm = np.random.default_rng(1).permutation(len(s))
        fp = G.query(s[perm], t[perm], k_max=25, fixed_k=True, **kw)
        assert np.array_equal(fp.r, fa.r[perm])
    # graph replay and the compacting default path with this kernel
    kw = dict(mode="fp32", kernel=kernel, rhs_tile=32, k_max=300, rel_tol=1e-7)
    a = G.query(s, t, **kw)
    b = G.query(s, t, graph=False, **kw)
    assert np.array_equal(a.r, b.r)
    assert rel(a.r, ref).max() < FP32_TOL
    # new weights: the next query follows them
    w2 = F.lognormal_edge_weights(g.m, 0.0, 0.7, 91)
    g2 = F.weighted(g, w2)
    G.set_weights(g2.w)
    ref2, _, _ = lanczos.lanczos_batch(g2, s, t, k_max=300, stop_tol=1e-14, threads=0)
    r2 = G.query(s, t, mode="fp32", kernel=kernel, rhs_tile=64, compact=False, k_max=300, rel_tol=0.0,
                 resid_tol=1e-7).r
    assert rel(r2, ref2).max() < FP32_TOL


def _weakly_coupled(kind: str, eps: float):
    """Cliques joined through one edge of weight eps: the Krylov space of a pair across the
    weak edge is nearly invariant at some step, where beta_{i+1} / (|alpha_i| + beta_i)
    falls to 1e-5 .. 1e-8 before the recurrence goes on."""
    parts = [F.complete(40), F.path(10), F.complete(40)] if kind == "K40-P10-K40" else [F.complete(50), F.path(8)]
    links = [(0, 0, 1, 0, eps), (1, 9, 2, 0, 1.0)] if kind == "K40-P10-K40" else [(0, 0, 1, 0, eps)]
    off, A, B, Wt, offs = 0, [], [], [], []
    for g in parts:
        a, b, _ = g.undirected_edges()
        A.append(a + off)
        B.append(b + off)
        Wt.append(np.ones(a.size))
        offs.append(off)
        off += g.n
    for i, u, j, v, w in links:
        A.append(np.array([offs[i] + u]))
        B.append(np.array([offs[j] + v]))
        Wt.append(np.array([w]))
    g = to_csr(off, np.concatenate(A), np.concatenate(B), np.concatenate(Wt).astype(np.float32))
    pairs = [(1, 55), (3, 45)] if kind == "K40-P10-K40" else [(1, 57), (4, 52)]
    return g, np.array([p[0] for p in pairs], np.int32), np.array([p[1] for p in pairs], np.int32)


@pytest.mark.parametrize("kind,eps", [("K40-P10-K40", 1e-2), ("K40-P10-K40", 1e-3), ("K50+P8", 1e-2),
                                      ("K50+P8", 1e-3)])
def test_near_invariant_krylov_steps(rd, kind, eps):
    """Steps where beta_{i+1} is tiny against alpha_i (the cancellation regime of
    beta_{i+1}^2 = ||w||^2 - alpha_i^2 - gamma^2): the FP64 and double-float paths follow the
    oracle's r_k history at fixed k and converge to the dense pseudo-inverse value. The
    tolerance is 1e-8, above the FP64 oracle's own error on these graphs (up to 2.5e-9 against
    the dense reference: the weak edge makes them ill-conditioned)."""
    g, s, t = _weakly_coupled(kind, eps)
    ref = dense.DenseRD.of(g).r(s, t)
    # the regime is reached: beta_{i+1} / (|alpha_i| + beta_i) below 1e-4 at some step
    o = lanczos.lanczos_pair(g, int(s[0]), int(t[0]), k_max=60, stop_tol=1e-15)
    k = o["k"]
    ratio = o["beta"][1:k] / np.maximum(np.abs(o["alpha"][:k - 1]) + o["beta"][:k - 1], 1e-300)
    assert ratio.min() < 1e-4, ratio.min()
    G = rd.Graph.from_csr(g)
    for mode in ("fp64", "df64"):
        for onchip in (False, True):
            if mode == "df64" and onchip:
                continue  # double-float vectors: multi-kernel path only
            # the weak edge slows convergence: up to about 500 steps to residual 1e-11
            res = G.query(s, t, mode=mode, k_max=3000, rel_tol=0.0, resid_tol=1e-11, onchip=onchip)
            if mode == "fp64":
                assert np.all(res.status == 0), (mode, onchip, res.status, res.iters)
            else:
                # double-float vectors (about 48 bits) can lose definiteness of I - T_k after such
                # a step: the pair then stops flagged RD_ERR_NUMERIC, never silently
                assert np.all((res.status == 0) | (res.status == rd.RD_ERR_NUMERIC)), res.status
                assert np.any(res.status == 0)
            ok = res.status == 0
            assert rel(res.r[ok], ref[ok]).max() < 1e-8, (mode, onchip, rel(res.r, ref).max())
    for kk in (4, 8, 12, 14):
        orc = np.array([lanczos.lanczos_pair(g, int(a), int(b), k_max=kk)["r"] for a, b in zip(s, t)])
        res = G.query(s, t, mode="fp64", k_max=kk, fixed_k=True, onchip=False)
        m = res.iters == kk
        assert m.any()
        assert rel(res.r[m], orc[m]).max() < 1e-8, (kk, rel(res.r[m], orc[m]).max())


@pytest.mark.parametrize("mode,tol,hist_tol", [("fp64", FP64_TOL, 1e-11), ("fp32", FP32_TOL, 2e-5)])
def test_cluster_whole_recurrence_vs_oracle(rd, mode, tol, hist_tol):
    """Small graphs and few pairs: each pair's whole recurrence runs on a thread-block cluster
    (CTAs holding slices of the vectors, reading each other's through distributed shared
    memory). Against the dense pseudo-inverse or the grid closed form at convergence, the
    oracle's r_k at fixed k, and the one-CTA kernel; a vertex count that no cluster size
    divides, weights, and a heavy row (star centre) included."""
    star = F.star(900)
    cases = [("grid64", W.grid64()[0], np.array([0], np.int32), np.array([4095], np.int32)),
             ("rc1000ln", F.random_connected(1000, 3000, 5, "lognormal"), None, None),
             ("grid37del", F.grid_deleted(37, 0.05, 2), None, None),
             ("star900", star, np.array([3, 10, 0], np.int32), np.array([500, 899, 7], np.int32))]
    for name, g, s, t in cases:
        if s is None:
            s, t = F.random_pairs(g.n, 3, 11)
        ref = (np.array([CF.grid_r(64, 64, 0, 4095)]) if name == "grid64" else dense.DenseRD.of(g).r(s, t))
        G = rd.Graph.from_csr(g)
        kw = dict(mode=mode, k_max=600, rel_tol=0.0, resid_tol=1e-11 if mode == "fp64" else 1e-6)
        res = G.query(s, t, **kw)
        ctas = G.last_stats()["onchip_ctas"]
        assert ctas > 1, (name, ctas)
        assert np.all(res.status == 0), (name, res.status)
        assert rel(res.r, ref).max() < tol, (name, ctas, rel(res.r, ref).max())
        one = G.query(s, t, cluster=False, **kw)
        assert G.last_stats()["onchip_ctas"] == 1
        assert rel(res.r, one.r).max() < tol, name
        k = 12
        orc = [lanczos.lanczos_pair(g, int(a), int(b), k_max=k) for a, b in zip(s, t)]
        fk = G.query(s, t, mode=mode, k_max=k, fixed_k=True)
        assert G.last_stats()["onchip_ctas"] > 1
        # pairs that run all k steps match the oracle's r_k; pairs that break down earlier (the
        # star's Krylov spaces are tiny) hold the exact value, T_i being exact at breakdown
        ko = np.array([o["k"] for o in orc])
        ro = np.array([o["r"] for o in orc])
        m = (fk.iters == k) & (ko == k)
        if m.any():
            assert rel(fk.r[m], ro[m]).max() < hist_tol, (name, rel(fk.r[m], ro[m]).max())
        b = fk.iters < k
        if b.any():
            assert rel(fk.r[b], ref[b]).max() < tol, (name, fk.iters, rel(fk.r[b], ref[b]).max())
        assert m.any() or b.all(), (name, fk.iters, ko)
        assert np.array_equal(G.query(s, t, mode=mode, k_max=k, fixed_k=True).r, fk.r)  # deterministic


def test_scaling_by_four_is_bitwise(rd):
    g = F.grid_deleted(30, 0.05, 5)
    s, t = F.random_pairs(g.n, 8, 3)
    G1 = rd.Graph.from_csr(g)
    G4 = rd.Graph(g.row_ptr, g.col, (4.0 * g.w).astype(np.float32))
    for mode in ["fp64", "fp32"]:
        # the same kernel configuration on both graphs (the autotuner could time them apart)
        r1 = G1.query(s, t, mode=mode, k_max=40, fixed_k=True, tune=False).r
        r4 = G4.query(s, t, mode=mode, k_max=40, fixed_k=True, tune=False).r
        assert np.array_equal(r4 * 4.0, r1)


def test_symmetry_in_s_t(rd):
    g = F.random_connected(200, 400, 12, "lognormal")
    s, t = F.random_pairs(g.n, 16, 5)
    G = rd.Graph.from_csr(g)
    a = G.query(s, t, mode="fp64", rel_tol=0.0, resid_tol=1e-12).r
    b = G.query(t, s, mode="fp64", rel_tol=0.0, resid_tol=1e-12).r
    assert rel(a, b).max() < 1e-10


# grad_w_out is float32 by the ABI, so even the FP64 path is compared at FP32 output precision
@pytest.mark.parametrize("mode,tol", [("fp64", 1e-6), ("fp32", 2e-4)])
def test_edge_grad_vs_dense(rd, mode, tol):
    g = F.random_connected(120, 260, 31, "lognormal")
    s, t = F.random_pairs(g.n, 6, 9)
    gbar = np.linspace(-1.0, 2.0, 6)
    D = dense.DenseRD.of(g)
    ref = D.edge_grad(s, t, gbar)
    G = rd.Graph.from_csr(g)
    gw, r = G.edge_grad(s, t, gbar, mode=mode, k_max=400, rel_tol=0.0,
                        resid_tol=1e-13 if mode == "fp64" else 1e-6)
    assert rel(r, D.r(s, t)).max() < (FP64_TOL if mode == "fp64" else FP32_TOL)
    scale = np.abs(ref).max()
    assert np.abs(gw - ref).max() / scale < tol, np.abs(gw - ref).max() / scale


def test_potential_vs_dense(rd):
    g = F.random_connected(90, 200, 13, "uniform")
    s, t = F.random_pairs(g.n, 4, 6)
    D = dense.DenseRD.of(g)
    G = rd.Graph.from_csr(g)
    phi, r = G.potential(s, t, mode="fp64", rel_tol=0.0, resid_tol=1e-13)
    for p in range(4):
        ref = D.potential(int(s[p]), int(t[p]))
        got = phi[p].astype(np.float64)
        # defined up to a constant: compare edge differences
        rows = g.rows()
        d_ref = ref[rows] - ref[g.col]
        d_got = got[rows] - got[g.col]
        assert np.abs(d_got - d_ref).max() < 1e-6 * np.abs(d_ref).max()


def test_torch_device_io_and_autograd(rd):
    import torch

    g = F.random_connected(100, 220, 19, "uniform")
    s, t = F.random_pairs(g.n, 5, 4)
    G = rd.Graph.from_csr(g)
    sd = torch.from_numpy(s).cuda()
    td = torch.from_numpy(t).cuda()
    res = G.query(sd, td, mode="fp64", rel_tol=0.0, resid_tol=1e-12)
    assert res.r.is_cuda
    ref = dense.DenseRD.of(g).r(s, t)
    assert rel(res.r.cpu().numpy(), ref).max() < FP64_TOL
    w = torch.from_numpy(g.w).cuda().requires_grad_(True)
    opts = dict(mode="fp64", rel_tol=0.0, resid_tol=1e-13)
    r = rd.ResistanceDistance.apply(w, G, sd, td, opts)
    loss = (r * torch.arange(1, 6, device="cuda", dtype=torch.float64)).sum()
    loss.backward()
    refg = dense.DenseRD.of(g).edge_grad(s, t, np.arange(1, 6, dtype=np.float64))
    got = w.grad.cpu().numpy().astype(np.float64)
    assert np.abs(got - refg).max() / np.abs(refg).max() < 1e-6


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_compaction_matches_fixed_layout(rd, mode):
    """Packing converged pairs into narrower blocks changes no pair's result beyond the
    reduction-order rounding of the narrower kernels (which can move a borderline stop
    decision by one step, so both runs are also compared with the oracle)."""
    if mode == "fp64":
        g = F.grid_deleted(60, 0.05, 11)     # distances vary, so pairs stop at different k
        s, t = F.random_pairs(g.n, 200, 13)
        kw = dict(mode=mode, k_max=600, rel_tol=1e-10)
        ref = dense.DenseRD.of(g).r(s, t)
        tol_ab, tol_ref = 1e-8, 1e-8
    else:
        # mean degree 4: the pairs need 10 to 16 steps, so half of them stop while the rest run on
        g, s, t = W.chunglu(20000, 2.1, 4.0, 40000, 200, 31)
        kw = dict(mode=mode, k_max=200, rel_tol=1e-7)
        ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=200, stop_tol=1e-13, threads=0)
        tol_ab, tol_ref = 2e-6, FP32_TOL
    G = rd.Graph.from_csr(g)
    kw["onchip"] = False
    a = G.query(s, t, **kw)
    st = G.last_stats()
    b = G.query(s, t, compact=False, **kw)
    assert st["compactions"] >= 1 and st["device_loop"] == 1
    assert np.abs(a.iters.astype(int) - b.iters.astype(int)).max() <= 1
    assert rel(a.r, b.r).max() < tol_ab
    assert rel(a.r, ref).max() < tol_ref
    # the host-driven loop packs at the same steps: bitwise the same results
    c = G.query(s, t, device_loop=False, **kw)
    assert np.array_equal(c.r, a.r) and np.array_equal(c.iters, a.iters)
    assert G.last_stats()["compactions"] >= st["compactions"]


@pytest.mark.parametrize("mode", ["fp64", "df64"])
def test_async_kernel_8byte_elements(rd, mode):
    """The async row-stream SpMM with two 8-byte elements per 16-byte lane slot (FP64, or
    double-float as hi/lo pairs): on a weighted power-law graph with heavy rows and on a
    weighted road-like grid, every slab width agrees with the oracle at convergence, with the
    row-group kernel at fixed k, and with itself bitwise on a repeat."""
    cl, s_cl, t_cl = W.chunglu(20000, 2.1, 20.0, 200000, 37, 77, weights="lognormal")
    assert np.diff(cl.row_ptr).max() > 256  # heavy rows present
    gd = F.grid_deleted(48, 0.05, 5)
    gd = F.weighted(gd, F.lognormal_edge_weights(gd.m, 0.0, 0.5, 6))
    s_g, t_g = F.random_pairs(gd.n, 21, 8)
    for g, s, t, k_max in ((cl, s_cl, t_cl, 300), (gd, s_g, t_g, 3000)):
        G = rd.Graph.from_csr(g)
        ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=k_max, stop_tol=1e-15, threads=0)
        for tile in [16, 32, 64]:
            kw = dict(mode=mode, kernel="async", rhs_tile=tile, compact=False)
            res = G.query(s, t, k_max=k_max, rel_tol=0.0, resid_tol=1e-11, **kw)
            st = G.last_stats()
            assert st["kernel"] == 5 and st["rhs_tile"] == tile
            assert np.all(res.status >= 0)
            assert rel(res.r, ref).max() < FP64_TOL, (tile, rel(res.r, ref).max())
            fa = G.query(s, t, k_max=20, fixed_k=True, **kw)
            fg = G.query(s, t, mode=mode, kernel="group", rhs_tile=tile, compact=False, k_max=20, fixed_k=True)
            assert rel(fa.r, fg.r).max() < 1e-11, (tile, rel(fa.r, fg.r).max())
            assert np.array_equal(G.query(s, t, k_max=20, fixed_k=True, **kw).r, fa.r)
        G.close()


def test_async_kernel_scattered_heavy_rows(rd):
    """The async kernel's row groups take contiguous shares of the tasks and stream each run of
    light rows between heavy rows without a break; the pre-pass streams runs of contiguous
    chunks. On R-MAT, whose heavy rows are scattered among light ones (not the leading ids as
    in Chung-Lu), every tile width agrees with the oracle and with the row-stream kernel."""
    from graphgen.graph import largest_component

    g = largest_component(F.rmat(15, 16, 0.57, 0.19, 0.19, 12))
    d = np.diff(g.row_ptr)
    heavy = np.nonzero(d > 256)[0]
    assert heavy.size > 10 and np.any(np.diff(heavy) > 1)  # heavy rows present, not contiguous
    s, t = F.random_pairs(g.n, 53, 19)
    G = rd.Graph.from_csr(g)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=300, stop_tol=1e-14, threads=0)
    for tile in [16, 32, 64, 128]:
        kw = dict(mode="fp32", kernel="async", rhs_tile=tile, compact=False)
        res = G.query(s, t, k_max=300, rel_tol=0.0, resid_tol=1e-7, **kw)
        assert G.last_stats()["kernel"] == 5
        assert rel(res.r, ref).max() < FP32_TOL, (tile, rel(res.r, ref).max())
        fa = G.query(s, t, k_max=20, fixed_k=True, **kw)
        fs = G.query(s, t, mode="fp32", kernel="stream", rhs_tile=tile, compact=False, k_max=20, fixed_k=True)
        assert rel(fa.r, fs.r).max() < 2e-6, (tile, rel(fa.r, fs.r).max())


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_flow_kirchhoff_and_dense(rd, mode):
    """Electric flows: f(e) = phi(u) - phi(v) against the dense potential, and Kirchhoff's
    current law: the currents w_e f(e) out of every vertex sum to +1 at s, -1 at t, 0 elsewhere."""
    g = F.random_connected(150, 400, 23, "lognormal")
    s, t = F.random_pairs(g.n, 5, 8)
    G = rd.Graph.from_csr(g)
    f, r = G.flow(s, t, mode=mode, k_max=600, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-6)
    D = dense.DenseRD.of(g)
    rows = g.rows()
    tol = 1e-6 if mode == "fp64" else 1e-4
    for p in range(len(s)):
        phi = D.potential(int(s[p]), int(t[p]))
        ref = phi[rows] - phi[g.col]
        assert np.abs(f[p] - ref).max() < tol * np.abs(ref).max()
        net = np.zeros(g.n)
        np.add.at(net, rows, g.w.astype(np.float64) * f[p].astype(np.float64))
        want = np.zeros(g.n)
        want[s[p]] += 1.0
        want[t[p]] -= 1.0
        assert np.abs(net - want).max() < 10 * tol


def test_power_method_matches_oracle_and_needs_more_steps(rd):
    """Algorithm 1 on the GPU equals the FP64 oracle step by step; on a grid (large
    condition number) it needs many times more steps than the Lanczos iteration to reach
    relative error 1e-6 (the speed-up the paper reports for road networks)."""
    g = F.grid_deleted(30, 0.05, 7)
    s, t = F.random_pairs(g.n, 4, 9)
    G = rd.Graph.from_csr(g)
    steps = 20000
    r, hist = G.power_method(s, t, steps, mode="fp64", history=True)
    for p in range(2):
        ref = power.power_method(g, int(s[p]), int(t[p]), steps)
        assert np.abs(hist[:, p] - ref).max() < 1e-12 * np.abs(ref).max() + 1e-14
    exact = dense.DenseRD.of(g).r(s, t)
    lz = G.query(s, t, mode="fp64", k_max=2000, rel_tol=0.0, resid_tol=1e-12)
    k_lz = np.array([np.argmax(np.abs(lanczos.lanczos_pair(g, int(a), int(b), 300)["r_hist"] / e - 1) <= 1e-6) + 1
                     for a, b, e in zip(s, t, exact)])
    rel_pm = np.abs(hist / exact[None, :] - 1)
    k_pm = np.array([np.argmax(rel_pm[:, p] <= 1e-6) for p in range(len(s))])
    assert np.all(rel_pm[-1] <= 1e-6)
    assert np.all(k_pm > 5 * k_lz), (k_pm, k_lz)
    assert rel(lz.r, exact).max() < 1e-9


def test_triangle_weights_then_weighted_query(rd):
    """Triangle-count weights (the weighted setting of the paper's experiments): each stored
    entry gets the number of triangles through its edge (1 if none), as (A A) o A counts
    them; the weighted query then matches the dense oracle on those weights."""
    import scipy.sparse as sp

    g, s, t = W.chunglu(5000, 2.1, 20.0, 50000, 8, 5)
    G = rd.Graph.from_csr(g)
    w = G.triangle_weights()
    A = sp.csr_matrix((np.ones(g.nnz), g.col, g.row_ptr), shape=(g.n, g.n))
    tri = (A @ A).multiply(A).tocsr()
    tri.sort_indices()
    ref = np.asarray(tri[g.rows(), g.col]).ravel()
    ref = np.where(ref > 0, ref, 1.0)
    assert np.array_equal(w, ref.astype(np.float32))
    k = F.complete(6)
    assert np.all(rd.Graph.from_csr(k).triangle_weights() == 4.0)      # K_6: n - 2 triangles per edge
    gw = g.with_weights(w)
    G.set_weights(w)
    res = G.query(s, t, mode="fp64", rel_tol=0.0, resid_tol=1e-12)
    assert rel(res.r, dense.DenseRD.of(gw).r(s, t)).max() < FP64_TOL


@pytest.mark.parametrize("family", ["er", "ba"])
def test_er_ba_workloads_vs_dense(rd, family):
    """Erdos-Renyi and Barabasi-Albert graphs (the scalability and density experiments):
    converged queries against the dense oracle, fixed k = 20 against the oracle's rhat_20."""
    import math

    n = 1500
    g = F.erdos_renyi(n, int(n * math.log(n)), 4) if family == "er" else F.barabasi_albert(n, 7, 4)
    s, t = F.random_pairs(g.n, 20, 6)
    G = rd.Graph.from_csr(g)
    ref = dense.DenseRD.of(g).r(s, t)
    for mode, tol in [("fp64", FP64_TOL), ("fp32", FP32_TOL)]:
        res = G.query(s, t, mode=mode, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-6)
        assert rel(res.r, ref).max() < tol
    r20 = G.query(s, t, mode="fp64", k_max=20, fixed_k=True).r
    for p in range(3):
        assert rel([r20[p]], [lanczos.lanczos_pair(g, int(s[p]), int(t[p]), 20)["r"]])[0] < 1e-11


def test_plain_kernels_agree(rd):
    """The single-pair path: warp-per-task SpMV, row-group and row-stream kernels agree."""
    g, s, t = W.chunglu(30000, 2.1, 20.0, 300000, 6, 17)
    G = rd.Graph.from_csr(g)
    out = [G.query(s, t, mode=m, k_max=40, fixed_k=True, plain=True, kernel=k).r
           for m in ["fp64"] for k in ["tuned", "group", "stream", "group_sorted"]]
    assert G.last_stats()["kernel"] == 3 and G.last_stats()["row_order"] == 1
    assert max(rel(o, out[0]).max() for o in out[1:]) < 1e-12
    r32 = G.query(s, t, mode="fp32", k_max=40, fixed_k=True, plain=True).r
    assert rel(r32, out[0]).max() < 2e-5


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-11), ("fp32", 2e-6)])
def test_onchip_path_matches_multikernel_path(rd, mode, tol):
    """Small graphs run as one whole-recurrence kernel (one block per pair); the result equals
    the multi-kernel path's within reduction-order rounding, for plain and weighted graphs with
    heavy rows (a star hub) and tolerance stops."""
    a = F.random_connected(3000, 9000, 41, "lognormal")
    hub = F.star(400)
    ea, eb, wa = a.undirected_edges()
    ha, hb, _ = hub.undirected_edges()
    g = to_csr(3000, np.concatenate([ea, ha]), np.concatenate([eb, hb]),
               np.concatenate([wa, np.ones(ha.size, np.float32)]))
    s, t = F.random_pairs(g.n, 33, 4)
    G = rd.Graph.from_csr(g)
    for kw in [dict(k_max=30, fixed_k=True), dict(k_max=400, rel_tol=1e-9 if mode == "fp64" else 1e-6)]:
        on = G.query(s, t, mode=mode, **kw)
        off = G.query(s, t, mode=mode, onchip=False, **kw)
        assert np.abs(on.iters.astype(int) - off.iters.astype(int)).max() <= 1
        assert rel(on.r, off.r).max() < (tol if "fixed_k" in kw else 50 * tol)
    ref = dense.DenseRD.of(g).r(s, t)
    res = G.query(s, t, mode=mode, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-6)
    assert rel(res.r, ref).max() < (FP64_TOL if mode == "fp64" else FP32_TOL)


def test_workspace_allocation_failure_is_reported(rd):
    """A request whose workspace cannot be allocated returns RD_ERR_OOM and leaves the graph
    usable (allocation failure is the one device fault the library injects on purpose)."""
    g = F.path(200000)
    G = rd.Graph.from_csr(g)
    s1, t1 = np.array([0, 5], np.int32), np.array([7, 99], np.int32)
    before = G.query(s1, t1, mode="fp64", k_max=50, fixed_k=True).r
    big = 1 << 22                      # 4M pairs x 200k rows x 2 blocks x 4 bytes: ~6.4 TB
    s = np.zeros(big, np.int32)
    t = np.ones(big, np.int32)
    with pytest.raises(rd.RDError) as e:
        G.query(s, t, mode="fp32", k_max=4)
    assert e.value.status == rd.RD_ERR_OOM
    after = G.query(s1, t1, mode="fp64", k_max=50, fixed_k=True).r
    assert np.array_equal(before, after)


@pytest.mark.parametrize("mode,tol", [("fp64", FP64_TOL), ("fp32", FP32_TOL)])
def test_autotuner_choice_is_used_and_correct(rd, mode, tol):
    """rd_autotune times the candidates on this graph and keeps the fastest; later queries use
    it (stats say so), agree with the oracle, and with the fixed-rule configuration."""
    g, s, t = W.chunglu(30000, 2.1, 20.0, 300000, 48, 91)
    G = rd.Graph.from_csr(g)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=200, stop_tol=1e-14, threads=0)
    pick = G.autotune(len(s), mode=mode)
    assert pick["kernel"] in ((1, 2, 3) if mode == "fp64" else (1, 2, 3, 5)) and pick["rhs_tile"] >= 8
    res = G.query(s, t, mode=mode, k_max=200, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-7,
                  compact=False)
    st = G.last_stats()
    assert st["tuned"] == 1 and st["rhs_tile"] == pick["rhs_tile"] and st["kernel"] == pick["kernel"]
    assert rel(res.r, ref).max() < tol
    fixed = G.query(s, t, mode=mode, k_max=200, rel_tol=0.0, resid_tol=1e-12 if mode == "fp64" else 1e-7,
                    compact=False, tune=False)
    assert G.last_stats()["tuned"] == 0
    assert rel(fixed.r, ref).max() < tol
    # the single-column path is tuned separately
    one = G.autotune(1, mode=mode, plain=True)
    assert one["rhs_tile"] == 1 and one["kernel"] in (1, 2, 3, 4)
    p = G.query(s[:3], t[:3], mode=mode, plain=True, k_max=200, rel_tol=0.0,
                resid_tol=1e-12 if mode == "fp64" else 1e-7)
    assert G.last_stats()["kernel"] == one["kernel"]
    assert rel(p.r, ref[:3]).max() < tol


def test_autotuner_first_use_and_arguments(rd):
    """A query with default options tunes its width classes on first use (compacting query:
    down to the narrowest tile); explicit tiles bypass the table; bad calls are rejected."""
    g, s, t = W.chunglu(20000, 2.1, 20.0, 200000, 100, 5)
    G = rd.Graph.from_csr(g)
    a = G.query(s, t, k_max=200, rel_tol=1e-6)
    assert G.last_stats()["tuned"] == 1
    b = G.query(s, t, k_max=200, rel_tol=1e-6)
    assert np.array_equal(a.r, b.r)              # same table entry, same summation order
    G.query(s, t, k_max=200, rel_tol=1e-6, rhs_tile=32)
    assert G.last_stats()["tuned"] == 0 and G.last_stats()["rhs_tile"] == 32
    with pytest.raises(rd.RDError) as e:
        G.autotune(16, rhs_tile=16)
    assert e.value.status == rd.RD_ERR_INVALID_ARG
    with pytest.raises(rd.RDError) as e:
        G.autotune(0)
    assert e.value.status == rd.RD_ERR_INVALID_ARG


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_graph_replay_is_bitwise_the_launch_loop(rd, mode):
    """Steps replayed from the captured one-step CUDA graph (step index in device memory),
    and the device-resident loop (a conditional while node repeating the step until every
    pair stops or a column compaction is due), give bitwise the results of launching every
    kernel from the host: compacting query with the error-estimate stop, fixed k, a k_max
    reached with pairs still active, the plain path, and the gradient (potential built
    during the forward steps, or by the replay pass, which must regenerate the forward
    vectors)."""
    g, s, t = W.chunglu(20000, 2.1, 20.0, 200000, 70, 13)
    G = rd.Graph.from_csr(g)
    for kw in (dict(k_max=5, rel_tol=1e-12), dict(k_max=200, rel_tol=1e-7),
               dict(k_max=200, rel_tol=0.0, resid_tol=1e-9), dict(k_max=7, fixed_k=True),
               dict(k_max=200, rel_tol=1e-7, compact=False)):
        a = G.query(s, t, mode=mode, **kw)
        ga = G.last_stats()
        assert ga["device_loop"] == 1 and ga["steps"] <= kw["k_max"], kw
        b = G.query(s, t, mode=mode, graph=False, **kw)
        gb = G.last_stats()
        assert gb["device_loop"] == 0
        assert np.array_equal(a.r, b.r), kw
        assert np.array_equal(a.iters, b.iters) and np.array_equal(a.status, b.status), kw
        # the device loop tests the current count before packing, so it skips a packing after
        # the last pair stopped that the lagged host poll still makes
        assert ga["compactions"] <= gb["compactions"], kw
        c = G.query(s, t, mode=mode, device_loop=False, **kw)  # one-step graph, host-driven
        assert G.last_stats()["device_loop"] == 0
        assert np.array_equal(c.r, b.r) and np.array_equal(c.iters, b.iters), kw
        assert G.last_stats()["compactions"] == gb["compactions"], kw
    pa = G.query(s[:5], t[:5], mode=mode, plain=True, k_max=200, rel_tol=1e-7)
    pb = G.query(s[:5], t[:5], mode=mode, plain=True, k_max=200, rel_tol=1e-7, graph=False)
    assert np.array_equal(pa.r, pb.r) and np.array_equal(pa.iters, pb.iters)
    ga, ra = G.edge_grad(s[:16], t[:16], None, mode=mode, k_max=200, rel_tol=0.0, resid_tol=1e-9)
    gb, rb = G.edge_grad(s[:16], t[:16], None, mode=mode, k_max=200, rel_tol=0.0, resid_tol=1e-9, graph=False)
    assert np.array_equal(ra, rb) and np.array_equal(ga, gb)
    kw = dict(mode=mode, k_max=200, rel_tol=0.0, resid_tol=1e-9, potential_mode="replay")
    ga, ra = G.edge_grad(s[:16], t[:16], None, **kw)
    gb, rb = G.edge_grad(s[:16], t[:16], None, graph=False, **kw)
    assert np.array_equal(ra, rb) and np.array_equal(ga, gb)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=200, stop_tol=1e-14, threads=0)
    assert rel(a.r, ref).max() < 1e-7        # the last query's rel_tol


@pytest.mark.parametrize("family", ["chunglu", "rmat", "ba", "grid_del", "grid"])
def test_error_estimate_stop_meets_rel_tol(rd, family):
    """The rel_tol stop (geometric tail estimate) returns estimates within rel_tol of the
    converged value on the method's workload families, and on fast-mixing graphs stops no
    later than the delayed-sum estimate."""
    from graphgen.graph import largest_component

    if family == "chunglu":
        g, s, t = W.chunglu(30000, 2.1, 20.0, 300000, 32, 41)
    elif family == "rmat":
        g = largest_component(F.rmat(14, 16, 0.57, 0.19, 0.19, 8))
        s, t = F.random_pairs(g.n, 32, 6)
    elif family == "ba":
        g = F.barabasi_albert(8000, 4, 6)
        s, t = F.random_pairs(g.n, 32, 7)
    elif family == "grid_del":
        g = F.grid_deleted(40, 0.05, 11)
        s, t = F.random_pairs(g.n, 16, 8)
    else:
        g = F.grid(48)
        s, t = F.random_pairs(g.n, 16, 9)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=5000, stop_tol=1e-15, threads=0)
    G = rd.Graph.from_csr(g)
    for tol in (1e-4, 1e-6, 1e-8):
        res = G.query(s, t, mode="fp64", k_max=5000, rel_tol=tol)
        assert np.all(res.status == 0)
        assert rel(res.r, ref).max() <= tol, (family, tol, rel(res.r, ref).max())
        if family in ("chunglu", "rmat", "ba"):
            old = G.query(s, t, mode="fp64", k_max=5000, rel_tol=tol, estimate="delayed")
            assert np.all(res.iters <= old.iters)


@pytest.mark.parametrize("kernel", ["tuned", "group", "stream", "tasks"])
def test_double_float_mode_vs_oracle(rd, kernel):
    """RD_MODE_DF64 (vectors as FP32 pairs, FP64-class accuracy on the FP32 units): fixed-k
    estimates equal the FP64 oracle's, converged values equal the dense pseudo-inverse, on
    unweighted and weighted graphs, batched (with compaction and graph replay) and plain."""
    for g in (F.grid_deleted(24, 0.05, 9), F.random_connected(300, 900, 31, "lognormal")):
        s, t = F.random_pairs(g.n, 9, 2)
        G = rd.Graph.from_csr(g)
        plain = kernel == "tasks"
        kw = dict(kernel=kernel, onchip=False, plain=plain)
        for k in (1, 3, 17, 40):
            ref = np.array([lanczos.lanczos_pair(g, int(a), int(b), k_max=k)["r"] for a, b in zip(s, t)])
            res = G.query(s, t, mode="df64", k_max=k, fixed_k=True, **kw)
            assert rel(res.r, ref).max() < 1e-11, (k, rel(res.r, ref).max())
        exact = dense.DenseRD.of(g).r(s, t)
        res = G.query(s, t, mode="df64", k_max=2000, rel_tol=0.0, resid_tol=1e-12, **kw)
        assert np.all(res.status == 0)
        assert rel(res.r, exact).max() < FP64_TOL
        if not plain:
            gb = G.query(s, t, mode="df64", k_max=2000, rel_tol=0.0, resid_tol=1e-12, graph=False, **kw)
            assert np.array_equal(gb.r, res.r)


def test_double_float_mode_batched_chunglu(rd):
    """Batched double-float query with the error-estimate stop, compaction and the tuned
    kernels on a power-law graph: within 1e-9 of the oracle; the other entry points run the
    mode as FP64."""
    # mean degree 4: the pairs need 21 to 27 steps, so most stop while the rest run on packed
    g, s, t = W.chunglu(30000, 2.1, 4.0, 60000, 100, 23)
    G = rd.Graph.from_csr(g)
    ref, _, _ = lanczos.lanczos_batch(g, s, t, k_max=300, stop_tol=1e-15, threads=0)
    res = G.query(s, t, mode="df64", k_max=300, rel_tol=0.0, resid_tol=1e-11)
    st = G.last_stats()
    assert st["compactions"] >= 1 and st["device_loop"] == 1
    assert rel(res.r, ref).max() < FP64_TOL
    # the device loop packs with the fused normalise pass (8-byte elements): bitwise the
    # normalise pass followed by the separate packing of the host-driven loop
    hl = G.query(s, t, mode="df64", k_max=300, rel_tol=0.0, resid_tol=1e-11, device_loop=False)
    assert np.array_equal(hl.r, res.r) and np.array_equal(hl.iters, res.iters)
    r64 = G.query(s, t, mode="fp64", k_max=300, rel_tol=0.0, resid_tol=1e-11).r
    assert rel(res.r, r64).max() < 1e-10
    gd, rd_ = G.edge_grad(s[:4], t[:4], None, mode="df64", k_max=300, rel_tol=0.0, resid_tol=1e-11)
    g6, r6 = G.edge_grad(s[:4], t[:4], None, mode="fp64", k_max=300, rel_tol=0.0, resid_tol=1e-11)
    assert np.array_equal(gd, g6) and np.array_equal(rd_, r6)


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-11), ("df64", 1e-11), ("fp32", 2e-5)])
def test_sparse_first_step_matches_dense_first_step(rd, mode, tol):
    """The first step computed from the sparse start vector (only the rows adjacent to s and
    t) agrees with the SpMM over every row: fixed-k estimates and gradients, converged values
    against the dense pseudo-inverse; on a power-law graph with hub endpoints (hub-hub pairs
    share many neighbours), a grid with adjacent pairs and pairs whose endpoints share one or
    two neighbours, and a weighted graph. Rows not sorted by column, or weights not symmetric
    bit for bit, take the SpMM."""
    cl, s_cl, t_cl = W.chunglu(20000, 2.1, 20.0, 200000, 24, 77)
    hubs = np.argsort(np.diff(cl.row_ptr))[-3:].astype(np.int32)
    s_cl = np.concatenate([s_cl, hubs, hubs[2:], t_cl[:1]]).astype(np.int32)
    t_cl = np.concatenate([t_cl, np.roll(hubs, 1), s_cl[:1], hubs[:1]]).astype(np.int32)
    grid = F.grid(20)
    s_g = np.array([0, 21, 21, 0, 105, 399, 7], np.int32)
    t_g = np.array([1, 42, 23, 399, 106, 398, 7], np.int32)
    wg = F.random_connected(300, 900, 31, "lognormal")
    s_w, t_w = F.random_pairs(wg.n, 12, 4)
    for g, s, t in ((cl, s_cl, t_cl), (grid, s_g, t_g), (wg, s_w, t_w)):
        G = rd.Graph.from_csr(g)
        kw = dict(mode=mode, k_max=9, fixed_k=True, onchip=False)
        a = G.query(s, t, **kw)
        assert G.last_stats()["sparse_first"] == 1
        b = G.query(s, t, sparse_first=False, **kw)
        assert G.last_stats()["sparse_first"] == 0
        nz = s != t
        assert np.all(a.r[~nz] == 0.0) and np.array_equal(a.status, b.status)
        assert rel(a.r[nz], b.r[nz]).max() < tol, (g.name, rel(a.r[nz], b.r[nz]).max())
        ref = np.array([lanczos.lanczos_pair(g, int(x), int(y), k_max=9)["r"] if x != y else 0.0
                        for x, y in zip(s, t)])
        assert rel(a.r[nz], ref[nz]).max() < tol
        conv = G.query(s, t, mode=mode, k_max=3000, rel_tol=0.0, resid_tol=1e-12 if mode != "fp32" else 1e-6)
        assert np.all(conv.status == 0)
        if g.n <= 400 or g is wg:
            exact = dense.DenseRD.of(g).r(s[nz], t[nz])
            assert rel(conv.r[nz], exact).max() < (FP64_TOL if mode != "fp32" else FP32_TOL)
        if mode != "df64":
            gk = dict(mode=mode, k_max=12, fixed_k=True)
            ga, ra = G.edge_grad(s[nz][:8], t[nz][:8], None, **gk)
            gb, rb = G.edge_grad(s[nz][:8], t[nz][:8], None, sparse_first=False, **gk)
            assert rel(ra, rb).max() < tol
            assert np.abs(ga - gb).max() <= 50 * tol * np.abs(gb).max()
    # rows in decreasing column order
    col = grid.col.copy()
    for u in range(grid.n):
        col[grid.row_ptr[u]:grid.row_ptr[u + 1]] = col[grid.row_ptr[u]:grid.row_ptr[u + 1]][::-1]
    G2 = rd.Graph(grid.row_ptr, col, None)
    r2 = G2.query(s_g, t_g, mode="fp64", k_max=3000, rel_tol=0.0, resid_tol=1e-12, onchip=False)
    assert G2.last_stats()["sparse_first"] == 0
    nz = s_g != t_g
    assert rel(r2.r[nz], dense.DenseRD.of(grid).r(s_g[nz], t_g[nz])).max() < FP64_TOL
    # one weight of one direction moved by one ulp
    w = wg.w.copy()
    w[0] = np.nextafter(w[0], np.float32(np.inf))
    G3 = rd.Graph(wg.row_ptr, wg.col, w)
    G3.query(s_w, t_w, mode="fp64", k_max=20, fixed_k=True, onchip=False)
    assert G3.last_stats()["sparse_first"] == 0
    G3.set_weights(wg.w)
    G3.query(s_w, t_w, mode="fp64", k_max=20, fixed_k=True, onchip=False)
    assert G3.last_stats()["sparse_first"] == 1


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-9), ("fp32", 3e-4)])
def test_direct_potential_matches_replay_pass(rd, mode, tol):
    """The potential accumulated during the forward steps (p_i = q_i + lambda_i p_{i-1},
    x += mu_i p_i from the LDL^T factors of I - T_i) equals the replay pass's sum of
    ||b|| z_j q_j: gradients, potentials and flows, at fixed k and converged (pairs stopping
    at different steps), on a weighted power-law graph and on a grid; the direct form needs
    one SpMM step per Lanczos step instead of two."""
    cl, s_cl, t_cl = W.chunglu(20000, 2.1, 20.0, 200000, 24, 5, weights="lognormal")
    gd = F.grid_deleted(40, 0.05, 3)
    s_g, t_g = F.random_pairs(gd.n, 12, 4)
    for g, s, t in ((cl, s_cl, t_cl), (gd, s_g, t_g)):
        G = rd.Graph.from_csr(g)
        for kw in (dict(k_max=11, fixed_k=True),
                   dict(k_max=3000, rel_tol=0.0, resid_tol=1e-10 if mode == "fp64" else 1e-6)):
            ga, ra = G.edge_grad(s, t, None, mode=mode, **kw)
            steps_direct = G.last_stats()["spmm_launches"]
            gb, rb = G.edge_grad(s, t, None, mode=mode, potential_mode="replay", **kw)
            assert np.array_equal(ra, rb)                   # the same forward pass
            assert G.last_stats()["spmm_launches"] > steps_direct
            assert np.abs(ga - gb).max() <= tol * np.abs(gb).max(), (g.name, kw, np.abs(ga - gb).max())
            pa, _ = G.potential(s[:6], t[:6], mode=mode, **kw)
            pb, _ = G.potential(s[:6], t[:6], mode=mode, potential_mode="replay", **kw)
            assert np.abs(pa - pb).max() <= tol * np.abs(pb).max()
            fa, _ = G.flow(s[:6], t[:6], mode=mode, **kw)
            fb, _ = G.flow(s[:6], t[:6], mode=mode, potential_mode="replay", **kw)
            assert np.abs(fa - fb).max() <= tol * np.abs(fb).max()


def test_autotune_in_double_float_mode_on_a_fresh_graph(rd):
    """rd_autotune as the first call in RD_MODE_DF64: the candidates it times read the
    double-float degrees, which it makes itself; the query that follows uses the table."""
    g = F.grid_deleted(40, 0.05, 5)
    s, t = F.random_pairs(g.n, 12, 8)
    G = rd.Graph.from_csr(g)
    cfg = G.autotune(12, mode="df64")
    res = G.query(s, t, mode="df64", k_max=2000, rel_tol=0.0, resid_tol=1e-11)
    assert G.last_stats()["tuned"] == 1 and G.last_stats()["rhs_tile"] == cfg["rhs_tile"]
    assert rel(res.r, dense.DenseRD.of(g).r(s, t)).max() < FP64_TOL


def test_double_float_query_follows_new_weights(rd):
    """rd_graph_set_weights after a double-float query: the next one uses the new degrees."""
    g = F.grid_deleted(40, 0.05, 5)
    s, t = F.random_pairs(g.n, 5, 8)
    G = rd.Graph.from_csr(g)
    kw = dict(mode="df64", k_max=3000, rel_tol=0.0, resid_tol=1e-11)
    G.query(s, t, **kw)
    g2 = F.weighted(g, F.lognormal_edge_weights(g.m, 0.0, 0.7, 91))
    G.set_weights(g2.w)
    res = G.query(s, t, **kw)
    assert rel(res.r, dense.DenseRD.of(g2).r(s, t)).max() < FP64_TOL


@pytest.mark.parametrize("name", ["star700", "chunglu", "path3", "loops"])
def test_new_weights_checked_and_followed(rd, name):
    """rd_graph_set_weights in one pass over the weights: the same answers, bit for bit, as a graph
    created with those weights (rows of one entry up to heavy rows, a first set on an unweighted
    graph, dropped self-loops); asymmetric weights turn the sparse first step off and symmetric
    ones on again; a bad weight is refused and the graph still takes good ones."""
    if name == "chunglu":
        g, s, t = W.chunglu(20000, 2.1, 20.0, 200000, 9, 77)
        assert np.diff(g.row_ptr).max() > 256
    else:
        g = {"star700": lambda: F.star(700), "path3": lambda: F.path(3),
             "loops": lambda: F.random_connected(300, 900, 3, None)}[name]()
        s, t = F.random_pairs(g.n, 4, 3)
    rp, col = g.row_ptr, g.col
    w1, w2 = (F.weighted(g, F.lognormal_edge_weights(g.m, 0.0, 0.5, sd)).w for sd in (4, 5))
    if name == "loops":  # a self-loop at vertex 0, in front of its row
        col = np.concatenate([[0], col]).astype(np.int32)
        rp = rp + (np.arange(rp.size) > 0)
        w1, w2 = (np.concatenate([[1.0], w]).astype(np.float32) for w in (w1, w2))
    kw = dict(mode="fp64", k_max=30, fixed_k=True, onchip=False, tune=False)
    G = rd.Graph(rp, col)
    ref = {k: rd.Graph(rp, col, w).query(s, t, **kw).r for k, w in (("w1", w1), ("w2", w2))}
    for k, w in (("w1", w1), ("w2", w2), ("w1", w1)):
        G.set_weights(w)
        assert np.array_equal(G.query(s, t, **kw).r, ref[k])
        assert G.last_stats()["sparse_first"] == 1
    asym = w2.copy()
    asym[-1] *= 2.0
    G.set_weights(asym)
    G.query(s, t, **kw)
    assert G.last_stats()["sparse_first"] == 0
    for bad in (0.0, -1.0, np.inf, np.nan):
        wb = w2.copy()
        wb[wb.size // 2] = bad
        with pytest.raises(rd.RDError):
            G.set_weights(wb)
    G.set_weights(w2)
    assert np.array_equal(G.query(s, t, **kw).r, ref["w2"])
    assert G.last_stats()["sparse_first"] == 1


@pytest.mark.parametrize("mode", ["fp32", "fp64"])
@pytest.mark.parametrize("pairs", [1, 3, 31, 33, 70])
def test_pair_major_outputs(rd, mode, pairs):
    """The transposed outputs of potentials and flows at the edges of their tiles (128 items by 32
    pairs; vertex and entry counts no multiple of 128; dropped self-loops): each pair's row is the
    one the pair has alone, and every flow is the difference of its two potentials."""
    g = F.random_connected(301, 700, 23, "lognormal")
    rows = np.concatenate([g.rows(), [7, 300]])
    cols = np.concatenate([g.col, [7, 300]])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order].astype(np.int32)
    w = np.concatenate([g.w, [1.0, 1.0]]).astype(np.float32)[order]
    rp = np.zeros(g.n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=g.n), out=rp[1:])
    G = rd.Graph(rp, cols, w)
    assert G.nnz == g.nnz and g.nnz % 128 and g.n % 128
    s, t = F.random_pairs(g.n, pairs, 8)
    kw = dict(mode=mode, k_max=40, fixed_k=True)
    phi, _ = G.potential(s, t, **kw)
    f, _ = G.flow(s, t, **kw)
    # FP32 potentials subtract exactly as the kernel subtracts them; FP64 ones are rounded to
    # float first here (one rounding each, relative to the potential) and after in the kernel
    tol = 0.0 if mode == "fp32" else 3 * 2.0**-24 * np.abs(phi).max()
    assert np.abs(f - (phi[:, rows] - phi[:, cols])).max() <= tol
    assert np.all(f[:, rows == cols] == 0.0)
    for p in {0, pairs // 2, pairs - 1}:
        one, _ = G.potential(s[p:p + 1], t[p:p + 1], **kw)
        # the narrower kernel sums in another order: 40 steps of FP32 (FP64) rounding
        assert np.abs(one[0] - phi[p]).max() < (1e-4 if mode == "fp32" else 1e-6) * np.abs(phi[p]).max()


@pytest.mark.parametrize("mode,tol", [("fp64", FP64_TOL), ("fp32", FP32_TOL)])
@pytest.mark.parametrize("n,extra,pairs", [(2, 0, 1), (33, 40, 1), (129, 300, 3), (257, 500, 40), (513, 6000, 5),
                                           (1025, 1500, 2), (1500, 9000, 90), (4700, 60000, 1)])
def test_whole_recurrence_sizes(rd, mode, tol, n, extra, pairs):
    """The whole-recurrence kernel at the edges of its layouts: one vertex pair, row counts around
    the thread counts and not divisible by the cluster size, sparse graphs that gather from the
    other CTAs and dense ones that keep copies, entries that do not fit in shared memory, one CTA
    per pair; against the dense pseudo-inverse, and repeatable bit for bit."""
    g = F.random_connected(n, extra, 3, "lognormal" if n % 2 else None)
    s, t = F.random_pairs(g.n, pairs, 11)
    G = rd.Graph.from_csr(g)
    kw = dict(mode=mode, k_max=2000, rel_tol=0.0, resid_tol=1e-11 if mode == "fp64" else 1e-6)
    res = G.query(s, t, **kw)
    assert G.last_stats()["onchip_ctas"] >= 1
    assert np.all(res.status == 0)
    assert rel(res.r, dense.DenseRD.of(g).r(s, t)).max() < tol
    assert np.array_equal(G.query(s, t, **kw).r, res.r)
    one = G.query(s, t, cluster=False, **kw)
    assert G.last_stats()["onchip_ctas"] == 1
    assert rel(one.r, res.r).max() < tol


@pytest.mark.parametrize("mode", ["fp32", "fp64"])
@pytest.mark.parametrize("k_max,pairs", [(1, 3), (2, 1), (3, 5), (7, 17), (8, 1), (9, 17), (16, 2), (17, 5), (30, 33)])
def test_potential_passes(rd, mode, k_max, pairs):
    """The potential updated once per pass of kept vectors: bit for bit the update with every step
    (which the launch-per-kernel loop makes), around the pass length, with one pair, pairs that
    need no steps, and pairs that stop inside a pass; gradients and flows follow."""
    g = F.random_connected(301, 700, 23, "lognormal")
    s, t = F.random_pairs(g.n, pairs, 8)
    if pairs > 4:
        t[1] = s[1]
    G = rd.Graph.from_csr(g)
    for kw in (dict(k_max=k_max, fixed_k=True), dict(k_max=k_max, rel_tol=1e-3)):
        kw = dict(kw, mode=mode, tune=False)
        phi, r = G.potential(s, t, **kw)
        phi0, r0 = G.potential(s, t, graph=False, **kw)
        assert np.array_equal(r, r0)
        assert np.array_equal(phi, phi0)
        gw, _ = G.edge_grad(s, t, np.linspace(-1, 1, pairs), **kw)
        gw0, _ = G.edge_grad(s, t, np.linspace(-1, 1, pairs), graph=False, **kw)
        assert np.array_equal(gw, gw0)
    dense_first, _ = G.potential(s, t, sparse_first=False, mode=mode, k_max=k_max, fixed_k=True, tune=False)
    ref, _ = G.potential(s, t, sparse_first=False, graph=False, mode=mode, k_max=k_max, fixed_k=True, tune=False)
    assert np.array_equal(dense_first, ref)


@pytest.mark.parametrize("kernel", ["group", "stream", "async"])
@pytest.mark.parametrize("scale", [1.0, 1e-38, 1e-40, 1e37])
def test_fp64_weights_of_every_size(rd, kernel, scale):
    """FP64 steps take FP32 edge weights exactly from denormals to the largest: on a path the
    resistance is the sum of 1/w."""
    w = (np.array([1.0, 3.0, 20.0, 7.0]) * scale).astype(np.float32)
    assert np.all(w > 0) and np.all(np.isfinite(w))
    G = rd.Graph.from_csr(F.weighted(F.path(5), w))
    ref = np.cumsum(1.0 / w.astype(np.float64))
    s, t = np.zeros(4, np.int32), np.arange(1, 5, dtype=np.int32)
    res = G.query(s, t, mode="fp64", k_max=50, rel_tol=0.0, resid_tol=1e-12, onchip=False, kernel=kernel)
    assert rel(res.r, ref).max() < FP64_TOL


@pytest.mark.parametrize("mode,tol", [("fp32", 2e-5), ("fp64", 1e-11), ("df64", 1e-11)])
@pytest.mark.parametrize("graph", ["grid150w", "tree", "star+path"])
@pytest.mark.parametrize("pairs", [5, 20, 40, 70])
def test_short_row_graphs_match_oracle_history(rd, mode, tol, graph, pairs):
    """Graphs of short rows, where the row pipeline is a candidate of the tuner: rows of one to four
    entries, a tree with some of more than four, a hub among rows of two, at several tile widths;
    whatever kernel the tuner takes has the oracle's r_k after k steps (the bars that
    test_fixed_k_matches_oracle_history sets for it) and repeats bit for bit."""
    if graph == "grid150w":
        g = F.grid_deleted(150, 0.05, 5)
    elif graph == "tree":
        g = F.random_tree(20001, 7)
    else:
        a, b, _ = F.star(700).undirected_edges()
        c, d, _ = F.path(20000).undirected_edges()
        g = to_csr(20699, np.concatenate([a, c + 699]), np.concatenate([b, d + 699]))
    s, t = F.random_pairs(g.n, pairs, 9)
    G = rd.Graph.from_csr(g)
    for k in (2, 12, 25):
        res = G.query(s, t, mode=mode, k_max=k, fixed_k=True)
        ref = np.array([lanczos.lanczos_pair(g, int(a), int(b), k_max=k)["r"] for a, b in zip(s[:5], t[:5])])
        m = res.iters[:5] == k
        assert m.any()
        assert rel(res.r[:5][m], ref[m]).max() < tol, (k, rel(res.r[:5][m], ref[m]).max())
        assert np.array_equal(G.query(s, t, mode=mode, k_max=k, fixed_k=True).r, res.r)


@pytest.mark.parametrize("onchip", [True, False])
@pytest.mark.parametrize("pairs", [5, 70])
def test_arrays_a_copy_takes_but_a_kernel_cannot(rd, onchip, pairs):
    """Device arrays at a byte offset (no kernel may load them) and ids whose own memory receives the
    iteration counts give the results of ordinary arrays."""
    import ctypes as C

    import torch

    g = F.grid_deleted(30, 0.05, 5)
    s, t = F.random_pairs(g.n, pairs, 8)
    G = rd.Graph.from_csr(g)
    kw = dict(mode="fp64", k_max=500, rel_tol=0.0, resid_tol=1e-10, onchip=onchip, tune=False)
    ref = G.query(s, t, **kw)
    o = rd._opts(**kw)

    def dev(x, off):
        """A device copy of x starting `off` bytes past an aligned address."""
        b = torch.zeros(x.nbytes + 16, dtype=torch.uint8, device="cuda")
        b[off:off + x.nbytes] = torch.from_numpy(x.reshape(-1).view(np.uint8).copy()).cuda()
        return b, b.data_ptr() + off

    def host(b, off, like):
        return b[off:off + like.nbytes].cpu().numpy().view(like.dtype)

    s, t = s.astype(np.int32), t.astype(np.int32)
    for oi, oo in ((1, 3), (4, 4), (2, 0)):
        (bs, ps), (bt, pt) = dev(s, oi), dev(t, oi)
        outs = [dev(np.zeros_like(x), oo) for x in (ref.r, ref.iters, ref.err, ref.status)]
        torch.cuda.synchronize()
        st = rd.lib().rd_query(G.handle, ps, pt, pairs, C.byref(o), *(p for _, p in outs), None)
        assert st == 0
        for (b, _), x in zip(outs, (ref.r, ref.iters, ref.err, ref.status)):
            assert np.array_equal(host(b, oo, x), x)
    # iteration counts into s, statuses into t
    (bs, ps), (bt, pt) = dev(s, 0), dev(t, 0)
    (br, pr), (be, pe) = dev(ref.r * 0, 0), dev(ref.err * 0, 0)
    torch.cuda.synchronize()
    assert rd.lib().rd_query(G.handle, ps, pt, pairs, C.byref(o), pr, ps, pe, pt, None) == 0
    assert np.array_equal(host(br, 0, ref.r), ref.r) and np.array_equal(host(be, 0, ref.err), ref.err)
    assert np.array_equal(host(bs, 0, ref.iters), ref.iters) and np.array_equal(host(bt, 0, ref.status), ref.status)
    # potentials and gradients at a byte offset
    kp = dict(mode="fp64", k_max=40, fixed_k=True, tune=False)
    o = rd._opts(**kp)
    phi, r = G.potential(s, t, **kp)
    gr = np.linspace(-1, 1, pairs)
    gw, _ = G.edge_grad(s, t, gr, **kp)
    (bs, ps), (bt, pt), (bg, pg) = dev(s, 2), dev(t, 2), dev(gr, 4)
    (bp, pp), (br, pr), (bw, pw) = dev(phi * 0, 2), dev(r * 0, 4), dev(gw * 0, 1)
    torch.cuda.synchronize()
    assert rd.lib().rd_potential(G.handle, ps, pt, pairs, C.byref(o), pp, pr, None) in (0, 1)
    assert np.array_equal(host(bp, 2, phi.reshape(-1)), phi.reshape(-1)) and np.array_equal(host(br, 4, r), r)
    assert rd.lib().rd_edge_grad(G.handle, ps, pt, pairs, pg, C.byref(o), pw, None, None) in (0, 1)
    assert np.array_equal(host(bw, 1, gw), gw)


@pytest.mark.parametrize("mode", ["fp32", "fp64"])
@pytest.mark.parametrize("n,pairs,weighted,ctas", [(129, 1, True, 4), (130, 3, True, 4), (1000, 9, True, 16),
                                                   (1001, 30, True, 4), (1500, 20, True, 4), (4096, 19, True, 8),
                                                   (4097, 1, True, 16), (2049, 5, False, 16)])
def test_clusters_of_the_planned_size(rd, mode, n, pairs, weighted, ctas):
    """The whole-recurrence kernel runs on the cluster it plans (up to 16 CTAs a pair, 64 rows a CTA, every
    pair's cluster resident at once): the shared memory it asks for beside the vectors stays within its limit."""
    g = F.random_connected(n, 2 * n, 3, "lognormal" if weighted else None)
    s, t = F.random_pairs(g.n, pairs, 11)
    G = rd.Graph.from_csr(g)
    G.query(s, t, mode=mode, k_max=5, fixed_k=True)
    assert G.last_stats()["onchip_ctas"] == ctas


@pytest.mark.parametrize("mode,n,deg,pairs,weighted,ctas", [
    ("fp64", 7500, 6, 64, False, 2), ("fp64", 8001, 28, 70, True, 2),   # copies of q_i do not fit on two CTAs
    ("fp32", 14001, 28, 64, True, 2), ("fp32", 18001, 28, 64, False, 2),
    ("fp32", 6000, 56, 64, True, 2), ("fp32", 9001, 56, 30, True, 4),   # copies fit, the entries do not
    ("fp64", 8400, 56, 80, False, 1), ("fp32", 2500, 28, 300, True, 1), ("fp32", 7000, 28, 80, True, 1)])
def test_small_graphs_whose_entries_do_not_fit_on_chip(rd, mode, n, deg, pairs, weighted, ctas):
    """The whole-recurrence kernels that read the entries from global memory -- with copies of q_i, without, on
    one CTA and on clusters of the planned size -- give what the step kernels give after 30 steps."""
    g = F.random_connected(n, n * (deg // 2 - 1), 3, "lognormal" if weighted else None)
    s, t = F.random_pairs(g.n, pairs, 11)
    G = rd.Graph.from_csr(g)
    kw = dict(mode=mode, k_max=30, fixed_k=True)
    res = G.query(s, t, **kw)
    assert G.last_stats()["onchip_ctas"] == ctas
    ref = G.query(s, t, onchip=False, tune=False, **kw)
    assert G.last_stats()["onchip_ctas"] == 0
    assert rel(res.r, ref.r).max() < (FP64_TOL if mode == "fp64" else FP32_TOL)
    assert np.array_equal(G.query(s, t, **kw).r, res.r)


def test_large_batches_on_a_small_graph(rd):
    """Whole-recurrence batches on both sides of the line above which one launch checks the ids: every pair
    has the answer it has in a small batch, a bad id at any place is refused with the results left as they
    were, and 16 times the pairs take nowhere near 256 times as long."""
    import time

    import torch

    g = F.grid(5)
    G = rd.Graph.from_csr(g)
    kw = dict(mode="fp64", k_max=4, fixed_k=True)
    s0, t0 = (x.astype(np.int32) for x in np.divmod(np.arange(g.n * g.n), g.n))
    ref = np.concatenate([G.query(s0[i:i + 125], t0[i:i + 125], **kw).r for i in range(0, s0.size, 125)])
    seconds = {}
    for P in (1 << 14, (1 << 14) + 1, 1 << 16, 1 << 20):
        i = np.arange(P) % s0.size
        s, t = torch.from_numpy(s0[i]).cuda(), torch.from_numpy(t0[i]).cuda()
        best = np.inf
        for _ in range(3):
            torch.cuda.synchronize()
            at = time.perf_counter()
            r = G.query(s, t, **kw).r
            best = min(best, time.perf_counter() - at)
        seconds[P] = best
        assert G.last_stats()["onchip_ctas"] == 1
        assert np.array_equal(r.cpu().numpy(), ref[i])
    assert seconds[1 << 20] < 48 * seconds[1 << 16], seconds
    import ctypes as C

    o = rd._opts(**kw)
    for P, at in ((512, 511), (1 << 14, 0), ((1 << 14) + 1, 1 << 14), (70001, 4321)):
        i = np.arange(P) % s0.size
        s, t = torch.from_numpy(s0[i]).cuda(), torch.from_numpy(t0[i]).cuda()
        t[at] = g.n if at % 2 else -1
        r = torch.full((P,), 7.0, dtype=torch.float64, device="cuda")
        assert rd.lib().rd_query(G.handle, s.data_ptr(), t.data_ptr(), P, C.byref(o), r.data_ptr(), None, None,
                                 None, rd._stream_ptr()) == rd.RD_ERR_INVALID_ARG
        assert bool((r == 7.0).all())


@pytest.mark.parametrize("onchip", [True, False])
def test_error_estimate_of_long_fixed_runs(rd, onchip):
    """Runs of fixed length that go on long after they have converged: the increments fall through the
    whole range of FP64, and the estimate with them: a number below the run's rounding, or infinite where an
    increment rose (as rho >= 1 gives by definition), never NaN."""
    g = F.grid(16)
    s, t = F.random_pairs(g.n, 9, 8)
    G = rd.Graph.from_csr(g)
    for k in range(400, 2600, 75):
        res = G.query(s, t, mode="fp64", k_max=k, fixed_k=True, onchip=onchip, tune=False)
        assert np.all(res.status == 0) and np.all((res.err == np.inf) | (res.err < 1e-12)), (k, res.err)


def test_device_loop_makes_no_pass_after_the_last_step(rd):
    """A fixed-length query ends in either orientation of the device loop's body, and neither runs a normalise
    pass more than the other: a step costs the same from 2 to 3 steps as from 3 to 4 (with a pass or
    two after the last step they differed by two passes, 1.7 to 1)."""
    import time

    import torch

    G = rd.Graph.from_csr(F.grid(1500), label_components=False)
    s, t = (torch.from_numpy(x.astype(np.int32)).cuda() for x in F.random_pairs(G.n, 64, 8))
    best = {}
    for k in (2, 3, 4):
        ts = []
        for _ in range(25):
            torch.cuda.synchronize()
            at = time.perf_counter()
            G.query(s, t, mode="fp32", k_max=k, fixed_k=True, tune=False)
            ts.append(time.perf_counter() - at)
        best[k] = min(ts[5:])
        assert G.last_stats()["device_loop"] == 1
    assert abs((best[4] - best[3]) - (best[3] - best[2])) < 0.25 * (best[4] - best[2]) / 2, best


@pytest.mark.parametrize("call", ["query", "edge_grad"])
def test_new_weights_keep_the_captured_graphs(rd, call):
    """A call after new weights costs what it costs after the same weights (a step's captured graphs took
    the sum of the degrees as an argument, so every optimiser step captured them anew, at a third of the
    price of the call on a graph this small), and follows them: the results are a fresh graph's."""
    import time

    import torch

    g = F.random_connected(300, 900, 3, None)
    s, t = (torch.from_numpy(x.astype(np.int32)).cuda() for x in F.random_pairs(g.n, 2, 8))
    ws = [torch.from_numpy(F.weighted(g, F.lognormal_edge_weights(g.m, 0.0, 0.5, k)).w).cuda() for k in range(24)]
    kw = dict(mode="fp64", k_max=3 if call == "query" else 9, fixed_k=True, kernel="group")

    def run(G):
        if call == "query":
            return G.query(s, t, onchip=False, **kw).r
        return G.edge_grad(s, t, **kw)[0]

    G = rd.Graph(g.row_ptr, g.col, ws[0])
    median = {}
    for name, seq in (("first", ws[:4]), ("same", [ws[0]] * 24), ("new", ws), ("same again", [ws[0]] * 24)):
        ts = []
        for w in seq:
            G.set_weights(w)
            torch.cuda.synchronize()
            at = time.perf_counter()
            out = run(G)
            ts.append(time.perf_counter() - at)
        median[name] = np.median(ts)
    assert median["new"] < 1.15 * max(median["same"], median["same again"]), median
    G.set_weights(ws[7])
    assert torch.equal(run(G), run(rd.Graph(g.row_ptr, g.col, ws[7])))


@pytest.mark.parametrize("mode,bar", [("fp32", 2e-5), ("fp64", 1e-11), ("df64", 1e-11)])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [1999, 2017, 20033])
def test_row_pipeline_by_name(rd, mode, bar, weighted, n):
    """The row pipeline asked for by its number: rows of one to five entries, of a lane group and one more at
    every tile width, long light rows and heavy ones; vertex counts no multiple of a run or of the rows
    in flight; several slabs. Each tile has the row-group kernel's r_k (the bars that
    test_short_row_graphs_match_oracle_history sets on graphs of this kind) and repeats bit for bit."""
    a, b = [np.arange(n - 1)], [np.arange(1, n)]  # a path, and fans whose hubs lie anywhere in it
    hubs = {7: 2, 201: 3, 411: 6, 621: 7, 801: 14, 1001: 15, 1201: 30, 1403: 31, 1601: 250, 33: 700, n - 1: 300}
    for h, d in hubs.items():
        a.append(np.full(d, h))
        b.append((h + 3 + 2 * np.arange(d)) % n)
    a, b = np.concatenate(a), np.concatenate(b)
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    key = np.unique((lo * n + hi)[lo != hi])
    g = to_csr(n, key // n, key % n)
    if weighted:
        g = F.weighted(g, F.lognormal_edge_weights(g.m, 0.0, 0.5, 6))
    d = np.diff(g.row_ptr)
    assert {1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 252} <= set(d) and (d > 256).sum() == 2
    s, t = F.random_pairs(g.n, 75, 9)
    G = rd.Graph.from_csr(g)
    for tile in (16, 32, 64, 128):
        if tile == 128 and mode != "fp32":
            with pytest.raises(rd.RDError) as e:
                G.query(s, t, mode=mode, kernel="pipe", rhs_tile=tile, k_max=2, onchip=False)
            assert e.value.status == rd.RD_ERR_UNSUPPORTED
            continue
        for sparse_first in (True, False):
            kw = dict(mode=mode, rhs_tile=tile, k_max=8, fixed_k=True, compact=False, onchip=False,
                      sparse_first=sparse_first)
            res = G.query(s, t, kernel="pipe", **kw)
            st = G.last_stats()
            assert st["kernel"] == 6 and st["rhs_tile"] == tile and st["ld"] == -(-75 // tile) * tile
            assert rel(res.r, G.query(s, t, kernel="group", **kw).r).max() < bar
            assert np.array_equal(G.query(s, t, kernel="pipe", **kw).r, res.r)
    one = G.query(s[:1], t[:1], mode=mode, kernel="pipe", k_max=8, fixed_k=True, onchip=False)
    assert G.last_stats()["kernel"] == 4 and rel(one.r, res.r[:1]).max() < bar


def test_tuner_names_the_row_pipeline(rd):
    """Where the tuner takes the row pipeline its number comes back, and asking for that configuration runs it."""
    G = rd.Graph.from_csr(F.grid_deleted(400, 0.05, 5))
    s, t = F.random_pairs(G.n, 16, 9)
    for mode in ("fp32", "fp64", "df64"):
        pick = G.autotune(16, mode=mode)
        again = G.query(s, t, mode=mode, k_max=10, fixed_k=True, kernel=pick["kernel"], rhs_tile=pick["rhs_tile"],
                        rows_per_warp=pick["rows_per_warp"])
        st = G.last_stats()
        assert (st["kernel"], st["rhs_tile"], st["rows_per_warp"]) == tuple(pick[k] for k in ("kernel", "rhs_tile",
                                                                                           "rows_per_warp"))
        assert np.array_equal(again.r, G.query(s, t, mode=mode, k_max=10, fixed_k=True).r)
        assert G.last_stats()["kernel"] == pick["kernel"]


def test_narrow_queries_hold_no_packing_space(rd):
    """A query of up to 16 columns never packs them, and its workspace holds no blocks to pack into: one pair
    on a large graph takes a few vectors, 16 and 17 pairs what their blocks need."""
    import torch

    g = F.grid(2000)
    G = rd.Graph.from_csr(g, label_components=False)
    n4 = 4.0 * g.n
    s, t = F.random_pairs(g.n, 17, 8)
    used = 0.0
    for pairs, columns in ((1, 2), (16, 32), (17, 2 * 32 + 2 * 16)):
        free = torch.cuda.mem_get_info()[0]
        G.query(s[:pairs], t[:pairs], mode="fp32", k_max=3, fixed_k=True, tune=False)
        used += free - torch.cuda.mem_get_info()[0]
        # beside the vector blocks: heavy-row sums, the mask of the first pass (a bit a column and row)
        assert used < (columns + (columns + 31) // 32 + 1) * n4 + 64e6, (pairs, used / n4)


def test_kept_vectors_give_way_to_the_calls_outputs(rd):
    """Flows handed out in host memory with little device memory left: the vectors kept for a pass are given
    up, in the plan (they may take a quarter of what would be free) or once the staged output does not
    fit, and the call succeeds with the same flows; with room for them they are kept."""
    import torch

    g = F.random_connected(400_000, 4_400_000, 3, None)
    s, t = F.random_pairs(g.n, 32, 8)
    kw = dict(mode="fp32", k_max=9, fixed_k=True, kernel="group", rhs_tile=32)
    G = rd.Graph.from_csr(g, label_components=False)
    ref, r = G.flow(s, t, **kw)
    passes = G.last_stats()["launches"]
    G.close()
    # in vector blocks: 2 for the steps, 2 for the potential, 7 more for kept vectors; the flows 24
    block = 4 * g.n * 32
    assert 23.9 < 4 * g.nnz * 32 / block < 24.1
    torch.cuda.synchronize()
    for left, kept in ((30, False), (33, False), (60, True)):
        G = rd.Graph.from_csr(g, label_components=False)
        torch.cuda.empty_cache()
        hog = torch.empty(int(torch.cuda.mem_get_info()[0] - left * block - 8 * g.nnz - 16e6), dtype=torch.uint8,
                          device="cuda")
        f, r2 = G.flow(s, t, **kw)
        assert np.array_equal(f, ref) and np.array_equal(r2, r), left
        assert (G.last_stats()["launches"] == passes) == kept, left
        del hog
        G.close()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("call", ["potential", "edge_grad", "flow"])
def test_pass_calls_poll_as_asked(rd, call):
    """Runs of fixed length end soon after every pair has ended (here: broken down in the first pass, or, without
    deflation, lost definiteness in the fifteenth), not at k_max, and chunk_steps sets the
    steps between polls, rounded up to passes of 8; the outputs are those of the launch-per-kernel loop."""
    side = np.repeat(np.arange(4), 4)  # complete bipartite: pairs on one side break down exactly at once
    G = rd.Graph.from_csr(to_csr(8, side, 4 + np.tile(np.arange(4), 4)))
    s, t = np.array([0, 1, 0, 4, 6], np.int32), np.array([1, 2, 3, 5, 7], np.int32)
    kw = dict(mode="fp64", kernel="group")
    out, _ = getattr(G, call)(s, t, k_max=20000, fixed_k=True, **kw)
    assert G.last_stats()["steps"] <= 32
    ref, _ = getattr(G, call)(s, t, k_max=40, fixed_k=True, graph=False, **kw)
    assert np.array_equal(out, ref)
    h = F.grid(20)
    H = rd.Graph.from_csr(h)
    s, t = F.random_pairs(h.n, 5, 8)
    lost = dict(mode="fp32", kernel="group", fixed_k=True, deflate=False)
    last = int(H.query(s, t, k_max=20000, onchip=False, **lost).iters.max())
    assert 16 < last < 400
    out, _ = getattr(H, call)(s, t, k_max=20000, **lost)
    assert H.last_stats()["steps"] <= last + 3 * 8
    ref, _ = getattr(H, call)(s, t, k_max=last + 40, graph=False, **lost)
    assert np.array_equal(out, ref, equal_nan=True)
    kw = dict(kw, k_max=4000, rel_tol=0.0, resid_tol=1e-10)
    ref, _ = getattr(H, call)(s, t, **kw)
    needed = H.last_stats()["steps"]  # within a pass of the last pair's
    assert needed % 8 == 0 and 32 < needed < 400
    for chunk in (1, 8, 9, 64, 100):
        out, _ = getattr(H, call)(s, t, chunk_steps=chunk, **kw)
        every = -(-chunk // 8) * 8
        assert H.last_stats()["steps"] == -(-needed // every) * every
        assert np.array_equal(out, ref)


def test_mirrors_give_way_to_a_workspace(rd):
    """A weighted graph's mirrors (4 bytes an entry, to check new weights by) are given back when a query's
    workspace does not fit beside them; new weights are then searched for their mirrors and followed."""
    import torch

    g = F.random_connected(300_000, 6_000_000, 3, "lognormal")
    w2 = F.weighted(g, F.lognormal_edge_weights(g.m, 0.0, 0.5, 9)).w
    s, t = F.random_pairs(g.n, 64, 8)
    kw = dict(mode="fp32", k_max=5, fixed_k=True, kernel="group", rhs_tile=64, compact=False)
    ref = {}
    G = rd.Graph.from_csr(g, label_components=False)
    free = torch.cuda.mem_get_info()[0]
    ref["w"] = G.query(s, t, **kw).r
    need = free - torch.cuda.mem_get_info()[0]
    G.set_weights(w2)
    ref["w2"] = G.query(s, t, **kw).r
    G.close()
    mirrors = 4 * g.nnz
    assert need > mirrors > 40e6
    G = rd.Graph.from_csr(g, label_components=False)
    torch.cuda.empty_cache()
    hog = torch.empty(int(torch.cuda.mem_get_info()[0] - need + mirrors / 2), dtype=torch.uint8, device="cuda")
    assert np.array_equal(G.query(s, t, **kw).r, ref["w"])
    G.set_weights(w2)
    assert np.array_equal(G.query(s, t, **kw).r, ref["w2"])
    assert G.last_stats()["sparse_first"] == 1
    bad = w2.copy()
    bad[-1] *= 2.0
    G.set_weights(bad)
    G.query(s, t, **kw)
    assert G.last_stats()["sparse_first"] == 0
    del hog
    torch.cuda.empty_cache()


@pytest.mark.parametrize("mode", ["fp32", "fp64"])
def test_power_method_row_order(rd, mode):
    """The Power Method visits rows by degree where they differ in length and several columns share them, and in
    their own order on grids, where neighbours belong together, and for one column; the estimates are the
    oracle's."""
    for g, by_degree in ((F.grid_deleted(40, 0.05, 5), 0), (F.random_connected(900, 9000, 3, None), 1),
                         (F.star(700), 1)):
        G = rd.Graph.from_csr(g)
        s, t = F.random_pairs(g.n, 6, 8)
        r, hist = G.power_method(s, t, 12, mode=mode, history=True)
        assert G.last_stats()["row_order"] == by_degree
        for p in range(6):
            one, h1 = G.power_method(s[p:p + 1], t[p:p + 1], 12, mode=mode, history=True)
            assert G.last_stats()["row_order"] == 0
            ref = power.power_method(g, int(s[p]), int(t[p]), 12)
            assert np.abs(hist[:, p] - ref).max() < (1e-11 if mode == "fp64" else 1e-5) * np.abs(ref).max()
            assert np.abs(h1[:, 0] - ref).max() < (1e-11 if mode == "fp64" else 1e-5) * np.abs(ref).max()
