"""GPU parity at the full sizes of the five synthetic workloads, in the launch configuration
the benchmark uses: sampled outputs against the FP64 oracle, and properties that hold at
any size where the oracle cannot run to convergence.

These generate large graphs (seconds to minutes of host time) and are marked slow as well.
"""
import numpy as np
import pytest

from graphgen import families as F
from graphgen import workloads as W
from graphgen.graph import to_csr
from oracle import dense, lanczos
from tests import closed_forms as CF

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

FP64_TOL = 1e-9
FP32_TOL = 1e-5


@pytest.fixture(scope="module")
def rd():
    import torch

    assert torch.cuda.is_available()
    import paper_2601_11159_gb300 as rd

    rd.lib()
    return rd


def rel(a, b):
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    return np.abs(a - b) / np.abs(b)


def test_chunglu1m_256_pairs_bench_configuration(rd):
    """Chung-Lu n=1M, 256 pairs, FP32 vectors, estimated relative error 1e-6: 24 sampled pairs
    against the oracle run to a 1e-13 relative increment; plain path on 4 of them."""
    import torch

    g, s, t = W.chunglu1m()
    G = rd.Graph.from_csr(g)
    res = G.query(torch.from_numpy(s).cuda(), torch.from_numpy(t).cuda(), mode="fp32", k_max=200, rel_tol=1e-6)
    r = res.r.cpu().numpy()
    assert np.all(res.status.cpu().numpy() == 0)
    idx = np.arange(0, 256, 11)[:24]
    ref, _, _ = lanczos.lanczos_batch(g, s[idx], t[idx], k_max=200, stop_tol=1e-13, threads=0)
    e = rel(r[idx], ref)
    assert e.max() < 1e-6, e.max()            # the accuracy the workload asks for
    plain = G.query(s[idx[:4]], t[idx[:4]], mode="fp32", k_max=200, rel_tol=1e-6, plain=True)
    assert rel(plain.r, ref[:4]).max() < FP32_TOL


def test_roadgrid4096_fp64(rd):
    """4096^2 grid, 5% edges deleted, weights U[0.5, 2], 64 pairs at distance 1000, FP64.
    (a) Fixed k = 100: the GPU estimate equals the oracle's rhat_100 on two sampled pairs.
    (b) Run to relative residual 1e-8: every pair converges; Rayleigh bound (the graph is a
        subgraph of the full grid with weights <= 2, so r >= r_unit_grid / 2); the Gauss
        estimate only grows with k; r(s,t) = r(t,s)."""
    g, s, t = W.roadgrid4096()
    G = rd.Graph.from_csr(g)
    k = 100
    r100 = G.query(s, t, mode="fp64", k_max=k, fixed_k=True).r
    pick = np.array([0, 37])
    ref, _, _ = lanczos.lanczos_batch(g, s[pick], t[pick], k_max=k, stop_tol=0.0, threads=0)
    assert rel(r100[pick], ref).max() < FP64_TOL
    # long runs (about 17,000 steps) to convergence on 4 of the 64 pairs (all 64 share the code
    # path; a full 64-pair FP64 run takes minutes on this part's FP64 rate)
    res = G.query(s[:4], t[:4], mode="fp64", k_max=40000, rel_tol=0.0, resid_tol=1e-7)
    assert np.all(res.status == 0), np.unique(res.status)
    assert np.all(res.r >= r100[:4] * (1 - 1e-12))
    old = g.meta["lcc_old_id"]
    lower = np.array([CF.grid_r(4096, 4096, int(old[a]), int(old[b])) / 2.0 for a, b in zip(s[:4], t[:4])])
    assert np.all(res.r >= lower)
    back = G.query(t[:1], s[:1], mode="fp64", k_max=40000, rel_tol=0.0, resid_tol=1e-7)
    assert rel(back.r, res.r[:1]).max() < 1e-6


def test_grid4096_unit_converged_vs_closed_form(rd, capsys):
    """Large-kappa parity at full size against an exact reference: the undeleted unit-weight
    4096^2 grid (kappa ~ 1.4e7, the road-grid workload before deletion and weighting), 8 pairs
    at Manhattan distance 1000, run to relative residual 1e-10 in FP64 and in double-float
    vectors, against the exact spectral sum (an O(N^2) FP64 sum per pair) at 1e-9 relative.
    The FP32-vector path is run too and stays within its documented floor (about 2e-4 at
    this kappa)."""
    g = F.grid(4096)
    s, t = F.grid_distance_pairs(g, 8, 1000, 13)
    ref = np.array([CF.grid_r(4096, 4096, int(a), int(b)) for a, b in zip(s, t)])
    G = rd.Graph.from_csr(g)
    errs = {}
    for mode in ("fp64", "df64"):
        res = G.query(s, t, mode=mode, k_max=60000, rel_tol=0.0, resid_tol=1e-10)
        assert np.all(res.status == 0), (mode, np.unique(res.status))
        errs[mode] = (rel(res.r, ref).max(), int(res.iters.max()))
        assert errs[mode][0] < FP64_TOL, (mode, errs[mode])
    r32 = G.query(s, t, mode="fp32", k_max=60000, rel_tol=0.0, resid_tol=1e-6)
    errs["fp32"] = (rel(r32.r, ref).max(), int(r32.iters.max()))
    assert errs["fp32"][0] < 1e-3, errs["fp32"]
    with capsys.disabled():
        print(f"\ngrid4096 unit, 8 pairs at distance 1000: max rel. error / steps {errs}")


def test_roadgrid1024_converged_vs_oracle(rd, capsys):
    """Converged parity on a road-like grid small enough for the CPU oracle: 1024^2, 5% of the
    edges deleted, weights U[0.5, 2] (kappa ~ 1e6), 8 pairs at distance 256, against the FP64
    oracle run to a 1e-13 relative increment (stored by tests/golden/make_roadgrid1024_ref.py,
    which also checks two of the pairs against Jacobi-CG to 1e-9). FP64 and double-float
    vectors to relative residual 1e-12 within 1e-9; FP32 vectors within 1e-3 (their floor)."""
    import json
    import os
    import sys

    sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden"))
    import make_roadgrid1024_ref as M

    ref_doc = json.load(open(M.OUT))
    g, s, t = M.graph_and_pairs()
    assert M.checksum(g) == ref_doc["graph"]["sha1"], "the generator no longer makes the stored graph"
    assert s.tolist() == ref_doc["pairs"]["s"] and t.tolist() == ref_doc["pairs"]["t"]
    ref = np.array(ref_doc["oracle"]["r"])
    G = rd.Graph.from_csr(g)
    errs = {}
    for mode in ("fp64", "df64"):
        res = G.query(s, t, mode=mode, k_max=60000, rel_tol=0.0, resid_tol=1e-12)
        assert np.all(res.status == 0), (mode, np.unique(res.status))
        errs[mode] = (rel(res.r, ref).max(), int(res.iters.max()))
        assert errs[mode][0] < FP64_TOL, (mode, errs[mode])
    for mode, kw in (("fp32", dict(rel_tol=0.0, resid_tol=1e-6)), ("fp32 rel_tol 1e-6", dict(rel_tol=1e-6))):
        r32 = G.query(s, t, mode="fp32", k_max=60000, **kw)
        errs[mode] = (rel(r32.r, ref).max(), int(r32.iters.max()))
        assert errs[mode][0] < 1e-3, (mode, errs[mode])
    res = G.query(s, t, mode="df64", k_max=60000, rel_tol=1e-6)
    errs["df64 rel_tol 1e-6"] = (rel(res.r, ref).max(), int(res.iters.max()))
    assert errs["df64 rel_tol 1e-6"][0] < 1e-5
    with capsys.disabled():
        print(f"\nroadgrid1024, 8 pairs at distance 256: max rel. error / steps {errs}")


def test_chunglu4m_weighted_gradient(rd):
    """Chung-Lu n=4M, exponent 2.3, lognormal(0, 0.5) weights, 32 pairs: r on sampled pairs
    (FP32 and FP64); the edge gradient against (i) the oracle's potential gradient on sampled
    entries, (ii) central finite differences on 100 random edges, (iii) the dense
    pseudo-inverse gradient on a 2,000-vertex subgraph."""
    g, s, t = W.chunglu4m_w()
    G = rd.Graph.from_csr(g)
    idx = np.array([0, 9, 21, 30])
    ref, _, _ = lanczos.lanczos_batch(g, s[idx], t[idx], k_max=200, stop_tol=1e-13, threads=0)
    r32 = G.query(s, t, mode="fp32", k_max=200, rel_tol=1e-7).r
    r64 = G.query(s, t, mode="fp64", k_max=200, rel_tol=0.0, resid_tol=1e-12).r
    assert rel(r32[idx], ref).max() < FP32_TOL
    assert rel(r64[idx], ref).max() < FP64_TOL
    # the device-resident loop packs the columns where the host polls do: a step here moves
    # more than 1.5 GB, so both read the current active count, and the last packing leaves
    # one active pair (a one-column layout, which the fused normalise-and-pack cannot take)
    a = G.query(s, t, mode="fp32", k_max=200, rel_tol=1e-6)
    sa = G.last_stats()
    b = G.query(s, t, mode="fp32", k_max=200, rel_tol=1e-6, device_loop=False)
    sb = G.last_stats()
    assert sa["device_loop"] == 1 and sb["device_loop"] == 0
    assert np.array_equal(a.r, b.r) and np.array_equal(a.iters, b.iters)
    assert sa["compactions"] == sb["compactions"] >= 1, (sa["compactions"], sb["compactions"])

    # (i) one-hot upstream gradient on pair 0 vs the oracle potential of pair 0
    onehot = np.zeros(s.size)
    onehot[0] = 1.0
    gw, _ = G.edge_grad(s, t, onehot, mode="fp64", k_max=200, rel_tol=0.0, resid_tol=1e-12)
    orc = lanczos.lanczos_pair(g, int(s[0]), int(t[0]), k_max=60, stop_tol=1e-15, want_potential=True)
    phi = orc["phi"]
    rng = np.random.default_rng(3)
    ent = rng.choice(g.nnz, 300, replace=False)
    rows = np.searchsorted(g.row_ptr, ent, side="right") - 1
    gref = -0.5 * (phi[rows] - phi[g.col[ent]]) ** 2
    # include the largest entries (those touching s and t) as well
    for v in (int(s[0]), int(t[0])):
        e = np.arange(g.row_ptr[v], g.row_ptr[v + 1])
        ent = np.concatenate([ent, e[:20]])
        gref = np.concatenate([gref, -0.5 * (phi[v] - phi[g.col[e[:20]]]) ** 2])
    scale = np.abs(gref).max()
    assert np.abs(gw[ent] - gref).max() / scale < 1e-5

    # (ii) central finite differences on 100 random edges, objective sum_p r_p (FP64)
    ones = np.ones(s.size)
    gall, _ = G.edge_grad(s, t, ones, mode="fp64", k_max=200, rel_tol=0.0, resid_tol=1e-13)
    a, b, wu = g.undirected_edges()
    pick = rng.choice(a.size, 100, replace=False)
    base_w = g.w.copy()
    for j in pick[:100]:
        u, v = int(a[j]), int(b[j])
        e1 = g.row_ptr[u] + np.searchsorted(g.col[g.row_ptr[u]:g.row_ptr[u + 1]], v)
        e2 = g.row_ptr[v] + np.searchsorted(g.col[g.row_ptr[v]:g.row_ptr[v + 1]], u)
        h = 1e-3 * float(base_w[e1])
        vals = []
        for sign in (+1.0, -1.0):
            w2 = base_w.copy()
            w2[e1] += sign * h
            w2[e2] += sign * h
            G.set_weights(w2)
            vals.append(G.query(s, t, mode="fp64", k_max=200, rel_tol=0.0, resid_tol=1e-13).r.sum())
        fd = (vals[0] - vals[1]) / (2 * h)
        adj = float(gall[e1]) + float(gall[e2])
        assert abs(fd - adj) <= 1e-4 * abs(adj) + 1e-9, (u, v, fd, adj)
    G.set_weights(base_w)

    # (iii) 2,000-vertex BFS ball, induced subgraph, dense pseudo-inverse gradient
    start = int(rng.integers(g.n))
    seen = {start}
    frontier = [start]
    order = [start]
    while frontier and len(order) < 2000:
        nxt = []
        for u in frontier:
            for v in g.col[g.row_ptr[u]:g.row_ptr[u + 1]]:
                v = int(v)
                if v not in seen and len(order) < 2000:
                    seen.add(v)
                    order.append(v)
                    nxt.append(v)
        frontier = nxt
    keep = np.zeros(g.n, bool)
    keep[order] = True
    ra = g.rows()
    sel = keep[ra] & keep[g.col] & (ra < g.col)
    new = np.full(g.n, -1)
    new[np.array(sorted(order))] = np.arange(len(order))
    sub = to_csr(len(order), new[ra[sel]], new[g.col[sel]], g.w[sel])
    from graphgen.graph import largest_component

    sub = largest_component(sub)
    ss, tt = F.random_pairs(sub.n, 6, 2)
    D = dense.DenseRD.of(sub)
    S = rd.Graph.from_csr(sub)
    gs, _ = S.edge_grad(ss, tt, None, mode="fp64", k_max=2000, rel_tol=0.0, resid_tol=1e-13)
    gd = D.edge_grad(ss, tt)
    assert np.abs(gs - gd).max() / np.abs(gd).max() < 1e-6


def test_rmat24_batched_and_plain(rd):
    """R-MAT scale 24, edge factor 16, (0.57, 0.19, 0.19), 128 pairs in one batched query
    (FP32 vectors): 8 sampled pairs against the oracle; the plain one-pair path on the same
    pairs agrees with the batch."""
    g, s, t = W.rmat24()
    G = rd.Graph.from_csr(g)
    res = G.query(s, t, mode="fp32", k_max=200, rel_tol=1e-6)
    assert np.all(res.status == 0)
    idx = np.arange(0, 128, 16)
    ref, _, _ = lanczos.lanczos_batch(g, s[idx], t[idx], k_max=200, stop_tol=1e-13, threads=0)
    assert rel(res.r[idx], ref).max() < 1e-6
    plain = G.query(s[idx], t[idx], mode="fp32", k_max=200, rel_tol=1e-6, plain=True)
    assert rel(plain.r, res.r[idx]).max() < 2e-6


def test_entry_counts_up_to_the_limit(rd):
    """2^31 - 8 stored entries (a clique of 46,341 vertices with a path behind it, whose rows hold the
    last entries): a kernel that steps past a row's end must not wrap round. Pairs near the path's end
    have after three steps, without deflation, the r_k of a short path, whatever kernel is asked for."""
    import torch

    k, m = 46341, 20850
    n = k + m
    row = torch.arange(k - 1, dtype=torch.int32, device="cuda")
    col = (row[None, :] + (row[None, :] >= torch.arange(k, dtype=torch.int32, device="cuda")[:, None])).int().view(-1)
    v = torch.arange(k, n, dtype=torch.int32, device="cuda")
    path = torch.stack([v - 1, v + 1], 1).view(-1)[:-1]  # the last vertex has one neighbour
    one = torch.tensor([k], dtype=torch.int32, device="cuda")  # the clique's last vertex meets the path
    col = torch.cat([col, one, path])
    deg = torch.full((n,), 2, dtype=torch.int64, device="cuda")
    deg[:k] = k - 1
    deg[k - 1] += 1
    deg[-1] = 1
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(deg, 0)
    nnz = int(rp[-1])
    assert nnz == col.numel() == 2**31 - 8
    G = rd.Graph(rp, col, label_components=False)
    del col
    short = F.path(200)
    S = rd.Graph.from_csr(short)
    off = np.arange(1, 18)
    to = (off + 1) % 4
    kw = dict(k_max=3, fixed_k=True, deflate=False, sparse_first=False, onchip=False, tune=False)
    ref = S.query((199 - off).astype(np.int32), (199 - to).astype(np.int32), mode="fp64", **kw).r
    s, t = (n - 1 - off).astype(np.int32), (n - 1 - to).astype(np.int32)
    for kernel in ("group", "group_sorted", "stream", "async", "pipe"):
        for mode, tol in (("fp64", 1e-12), ("fp32", 1e-5), ("df64", 1e-11)):
            r = G.query(s, t, mode=mode, kernel=kernel, **kw).r
            assert rel(r, ref).max() < tol, (kernel, mode)
            # the row-stream kernels leave the last 1,024 entries of the range to the row-group kernel
            assert G.last_stats()["kernel"] == {"group_sorted": 3, "pipe": 6}.get(kernel, 1)
    one = G.query(s[:1], t[:1], mode="fp64", kernel="tasks", **kw).r
    assert rel(one, ref[:1]).max() < 1e-12


def test_blocks_past_32_bit_row_offsets(rd):
    """A path of 2^24 + 4,096 vertices with 4 KB of a vector block to a row (1,024 FP32 or 512 FP64
    columns): the last rows start 2^32 16-byte units and more into a block. Pairs near the path's end have after three
    steps, without deflation, the r_k of a short path, whatever kernel is asked for."""
    import torch

    n = 2**24 + 4096
    torch.cuda.empty_cache()
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    col = torch.stack([v - 1, v + 1], 1).view(-1)[1:-1].contiguous()  # the ends have one neighbour
    rp = torch.arange(n + 1, dtype=torch.int64, device="cuda") * 2 - 1
    rp[0], rp[-1] = 0, 2 * n - 2
    assert col.numel() == 2 * n - 2
    G = rd.Graph(rp, col, label_components=False)
    S = rd.Graph.from_csr(F.path(200))
    kw = dict(k_max=3, fixed_k=True, deflate=False, sparse_first=False, onchip=False, tune=False)
    for mode, columns, tol in (("fp32", 1024, 1e-5), ("fp64", 512, 1e-12), ("df64", 512, 1e-11)):
        off = 1 + np.arange(columns) % 17
        to = (off + 1) % 4
        ref = S.query((199 - off[:17]).astype(np.int32), (199 - to[:17]).astype(np.int32), mode="fp64", **kw).r
        ref = ref[np.arange(columns) % 17]
        s, t = (n - 1 - off).astype(np.int32), (n - 1 - to).astype(np.int32)
        for kernel in ("group", "stream", "async"):
            r = G.query(s, t, mode=mode, kernel=kernel, rhs_tile=64, **kw).r
            assert rel(r, ref).max() < tol, (kernel, mode)
            assert G.last_stats()["kernel"] == 1
