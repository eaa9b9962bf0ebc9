// Per-step vector and per-pair scalar kernels of the batched Lanczos iteration:
// start vector (Algorithm 3), FP64 finalisation of alpha/beta with an O(1)-per-step
// LDL^T update of I - T_k (the quadratic form of Section 3), normalisation
// v_{i+1} = w / beta_{i+1} (Algorithm 3), output, the tridiagonal solve for the
// potential of Algorithm 5 and the edge-weight gradient.
#include <math.h>

#include <algorithm>

#include "scalars.cuh"
#include "spmm.cuh"

namespace rd {

// ----------------------------------------------------------------- start
// q_1 = D^{-1/2} v_1 with v_1 = (e_s/sqrt(d_s) - e_t/sqrt(d_t)) / ||b||, so
// q_1[s] = 1/(d_s ||b||), q_1[t] = -1/(d_t ||b||); ||b||^2 = 1/d_s + 1/d_t.
template <typename T>
__global__ void k_init(const InitArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.npairs) return;
    const PairState& st = a.st;
    const int32_t s = a.s[p], t = a.t[p];
    if (a.replay) {
        if (st.status[p] == RD_OK || st.status[p] == RD_WARN_NOT_CONVERGED) {
            if (s != t && st.b2[p] > 0.0) {
                const double ds = a.deg64[s], dt = a.deg64[t];
                const double bn = sqrt(1.0 / ds + 1.0 / dt);
                T* q = static_cast<T*>(a.qcur);
                q[(int64_t)s * a.ld + p] = (T)(1.0 / (ds * bn));
                q[(int64_t)t * a.ld + p] = (T)(-1.0 / (dt * bn));
            }
        }
        return;
    }
    if (s < 0 || (int64_t)s >= a.n || t < 0 || (int64_t)t >= a.n) {
        atomicOr(a.err_flag, 1);
        st.status[p] = RD_ERR_INVALID_ARG;
        st.r[p] = NAN;
        return;
    }
    if (s == t) {
        st.status[p] = RD_OK;
        st.r[p] = 0.0;
        st.err[p] = 0.0;
        return;
    }
    if (a.comp && a.comp[s] != a.comp[t]) {
        st.status[p] = RD_ERR_DISCONNECTED;
        st.r[p] = INFINITY;
        return;
    }
    const double ds = a.deg64[s], dt = a.deg64[t];
    const double b2 = 1.0 / ds + 1.0 / dt;
    const double bn = sqrt(b2);
    T* q = static_cast<T*>(a.qcur);
    q[(int64_t)s * a.ld + p] = (T)(1.0 / (ds * bn));
    q[(int64_t)t * a.ld + p] = (T)(-1.0 / (dt * bn));
    st.b2[p] = b2;
    st.bnorm[p] = bn;
    st.err[p] = 1.0;
    st.status[p] = RD_OK;
    st.active[p] = 1;
    atomicAdd(&st.act_count[0], 1);
}

void launch_init(cudaStream_t st, const InitArgs& a)
{
    const int nb = (a.npairs + 127) / 128;
    if (a.df) k_init<df64><<<nb, 128, 0, st>>>(a);
    else if (a.elem_size == 8) k_init<double><<<nb, 128, 0, st>>>(a);
    else k_init<float><<<nb, 128, 0, st>>>(a);
}

// -------------------------------------------------------------- finalise
// Column p: reduce the SpMM block partials in block order, then
//   alpha_i = <w, v_i>, beta_{i+1}^2 = ||w||^2 - alpha_i^2 - gamma^2 (gamma: component along
//   D^{1/2}1, removed when deflating), and update the LDL^T factorisation of J_i = I - T_i:
//   delta_1 = 1 - alpha_1,  delta_i = (1 - alpha_i) - beta_i^2 / delta_{i-1}
//   g_1 = 1,                g_i = beta_i g_{i-1} / delta_{i-1}        (g = L^{-1} e_1)
//   S_i = S_{i-1} + g_i^2 / delta_i = e_1^T J_i^{-1} e_1,   r_i = ||b||^2 S_i
//   residual ||b - (I - Ahat) x_i|| / ||b|| = beta_{i+1} |g_i / delta_i|.
// Step i = j + 1 of pair p from the three reduced sums A = <w, v_i>, B = ||w||^2 and
// C = <w, D^{1/2}1> of w = Ahat v_i - beta_i v_{i-1}:
//   alpha_i = A, beta_{i+1}^2 = B - A^2 - C^2/sum(d) (deflated component removed),
//   LDL^T of J_i = I - T_i: delta_1 = 1 - alpha_1, delta_i = (1 - alpha_i) - beta_i^2/delta_{i-1},
//   g_1 = 1, g_i = beta_i g_{i-1}/delta_{i-1}, S_i = S_{i-1} + g_i^2/delta_i, r_i = ||b||^2 S_i,
//   residual ||b - (I - Ahat) x_i||/||b|| = beta_{i+1} |g_i/delta_i|.
// Writes the pair's state and history; returns true when the pair stops (then active = 0),
// else leaves alpha_i, the deflation constant c_i and beta_{i+1} in the outputs.
// The per-pair scalars of the update (a register copy of one pair's PairState entries).
struct PairScalars {
    double b2, delta, g, S, beta;  // beta: beta_i of the step being reduced
    double inv_delta;              // 1 / delta (0 before the first step)
    double r0, r1, r2, r3;         // increments of S: slot j % kRing holds step j's
    // slot access by a run-time index through selects, so that the scalars stay in registers
    // (an indexed array would live in local memory)
    __device__ __forceinline__ double ring(int q) const { return q == 0 ? r0 : (q == 1 ? r1 : (q == 2 ? r2 : r3)); }
    __device__ __forceinline__ void set_ring(int q, double v)
    {
        r0 = q == 0 ? v : r0;
        r1 = q == 1 ? v : r1;
        r2 = q == 2 ? v : r2;
        r3 = q == 3 ? v : r3;
    }
};
static_assert(kRing == 4, "PairScalars holds four ring slots");

// What one step produced (the values pair_update stores).
struct PairStepOut {
    bool ok;                       // false: a value was not finite or I - T_i lost definiteness
    bool warn_not_converged;       // k_max reached before a tolerance was met
    double alpha, cdef, beta_next, incr, gd, r, est;
};

__device__ __forceinline__ PairScalars pair_load(const PairState& st, int p, int64_t np)
{
    PairScalars s;
    s.b2 = st.b2[p];
    s.delta = st.delta[p];
    s.g = st.g[p];
    s.S = st.S[p];
    s.beta = st.beta[p];
    s.inv_delta = st.inv_delta[p];
    s.r0 = st.ring[p];
    s.r1 = st.ring[np + p];
    s.r2 = st.ring[2 * np + p];
    s.r3 = st.ring[3 * np + p];
    return s;
}

// Finite: tested on the exponent bits (an FP64 comparison would occupy the FP64 unit).
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// What the next vector needs of the three sums: alpha_i, the deflation constant c_i,
// beta_{i+1}^2, beta_{i+1} and 1/beta_{i+1}.
struct StepCoef {
    double alpha, cdef, beta2, beta, inv_beta;
};

// The chain between the sums and the next vector.
__device__ __forceinline__ StepCoef step_coef(const FinArgs& a, double inv_sumdeg, double A, double B, double C)
{
    StepCoef k;
    k.alpha = A;
    k.cdef = a.deflate ? C * inv_sumdeg : 0.0;
    const double gamma2 = a.deflate ? C * k.cdef : 0.0;
    const double b2 = B - A * A - gamma2;
    k.beta2 = b2;
    root_and_inverse(b2, &k.beta, &k.inv_beta);
    return k;
}

// The rest of one step on the scalars (see pair_update): the LDL^T factors, the estimate and the
// stop tests; returns true when the pair stops. The state in `s` is advanced exactly as
// pair_update advances the stored state. Divisions are what this chain is made of, so
// 1/delta_{i-1} is kept from the previous step, 1/sum(d) is passed in, 1/delta_i serves every
// quotient by it, and the estimate is one quotient (tail_estimate).
__device__ __forceinline__ bool pair_core(const FinArgs& a, PairScalars& s, int j, const StepCoef& k, PairStepOut& o)
{
    const double alpha = k.alpha;
    const double beta_i = s.beta;
    double delta, g;
    if (j == 0) {
        delta = 1.0 - alpha;
        g = 1.0;
    } else {
        const double idp = s.inv_delta;
        delta = (1.0 - alpha) - beta_i * beta_i * idp;
        g = s.g * beta_i * idp;
    }
    bool stop = false;
    o.ok = finite64(alpha) && finite64(k.beta2) && finite64(delta) && delta > 0.0;
    o.warn_not_converged = false;
    o.alpha = alpha;
    o.cdef = k.cdef;
    o.beta_next = 0.0;
    o.gd = 0.0;
    if (!o.ok) return true;  // frozen at its last good estimate
    const double inv_delta = 1.0 / delta;
    const double gd = g * inv_delta;
    const double incr = g * gd;
    const double S = s.S + incr;
    s.S = S;
    o.incr = incr;
    o.gd = gd;
    o.r = s.b2 * S;
    s.set_ring(j % kRing, incr);
    const double beta_next = k.beta;
    o.beta_next = beta_next;
    const double resid = beta_next * fabs(gd);
    s.delta = delta;
    s.inv_delta = inv_delta;
    s.g = g;
    const double brk = a.fp64 ? 1e-12 : 1e-6;
    const bool breakdown = beta_next <= brk * (fabs(alpha) + beta_i);  // T_i is exact
    stop = breakdown || (!a.fixed_k && a.resid_tol > 0.0 && resid <= a.resid_tol);
    // Relative error estimate of r_k = b2 * S_k: the increments still to come. Default:
    // their sum as a series whose ratio is the largest of the last kRing-1 increment
    // ratios (at least 1/2), with an extra margin 1/(1 - rho) for slowly converging
    // pairs: incr * rho / (1 - rho)^2. Alternative (est_delayed): the sum of the last
    // kRing increments, i.e. the error of the estimate kRing steps back. Without a rel_tol
    // test it only feeds the output, so it is formed on the step that ends the pair.
    const bool use_est = !a.fixed_k && a.rel_tol > 0.0;
    double est = 0.0;
    if (!breakdown && (use_est || stop || j + 1 >= a.k_max)) {
        if (!a.est_delayed && j + 1 >= kRing) {
            est = tail_estimate(s.ring(j % kRing), s.ring((j - 1) % kRing), s.ring((j - 2) % kRing),
                                s.ring((j - 3) % kRing), S);
        } else {
            double tail = 0.0;
            const int nr = j + 1 < kRing ? j + 1 : kRing;
            for (int q = 0; q < nr; ++q) tail += s.ring(q);
            est = tail / S;
        }
        if (!stop && use_est && j + 1 >= kRing && est <= a.rel_tol) stop = true;
    }
    o.est = est;
    if (!stop && j + 1 >= a.k_max) {
        stop = true;
        o.warn_not_converged = !a.fixed_k;
    }
    if (!stop) s.beta = beta_next;
    return stop;
}

// Store one step's results of pair p (the history, the running factorisation, the status).
__device__ __forceinline__ void pair_store(const PairState& st, int p, int j, int64_t np, const PairScalars& s,
                                           const PairStepOut& o, bool stop)
{
    if (!o.ok) {
        st.status[p] = RD_ERR_NUMERIC;
    } else {
        st.S[p] = s.S;
        st.r[p] = o.r;
        st.ring[(int64_t)(j % kRing) * np + p] = o.incr;
        st.err[p] = o.est;
        st.hist_alpha[(int64_t)j * np + p] = o.alpha;
        st.hist_beta[(int64_t)(j + 1) * np + p] = o.beta_next;
        st.k[p] = j + 1;
        st.delta[p] = s.delta;
        st.inv_delta[p] = s.inv_delta;
        st.g[p] = s.g;
        if (o.warn_not_converged) st.status[p] = RD_WARN_NOT_CONVERGED;
    }
    if (stop) st.active[p] = 0;
    else st.beta[p] = s.beta;
}

// One step of pair p on the stored state: writes the pair's state and history; returns true when
// the pair stops (then active = 0). `k` and `o` receive the step's coefficients and results.
__device__ __forceinline__ bool pair_update(const FinArgs& a, const PairState& st, int p, int j, double isd, double A, double B,
                                            double C, StepCoef& k, PairStepOut& o)
{
    PairScalars s = pair_load(st, p, a.pstride);
    k = step_coef(a, isd, A, B, C);
    const bool stop = pair_core(a, s, j, k, o);
    pair_store(st, p, j, a.pstride, s, o, stop);
    return stop;
}

// Columns per finalize block: 8 (one 64-byte segment of the block partials), or the next power
// of two >= ld for narrower tiles; the other threads of the block split the sum over the SpMM
// blocks. The kernel is bound by latency (a few dozen dependent loads and FP64 operations), so
// the sum is spread wide: 64 columns and 608 partials took 12 us on 2 blocks of 32 columns.
__host__ __device__ inline int fin_cols_per_block(int64_t ld)
{
    int cb = 1;
    while (cb < ld && cb < 8) cb <<= 1;
    return cb;
}

// In the device-resident loop (a.loop) the last block also decides how the loop goes on after
// step j (the step's count of active pairs is then complete), advances the step index and
// sets the index the step's normalise pass reads: the body of a step is then three or four
// kernels (pre-pass, SpMM, finalize, normalise) with no single-thread kernels between them.
// The test for a column compaction before step j + 1 reads the count `lag` steps back, as
// rd_query's host polls do, so that both pack the columns at the same step; when one is due, the
// step's normalise pass is left to the host, which runs it fused with the packing. To stop, record
// j (or j + 1 when nothing is left to do), the count the test read, the count entering the next
// step and which of the two it is in saved[0..3], and park both indices at the sentinel
// k_max + 1, whose active count is always 0, so that the remaining kernels of the body return: the
// normalise pass of this step too, whose vector nobody reads, and with it that of the body's other
// orientation (64 FP32 columns of a 1500^2 grid: 0.27 ms each).
template <typename T>
__global__ void __launch_bounds__(256) k_finalize(const FinArgs a)
{
    __shared__ double part[3][256];
    const int cb = fin_cols_per_block(a.ld);
    const int nsplit = 256 / cb;
    const int lane = threadIdx.x & (cb - 1), split = threadIdx.x / cb;
    const int64_t col = (int64_t)blockIdx.x * cb + lane;
    const PairState& st = a.st;
    const int j = a.step_dev ? *a.step_dev : a.step;  // 0-based step index; Lanczos step i = j + 1
    if (st.act_count[j] == 0) {
        // the step's normalise pass has nothing to do either
        if (a.loop == 2 && blockIdx.x == 0 && threadIdx.x == 0) *a.loop_norm = a.k_max + 1;
        return;
    }
    const double isd = __ldg(a.inv_sumdeg);
    // block partials b = split, split + nsplit, ...: four rows of loads in flight, summed
    // in block order (the order depends only on nblocks and ld, so runs are repeatable)
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (col < a.ld) {
        const int64_t slab = col / a.tp, cin = col % a.tp;
        const double* base = a.block_part + slab * a.nblocks * 3 * a.tp + cin;
        const int64_t bstride = 3 * (int64_t)a.tp;
        for (int b = split; b < a.nblocks; b += 4 * nsplit) {
            double x[4][3];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (b + u * nsplit < a.nblocks) {
                    const double* bp = base + (int64_t)(b + u * nsplit) * bstride;
                    x[u][0] = bp[0];
                    x[u][1] = bp[a.tp];
                    x[u][2] = bp[2 * a.tp];
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (b + u * nsplit < a.nblocks) {
                    s0 += x[u][0];
                    s1 += x[u][1];
                    s2 += x[u][2];
                }
            }
        }
    }
    part[0][threadIdx.x] = s0;
    part[1][threadIdx.x] = s1;
    part[2][threadIdx.x] = s2;
    __syncthreads();
    // fixed-order tree over the splits; the three sums go to different warps
    for (int w = 128; w >= cb; w >>= 1) {
        for (int i = threadIdx.x; i < 3 * w; i += 256) part[i / w][i % w] += part[i / w][i % w + w];
        __syncthreads();
    }
    const int p = split != 0 || col >= a.ld
                      ? -1
                      : (a.slot_pair ? a.slot_pair[col] : (col < a.npairs ? (int)col : -1));
    if (p >= 0 && st.active[p]) {
        const double A = part[0][lane], B = part[1][lane], C = part[2][lane];
        const int64_t ld = a.ld;
        const int64_t cfo = a.step_dev ? (int64_t)j * a.cf_stride : 0;
        T* cfs = static_cast<T*>(a.cf_step) + cfo;
        T* cfn = static_cast<T*>(a.cf_next) + cfo;
        // factors of the previous step, for the potential's direct update below
        const double lam = a.xcf && j > 0 ? st.beta[p] * st.inv_delta[p] : 0.0;
        StepCoef k;
        PairStepOut o;
        const bool stop = pair_update(a, st, p, j, isd, A, B, C, k, o);
        if (a.xcf && o.ok) {
            // p_i = q_i + lambda_i p_{i-1}, x += mu_i p_i (a stopping step still contributes)
            T* xc = static_cast<T*>(a.xcf) + (int64_t)j * 2 * ld;
            xc[col] = (T)lam;
            xc[ld + col] = (T)(st.bnorm[p] * o.gd);
        }
        if (stop) {
            // zero coefficients: the column's vectors become (and stay) zero
            cfs[1 * ld + col] = T(0);
            cfs[2 * ld + col] = T(0);
            cfs[3 * ld + col] = T(0);
            cfn[col] = T(0);
        } else {
            cfs[1 * ld + col] = (T)k.alpha;
            cfs[2 * ld + col] = (T)k.cdef;
            cfs[3 * ld + col] = (T)k.inv_beta;
            cfn[col] = (T)k.beta;
            atomicAdd(&st.act_count[j + 1], 1);
        }
    }
    if (!a.loop) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (atomicAdd(a.loop_ticket, 1) != (int)gridDim.x - 1) return;
    *a.loop_ticket = 0;
    __threadfence();
    const volatile int32_t* act_count = st.act_count;
    const int jn = j + 1;
    if (a.loop == 2) {
        *a.loop_norm = j;
        *a.loop_step = jn;
        return;
    }
    const int act = act_count[jn];
    const int act_lag = act_count[jn >= a.loop_lag ? jn - a.loop_lag : 0];
    const bool more = act > 0 && jn < a.k_max;
    const bool compact_due = a.loop_compact && jn >= a.loop_lag + 1 && jn >= *a.loop_cfrom && a.ld > 16 &&
                             (int64_t)act_lag * 2 <= a.ld;
    const bool pack = more && compact_due;
    *a.loop_norm = pack || !more ? a.k_max + 1 : j;
    *a.loop_step = more && !pack ? jn : a.k_max + 1;
    if (pack || !more) {
        a.loop_saved[0] = pack ? j : jn;
        a.loop_saved[1] = act_lag;
        a.loop_saved[2] = act;
        a.loop_saved[3] = pack ? 1 : 0;
    }
    cudaGraphSetConditional((cudaGraphConditionalHandle)a.loop_handle, more && !pack ? 1 : 0);
}

void launch_finalize(cudaStream_t st, const FinArgs& a)
{
    const int cb = fin_cols_per_block(a.ld);
    const int nb = (int)((a.ld + cb - 1) / cb);
    if (a.df) k_finalize<df64><<<nb, 256, 0, st>>>(a);
    else if (a.elem_size == 8) k_finalize<double><<<nb, 256, 0, st>>>(a);
    else k_finalize<float><<<nb, 256, 0, st>>>(a);
}

// ------------------------------------------------------------- normalise
// One element of q_{i+1} = (W - alpha_i q_i - c_i) * (1/beta_{i+1}); every normalise kernel
// forms it this way, so that the packed form (k_normalize_pack) equals the plain one bit for bit.
template <typename T>
__device__ __forceinline__ T lanczos_next(T w, T al, T qc, T c, T ib)
{
    return (w - al * qc - c) * ib;
}
template <>
__device__ __forceinline__ float lanczos_next<float>(float w, float al, float qc, float c, float ib)
{
    return __fmul_rn(__fsub_rn(__fmaf_rn(-al, qc, w), c), ib);
}
template <>
__device__ __forceinline__ double lanczos_next<double>(double w, double al, double qc, double c, double ib)
{
    return __dmul_rn(__dsub_rn(__fma_rn(-al, qc, w), c), ib);
}

// q_{i+1} = (W - alpha_i q_i - c_i) / beta_{i+1}, written over W; optionally
// phi += coef * q_i for the replay pass. 16-byte units; ld == 1 handled separately.
template <typename T, bool LD1>
__global__ void __launch_bounds__(256) k_normalize(const NormArgs<T> a)
{
    const int32_t* act = a.step_dev ? a.act_count + *a.step_dev : a.active_prev;
    if (act && *act == 0) return;
    const T* cfb = a.step_dev ? a.cf + (int64_t)(*a.step_dev) * a.cf_stride : a.cf;
    constexpr int V = 16 / (int)sizeof(T);
    const int64_t total = a.n * a.ld;
    const int64_t units = total / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t ld = a.ld;
    const T* cf_al = cfb + ld;
    const T* cf_c = cfb + 2 * ld;
    const T* cf_ib = cfb + 3 * ld;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < units; u += stride) {
        const int64_t e0 = u * V;
        T w[V], qc[V], qn[V];
        ld_stream<T, V>(w, a.w_to_qnext + e0);
        ld_stream<T, V>(qc, a.qcur + e0);
        if constexpr (LD1) {
            const T al = cf_al[0], c = cf_c[0], ib = cf_ib[0];
#pragma unroll
            for (int i = 0; i < V; ++i) qn[i] = lanczos_next<T>(w[i], al, qc[i], c, ib);
            if (a.phi) {
                const T cf = a.coef[0];
                T ph[V];
                ld_plain<T, V>(ph, a.phi + e0);
#pragma unroll
                for (int i = 0; i < V; ++i) ph[i] += cf * qc[i];
                st_plain<T, V>(a.phi + e0, ph);
            }
        } else {
            const int64_t c0 = e0 % ld;
            T al[V], c[V], ib[V];
            ld_plain<T, V>(al, cf_al + c0);
            ld_plain<T, V>(c, cf_c + c0);
            ld_plain<T, V>(ib, cf_ib + c0);
#pragma unroll
            for (int i = 0; i < V; ++i) qn[i] = lanczos_next<T>(w[i], al[i], qc[i], c[i], ib[i]);
            if (a.phi) {
                T cf[V], ph[V];
                ld_plain<T, V>(cf, a.coef + c0);
                ld_plain<T, V>(ph, a.phi + e0);
#pragma unroll
                for (int i = 0; i < V; ++i) ph[i] += cf[i] * qc[i];
                st_plain<T, V>(a.phi + e0, ph);
            }
        }
        st_plain<T, V>(a.w_to_qnext + e0, qn);
    }
    if constexpr (LD1) {
        // scalar tail (ld == 1 and n not a multiple of V)
        const int64_t t0 = units * V;
        for (int64_t e = t0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
            const T w = a.w_to_qnext[e], qc = a.qcur[e];
            a.w_to_qnext[e] = lanczos_next<T>(w, cf_al[0], qc, cf_c[0], cf_ib[0]);
            if (a.phi) a.phi[e] += a.coef[0] * qc;
        }
    }
}

// q_{i+1} as k_normalize, with the potential of each pair accumulated on the fly: the direct
// form of the Lanczos solve (D-Lanczos, Saad, Iterative Methods for Sparse Linear Systems,
// Section 6.7.1). With I - T_i = L D L^T (unit lower bidiagonal L, L[i][i-1] = -beta_i/delta_{i-1};
// D = diag(delta)) and g = L^{-1} e_1, the vectors P = Q L^{-T} obey p_i = q_i + lambda_i p_{i-1},
// lambda_i = beta_i/delta_{i-1}, and x_i = ||b|| Q_i (I - T_i)^{-1} e_1 = x_{i-1} + mu_i p_i with
// mu_i = ||b|| g_i/delta_i: after the last step x is the potential of the replay pass
// (sum_j ||b|| z_j q_j, z = (I - T_k)^{-1} e_1), without a second pass over the steps.
template <typename T, bool VECD>
__global__ void __launch_bounds__(256) k_normalize_pot(const NormArgs<T> a)
{
    const int32_t* act = a.step_dev ? a.act_count + *a.step_dev : a.active_prev;
    if (act && *act == 0) return;
    const int64_t j = a.step_dev ? *a.step_dev : 0;
    const int64_t ld = a.ld;
    const T* cfb = a.cf + j * a.cf_stride;
    const T* xcb = a.xcf + j * a.xcf_stride;
    const T* cf_al = cfb + ld;
    const T* cf_c = cfb + 2 * ld;
    const T* cf_ib = cfb + 3 * ld;
    const T* cf_lam = xcb;
    const T* cf_mu = xcb + ld;
    constexpr int V = VECD ? 16 / (int)sizeof(T) : 1;
    const int64_t units = a.n * ld / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < units; u += stride) {
        const int64_t e0 = u * V, c0 = e0 % ld;
        T w[V], qc[V], pv[V], xv[V], al[V], c[V], ib[V], lam[V], mu[V];
        ld_stream<T, V>(w, a.w_to_qnext + e0);
        ld_stream<T, V>(qc, a.qcur + e0);
        ld_plain<T, V>(pv, a.pvec + e0);
        ld_plain<T, V>(xv, a.xvec + e0);
        ld_plain<T, V>(al, cf_al + c0);
        ld_plain<T, V>(c, cf_c + c0);
        ld_plain<T, V>(ib, cf_ib + c0);
        ld_plain<T, V>(lam, cf_lam + c0);
        ld_plain<T, V>(mu, cf_mu + c0);
        T qn[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            qn[i] = lanczos_next<T>(w[i], al[i], qc[i], c[i], ib[i]);
            pv[i] = qc[i] + lam[i] * pv[i];
            xv[i] += mu[i] * pv[i];
        }
        st_plain<T, V>(a.pvec + e0, pv);
        st_plain<T, V>(a.xvec + e0, xv);
        st_plain<T, V>(a.w_to_qnext + e0, qn);
    }
}

// The same potential with the vectors of up to kPotSteps steps kept: at the end of a pass its
// vectors are read once, p and x go through registers step by step (the operations and rounding of
// k_normalize_pot), and where the pass is full and pairs go on, the last step's normalise pass is
// made on the way: q_{i+1} and q_i go to blocks 1 and 0, where the next pass starts. Bound by HBM:
// a step streams 3 blocks in its normalise pass and 1 here, plus 4 per pass for p and x (none in
// and no p out where one pass is all), against 7 per step; 32 FP32 columns of a 4M-vertex graph
// (511 MB a block), 8 steps: 4.45 ms with k_normalize_pot and 0.3 ms of zeroing; the call 17.5 ->
// 16.0 ms (18.1 -> 16.6 on another GPU).
template <typename T, bool VECD>
__global__ void __launch_bounds__(256) k_potential_pass(const PotPassArgs<T> a)
{
    constexpr int V = VECD ? 16 / (int)sizeof(T) : 1;
    const int base = *a.base;
    int cnt = 0;
    while (cnt < a.m && base + cnt < a.k_max && a.act_count[base + cnt] > 0) ++cnt;
    if (cnt == 0 && base > 0) return;
    const bool more = cnt == a.m && base + a.m < a.k_max && a.act_count[base + a.m] > 0;
    const int64_t ld = a.ld;
    const int64_t units = a.n * ld / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const T* xcf = a.xcf + (int64_t)base * 2 * ld;
    const T* cf = a.cf + (int64_t)(base + cnt - 1) * 4 * ld;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < units; u += stride) {
        const int64_t e0 = u * V, c0 = e0 % ld;
        T q[kPotSteps][V], pv[V], xv[V];
#pragma unroll
        for (int s = 0; s < kPotSteps; ++s)
            if (s < cnt) ld_stream<T, V>(q[s], a.blocks + (int64_t)(1 + s) * a.stride + e0);
        if (base > 0) {
            ld_stream<T, V>(pv, a.pvec + e0);
            ld_stream<T, V>(xv, a.xvec + e0);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) pv[i] = xv[i] = T(0);
        }
#pragma unroll
        for (int s = 0; s < kPotSteps; ++s)
            if (s < cnt) {
                T lam[V], mu[V];
                ld_plain<T, V>(lam, xcf + (int64_t)s * 2 * ld + c0);
                ld_plain<T, V>(mu, xcf + (int64_t)s * 2 * ld + ld + c0);
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    pv[i] = q[s][i] + lam[i] * pv[i];
                    xv[i] += mu[i] * pv[i];
                }
            }
        st_plain<T, V>(a.xvec + e0, xv);
        if (more) {
            T w[V], al[V], c[V], ib[V], ql[V], qn[V];
            ld_stream<T, V>(w, a.blocks + e0);
            ld_plain<T, V>(al, cf + ld + c0);
            ld_plain<T, V>(c, cf + 2 * ld + c0);
            ld_plain<T, V>(ib, cf + 3 * ld + c0);
#pragma unroll
            for (int s = 0; s < kPotSteps; ++s)
                if (s == cnt - 1)
#pragma unroll
                    for (int i = 0; i < V; ++i) ql[i] = q[s][i];
#pragma unroll
            for (int i = 0; i < V; ++i) qn[i] = lanczos_next<T>(w[i], al[i], ql[i], c[i], ib[i]);
            st_plain<T, V>(a.pvec + e0, pv);
            st_plain<T, V>(a.blocks + e0, ql);
            st_plain<T, V>(a.blocks + a.stride + e0, qn);
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(a.ticket, 1) != (int)gridDim.x - 1) return;
    *a.ticket = 0;
    *a.base = base + a.m;
}

template <typename T>
static void launch_pot_pass(int grid, cudaStream_t st, const PotPassArgs<T>& a)
{
    if (a.ld % (16 / (int64_t)sizeof(T)) == 0) k_potential_pass<T, true><<<grid, 256, 0, st>>>(a);
    else k_potential_pass<T, false><<<grid, 256, 0, st>>>(a);
}
void launch_potential_pass_f32(int grid, cudaStream_t st, const PotPassArgs<float>& a) { launch_pot_pass(grid, st, a); }
void launch_potential_pass_f64(int grid, cudaStream_t st, const PotPassArgs<double>& a) { launch_pot_pass(grid, st, a); }

template <typename T>
static void launch_norm(int grid, cudaStream_t st, const NormArgs<T>& a)
{
    constexpr int V = 16 / (int)sizeof(T);
    if (a.pvec) {
        if (a.ld % V == 0) k_normalize_pot<T, true><<<grid, 256, 0, st>>>(a);
        else k_normalize_pot<T, false><<<grid, 256, 0, st>>>(a);
    } else if (a.ld == 1) {
        k_normalize<T, true><<<grid, 256, 0, st>>>(a);
    } else {
        k_normalize<T, false><<<grid, 256, 0, st>>>(a);
    }
}

__global__ void k_step_advance(int32_t* step, int limit)
{
    if (*step < limit) *step += 1;
}

void launch_step_advance(cudaStream_t st, int32_t* step, int limit) { k_step_advance<<<1, 1, 0, st>>>(step, limit); }

// Entry of the device-resident step loop (before its conditional while node; k_finalize decides
// after every step): whether step j = *step runs at all. It does not when every pair has
// stopped, k_max is reached or a column compaction is due before it (tested as in k_finalize,
// and skipped before step *compact_from: the host moves that past a step where it packed, or
// found no narrower layout).
__global__ void k_loop_entry(const FinArgs a)
{
    const int j = *a.loop_step;
    const int32_t* act_count = a.st.act_count;
    const int act = act_count[j];
    const int act_lag = act_count[j >= a.loop_lag ? j - a.loop_lag : 0];
    const bool compact_due = a.loop_compact && j >= a.loop_lag + 1 && j >= *a.loop_cfrom && a.ld > 16 &&
                             (int64_t)act_lag * 2 <= a.ld;
    const bool go = act > 0 && j < a.k_max && !compact_due;
    if (!go) {
        a.loop_saved[0] = j;
        a.loop_saved[1] = act_lag;
        a.loop_saved[2] = act;
        a.loop_saved[3] = 0;
        *a.loop_step = a.k_max + 1;
    }
    cudaGraphSetConditional((cudaGraphConditionalHandle)a.loop_handle, go ? 1 : 0);
}

void launch_loop_entry(cudaStream_t st, const FinArgs& a) { k_loop_entry<<<1, 1, 0, st>>>(a); }

// ------------------------------------------------------- sparse first step
// q_1 is nonzero only in rows s and t of its column, so the first product
// W = D^{-1} A q_1 (Algorithm 3 with q_0 = 0) is nonzero only on the rows adjacent to s or
// t. One block per column: with L the endpoint of larger degree and S the other,
//   pass 1, rows u in N(L):  W_u <- w_{uL} q_1[L]                       (partial row sum)
//   pass 2, rows u in N(S):  u in N(L) (binary search in the sorted row L):
//                              W_u <- W_u + w_{uS} q_1[S]                (still unscaled)
//                            otherwise W_u <- (1/d_u) w_{uS} q_1[S]      (final)
//   pass 3, rows u in N(L):  W_u <- (1/d_u) W_u                           (final)
// and the column's sums A = sum d W q_1, B = sum d W^2, C = sum d W are taken in FP64 as one
// block partial. Needs rows strictly increasing in column and symmetric entries (row u
// holds L and S with the weights rows L and S hold u), so that these are the SpMM's rows.
template <typename T>
__device__ __forceinline__ void step0_term(T& acc, const float* w, int64_t e, T q)
{
    if (w) acc_mul_add_w(acc, __ldg(w + e), q);
    else acc_add(acc, q);
}

template <typename T>
__global__ void __launch_bounds__(256) k_step0_sparse(const Step0Args<T> a)
{
    __shared__ double red[8][3];
    const int p = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t s = a.s[p], t = a.t[p];
    bool live = s >= 0 && (int64_t)s < a.n && t >= 0 && (int64_t)t < a.n && s != t;
    T q1s = T(0), q1t = T(0);
    if (live) {
        q1s = a.q1[(int64_t)s * a.ld + p];
        q1t = a.q1[(int64_t)t * a.ld + p];
        live = to_double(q1s) != 0.0 || to_double(q1t) != 0.0;
    }
    double* out = a.block_part ? a.block_part + (int64_t)(p / a.tp) * 3 * a.tp + p % a.tp : nullptr;
    if (!live) {  // uniform over the block: the column stays zero
        if (threadIdx.x == 0 && out) out[0] = out[a.tp] = out[2 * a.tp] = 0.0;
        return;
    }
    const int64_t ds_n = a.row_ptr[s + 1] - a.row_ptr[s], dt_n = a.row_ptr[t + 1] - a.row_ptr[t];
    const bool s_large = ds_n >= dt_n;
    const int32_t L = s_large ? s : t, S = s_large ? t : s;
    const T q1L = s_large ? q1s : q1t, q1S = s_large ? q1t : q1s;
    const int64_t lb = a.row_ptr[L], le = a.row_ptr[L + 1];
    const int64_t sb = a.row_ptr[S], se = a.row_ptr[S + 1];
    const int64_t ld = a.ld;
    double sA = 0.0, sB = 0.0, sC = 0.0;
    auto add_sums = [&](int32_t u, T W) {
        const double d = a.deg64[u], x = to_double(W);
        sB += d * x * x;
        sC += d * x;
        if (u == s) sA += d * x * to_double(q1s);
        else if (u == t) sA += d * x * to_double(q1t);
    };
    for (int64_t e = lb + threadIdx.x; e < le; e += blockDim.x) {
        const int32_t u = __ldg(a.col + e);
        T acc = T(0);
        step0_term(acc, a.w, e, q1L);
        acc_finish(acc);
        a.wout[(int64_t)u * ld + p] = acc;
    }
    __syncthreads();
    for (int64_t e = sb + threadIdx.x; e < se; e += blockDim.x) {
        const int32_t u = __ldg(a.col + e);
        int64_t lo = lb, hi = le;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (__ldg(a.col + mid) < u) lo = mid + 1; else hi = mid;
        }
        T* wp = a.wout + (int64_t)u * ld + p;
        if (lo < le && __ldg(a.col + lo) == u) {
            T acc = *wp;
            step0_term(acc, a.w, e, q1S);
            acc_finish(acc);
            *wp = acc;
        } else {
            T acc = T(0);
            step0_term(acc, a.w, e, q1S);
            acc_finish(acc);
            const T W = a.invdeg[u] * acc;
            *wp = W;
            add_sums(u, W);
        }
    }
    __syncthreads();
    for (int64_t e = lb + threadIdx.x; e < le; e += blockDim.x) {
        const int32_t u = __ldg(a.col + e);
        T* wp = a.wout + (int64_t)u * ld + p;
        const T W = a.invdeg[u] * *wp;
        *wp = W;
        add_sums(u, W);
    }
    if (!out) return;
    // fixed-order reduction: xor tree within each warp, then warps in order
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        sA += __shfl_xor_sync(0xffffffffu, sA, off);
        sB += __shfl_xor_sync(0xffffffffu, sB, off);
        sC += __shfl_xor_sync(0xffffffffu, sC, off);
    }
    if (lane == 0) {
        red[warp][0] = sA;
        red[warp][1] = sB;
        red[warp][2] = sC;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double v = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w][threadIdx.x];
        out[threadIdx.x * a.tp] = v;
    }
}

template <typename T>
static void launch_step0(cudaStream_t st, const Step0Args<T>& a)
{
    if (a.npairs > 0) k_step0_sparse<T><<<a.npairs, 256, 0, st>>>(a);
}
// Step 0's normalise pass after the sparse first step, first part. W_1 is nonzero only on
// N(s) ∪ N(t) and q_1 only on {s, t}; elsewhere q_2 = (W_1 - alpha_1 q_1 - c_1) / beta_2 is the
// same value in every row of a column (left to the fill). One CTA per column updates each row
// of that union once, in place, with k_normalize's arithmetic, and marks its entry in the
// mask: N(L) of the endpoint of larger degree, then N(S) minus N(L) (binary search in the
// sorted row L), then s and t unless they are adjacent (then each is in the other's row).
// Columns whose first step wrote nothing (as k_step0_sparse decides) are left to the fill.
template <typename T>
__global__ void __launch_bounds__(256) k_normalize_step0(const Step0NormArgs<T> a)
{
    const int p = blockIdx.x;
    const int32_t s = a.s[p], t = a.t[p];
    const int64_t ld = a.ld;
    bool live = s >= 0 && (int64_t)s < a.n && t >= 0 && (int64_t)t < a.n && s != t;
    if (live)
        live = to_double(a.q1[(int64_t)s * ld + p]) != 0.0 || to_double(a.q1[(int64_t)t * ld + p]) != 0.0;
    if (!live) return;  // uniform over the block
    const T al = a.cf[ld + p], c = a.cf[2 * ld + p], ib = a.cf[3 * ld + p];
    // w_zero: a row the first step did not write (s or t when they are not adjacent: their
    // W_1 entries are zero, and the block holds no zeros there)
    auto upd = [&](int32_t u, bool w_zero) {
        const int64_t e = (int64_t)u * ld + p;
        a.w[e] = lanczos_next<T>(w_zero ? T(0) : a.w[e], al, a.q1[e], c, ib);
        atomicOr(a.mask + (e >> 5), 1u << (e & 31));
    };
    const int64_t ds_n = a.row_ptr[s + 1] - a.row_ptr[s], dt_n = a.row_ptr[t + 1] - a.row_ptr[t];
    const int32_t L = ds_n >= dt_n ? s : t, S = ds_n >= dt_n ? t : s;
    const int64_t lb = a.row_ptr[L], le = a.row_ptr[L + 1];
    const int64_t sb = a.row_ptr[S], se = a.row_ptr[S + 1];
    auto in_row_L = [&](int32_t u) {
        int64_t lo = lb, hi = le;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (__ldg(a.col + mid) < u) lo = mid + 1; else hi = mid;
        }
        return lo < le && __ldg(a.col + lo) == u;
    };
    for (int64_t e = lb + threadIdx.x; e < le; e += blockDim.x) upd(__ldg(a.col + e), false);
    for (int64_t e = sb + threadIdx.x; e < se; e += blockDim.x) {
        const int32_t u = __ldg(a.col + e);
        if (!in_row_L(u)) upd(u, false);
    }
    if (threadIdx.x == 0 && !in_row_L(S)) {
        upd(s, true);
        upd(t, true);
    }
}

// Second part: every entry the first part did not mark gets (0 - alpha_1 * 0 - c_1) / beta_2
// formed as k_normalize forms it from the zeros of W_1 and q_1 there, without reading the
// block (it holds no zeros there: the sparse first step leaves it unwritten). Thread t keeps
// one 16-byte column unit (its values in registers) and walks the rows t / units,
// + rows_per_pass, ...; a unit with marked entries is written element by element around them.
template <typename T>
__global__ void __launch_bounds__(256) k_normalize_step0_fill(const Step0NormArgs<T> a)
{
    constexpr int V = 16 / (int)sizeof(T);
    const int64_t ld = a.ld;
    const int64_t units = ld / V;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t rows_per_pass = (int64_t)gridDim.x * blockDim.x / units;
    const int64_t r0 = t / units;
    if (r0 >= rows_per_pass) return;
    const int64_t c0 = (t % units) * V;
    T v[V];
#pragma unroll
    for (int i = 0; i < V; ++i)
        v[i] = lanczos_next<T>(T(0), a.cf[ld + c0 + i], T(0), a.cf[2 * ld + c0 + i], a.cf[3 * ld + c0 + i]);
    for (int64_t u = r0; u < a.n; u += rows_per_pass) {
        const int64_t e0 = u * ld + c0;
        const uint32_t bits = (a.mask[e0 >> 5] >> (e0 & 31)) & ((1u << V) - 1u);
        if (bits == 0) {
            st_plain<T, V>(a.w + e0, v);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (!((bits >> i) & 1u)) a.w[e0 + i] = v[i];
        }
    }
}

template <typename T>
static void launch_norm0(int grid, cudaStream_t st, const Step0NormArgs<T>& a)
{
    if (a.npairs > 0) k_normalize_step0<T><<<a.npairs, 256, 0, st>>>(a);
    // at least one row per pass (the host takes this path only for whole 16-byte units)
    const int64_t units = a.ld / (16 / (int64_t)sizeof(T));
    const int g = (int)std::max<int64_t>(grid, (units + 255) / 256);
    k_normalize_step0_fill<T><<<g, 256, 0, st>>>(a);
}
void launch_normalize_step0_f32(int grid, cudaStream_t st, const Step0NormArgs<float>& a)
{
    launch_norm0<float>(grid, st, a);
}
void launch_normalize_step0_f64(int grid, cudaStream_t st, const Step0NormArgs<double>& a)
{
    launch_norm0<double>(grid, st, a);
}
void launch_normalize_step0_df64(int grid, cudaStream_t st, const Step0NormArgs<df64>& a)
{
    launch_norm0<df64>(grid, st, a);
}

void launch_step0_f32(cudaStream_t st, const Step0Args<float>& a) { launch_step0<float>(st, a); }
void launch_step0_f64(cudaStream_t st, const Step0Args<double>& a) { launch_step0<double>(st, a); }
void launch_step0_df64(cudaStream_t st, const Step0Args<df64>& a) { launch_step0<df64>(st, a); }

void launch_normalize_f32(int grid, cudaStream_t st, const NormArgs<float>& a) { launch_norm<float>(grid, st, a); }
void launch_normalize_f64(int grid, cudaStream_t st, const NormArgs<double>& a) { launch_norm<double>(grid, st, a); }
void launch_normalize_df64(int grid, cudaStream_t st, const NormArgs<df64>& a) { launch_norm<df64>(grid, st, a); }

// The normalise pass of the step after which the active columns are packed (a column
// compaction), fused with the packing: new column d takes old column o = old_slot[d] (-1:
// zero), and both q_{i+1} (formed from W, q_i and the step's coefficients as k_normalize
// forms it) and q_i are written in the packed layout. One read of W and q_i and one write of
// each packed block, against a normalise pass plus a packing pass that reads both full blocks
// again. Thread t keeps one 16-byte column unit (its slots and coefficients in registers)
// and walks the rows t / units, + rows_per_pass, ...
template <typename T>
__global__ void __launch_bounds__(256) k_normalize_pack(const NormPackArgs<T> a)
{
    constexpr int V = 16 / (int)sizeof(T);
    const int64_t units = a.ld_new / V;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t rows_per_pass = (int64_t)gridDim.x * blockDim.x / units;
    const int64_t r0 = t / units;
    if (r0 >= rows_per_pass) return;
    const int64_t cu = t % units;
    int o[V];
    T al[V], c[V], ib[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
        o[i] = a.old_slot[cu * V + i];
        const int os = o[i] >= 0 ? o[i] : 0;
        al[i] = a.cf[a.ld_old + os];
        c[i] = a.cf[2 * a.ld_old + os];
        ib[i] = a.cf[3 * a.ld_old + os];
    }
    for (int64_t u = r0; u < a.n; u += rows_per_pass) {
        const T* wr = a.w + u * a.ld_old;
        const T* qr = a.qcur + u * a.ld_old;
        T qn[V], qc[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            if (o[i] >= 0) {
                qc[i] = qr[o[i]];
                qn[i] = lanczos_next<T>(wr[o[i]], al[i], qc[i], c[i], ib[i]);
            } else {
                qc[i] = T(0);
                qn[i] = T(0);
            }
        }
        st_plain<T, V>(a.qnext_new + u * a.ld_new + cu * V, qn);
        st_plain<T, V>(a.qcur_new + u * a.ld_new + cu * V, qc);
    }
}

template <typename T>
static bool launch_npack(int grid, cudaStream_t st, const NormPackArgs<T>& a)
{
    constexpr int64_t V = 16 / (int64_t)sizeof(T);
    if (a.ld_new % V != 0 || (int64_t)grid * 256 < a.ld_new / V) return false;
    k_normalize_pack<T><<<grid, 256, 0, st>>>(a);
    return true;
}
bool launch_normalize_pack_f32(int grid, cudaStream_t st, const NormPackArgs<float>& a) { return launch_npack(grid, st, a); }
bool launch_normalize_pack_f64(int grid, cudaStream_t st, const NormPackArgs<double>& a) { return launch_npack(grid, st, a); }
bool launch_normalize_pack_df64(int grid, cudaStream_t st, const NormPackArgs<df64>& a) { return launch_npack(grid, st, a); }

// Double-float copy of an FP64 array (degrees and their inverses for RD_MODE_DF64).
__global__ void k_split_df(int64_t n, const double* __restrict__ src, df64* __restrict__ dst)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = df64(src[i]);
}

void launch_split_df(cudaStream_t st, int grid, int64_t n, const double* src, df64* dst)
{
    k_split_df<<<grid, 256, 0, st>>>(n, src, dst);
}

// ---------------------------------------------------------------- output
__global__ void k_output(const OutArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.npairs || *a.err_flag) return;
    const PairState& st = a.st;
    const int status = st.status[p];
    a.r_out[p] = st.r[p];
    if (a.iters_out) a.iters_out[p] = st.k[p];
    if (a.err_out) a.err_out[p] = st.err[p];
    if (a.status_out) a.status_out[p] = status;
    if (status == RD_WARN_NOT_CONVERGED) atomicOr(&a.summary[0], 1);
    if (status == RD_ERR_NUMERIC) atomicOr(&a.summary[1], 1);
}

void launch_output(cudaStream_t st, const OutArgs& a)
{
    k_output<<<(a.npairs + 127) / 128, 128, 0, st>>>(a);
}

// ---------------------------------------------------- tridiagonal solve
// z = (I - T_k)^{-1} e_1 per pair from the stored alpha_1..alpha_k, beta_2..beta_k by
// forward elimination and back substitution (I - T_k is SPD, so no pivoting);
// coef_j = ||b|| z_j is the weight of q_j in the potential
// phi = ||b|| D^{-1/2} V_k z (the potential of Algorithm 5). Also writes gbar[p], the upstream
// gradient of pair p (0 for pairs without a finite result and for padding columns).
template <typename T>
__global__ void k_zsolve(const ZsolveArgs a)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.ld) return;
    T* coef = static_cast<T*>(a.coef_hist);
    T* gbar = static_cast<T*>(a.gbar);
    const PairState& st = a.st;
    const int64_t ld = a.ld;
    const int status = p < a.npairs ? st.status[p] : RD_ERR_INVALID_ARG;
    const int k = p < a.npairs ? st.k[p] : 0;
    const bool use = (status == RD_OK || status == RD_WARN_NOT_CONVERGED) && k > 0;
    if (!coef) {  // the potential was accumulated during the steps: gbar is all that is needed
        gbar[p] = use ? (T)(a.grad_r ? a.grad_r[p] : 1.0) : T(0);
        return;
    }
    if (!use) {
        for (int j = 0; j < a.k_max; ++j) coef[(int64_t)j * ld + p] = T(0);
        gbar[p] = T(0);
        return;
    }
    gbar[p] = (T)(a.grad_r ? a.grad_r[p] : 1.0);
    double* zs = a.zscratch;  // [k_max][2][ld]: c'_j, d'_j
    const double* al = st.hist_alpha;
    const double* be = st.hist_beta;  // be[j*ld + p] = beta_{j+1}
    double cprev = 0.0, dprev = 0.0;
    for (int j = 0; j < k; ++j) {
        const double lower = j > 0 ? -be[(int64_t)j * ld + p] : 0.0;
        const double m = (1.0 - al[(int64_t)j * ld + p]) - lower * cprev;
        const double c = (j + 1 < k) ? -be[(int64_t)(j + 1) * ld + p] / m : 0.0;
        const double d = ((j == 0 ? 1.0 : 0.0) - lower * dprev) / m;
        zs[((int64_t)j * 2) * ld + p] = c;
        zs[((int64_t)j * 2 + 1) * ld + p] = d;
        cprev = c;
        dprev = d;
    }
    const double bn = sqrt(st.b2[p]);
    double x = 0.0;
    for (int j = k - 1; j >= 0; --j) {
        x = zs[((int64_t)j * 2 + 1) * ld + p] - zs[((int64_t)j * 2) * ld + p] * x;
        coef[(int64_t)j * ld + p] = (T)(bn * x);
    }
    for (int j = k; j < a.k_max; ++j) coef[(int64_t)j * ld + p] = T(0);
}

void launch_zsolve(cudaStream_t st, const ZsolveArgs& a)
{
    const int nb = (int)((a.ld + 127) / 128);
    if (a.elem_size == 8) k_zsolve<double><<<nb, 128, 0, st>>>(a);
    else k_zsolve<float><<<nb, 128, 0, st>>>(a);
}

// ---------------------------------------------------------- edge gradient
// grad[e] = -1/2 sum_p gbar_p (phi_p(u) - phi_p(v))^2 for stored entry e = (u -> v).
// Entries are processed in CSR order, kU consecutive entries per row group of GS lanes
// (VEC*GS columns per column chunk), so the gathers of kU entries are in flight at once;
// the row of each entry comes from the graph's entry-row array.
template <typename T, int VEC, int GS>
__global__ void __launch_bounds__(256) k_edge_grad(const EdgeGradArgs<T> a)
{
    constexpr int TP = VEC * GS;
    constexpr int NG = 32 / GS;
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = lane % GS, grp = lane / GS;
    const unsigned mask = group_mask<GS, 1>(lane);
    const int64_t ngroups = (int64_t)gridDim.x * (blockDim.x / 32) * NG;
    const int64_t gid = ((int64_t)blockIdx.x * (blockDim.x / 32) + warp) * NG + grp;
    const int nch = (int)(a.ld / TP);
    for (int64_t e0 = gid * kU; e0 < a.nnz; e0 += ngroups * kU) {
        int64_t u[kU], v[kU];
        float s[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) {
            const bool ok = e0 + k < a.nnz;
            u[k] = ok ? (int64_t)__ldg(a.entry_row + e0 + k) : 0;
            v[k] = ok ? (int64_t)__ldg(a.col + e0 + k) : 0;
            s[k] = 0.f;
        }
        for (int ch = 0; ch < nch; ++ch) {
            const int64_t c0 = (int64_t)ch * TP + cl * VEC;
            T gb[VEC], pu[kU][VEC], pv[kU][VEC];
            ld_gather<T, VEC>(gb, a.gbar + c0);
#pragma unroll
            for (int k = 0; k < kU; ++k) {
                ld_gather<T, VEC>(pu[k], a.phi + u[k] * a.ld + c0);
                ld_gather<T, VEC>(pv[k], a.phi + v[k] * a.ld + c0);
            }
#pragma unroll
            for (int k = 0; k < kU; ++k)
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    const T d = pu[k][i] - pv[k][i];
                    s[k] += (float)(gb[i] * d * d);
                }
        }
#pragma unroll
        for (int k = 0; k < kU; ++k) {
#pragma unroll
            for (int off = 1; off < GS; off <<= 1) s[k] += __shfl_xor_sync(mask, s[k], off);
            if (cl == 0 && e0 + k < a.nnz) a.grad_out[e0 + k] = -0.5f * s[k];
        }
    }
}

template <typename T>
static void launch_eg(int grid, cudaStream_t st, const EdgeGradArgs<T>& a)
{
    constexpr int VEC = 16 / (int)sizeof(T);
    const int64_t units = a.ld / VEC;  // ld is a multiple of VEC here
    if (units % 32 == 0) k_edge_grad<T, VEC, 32><<<grid, 256, 0, st>>>(a);
    else if (units % 16 == 0) k_edge_grad<T, VEC, 16><<<grid, 256, 0, st>>>(a);
    else if (units % 8 == 0) k_edge_grad<T, VEC, 8><<<grid, 256, 0, st>>>(a);
    else if (units % 4 == 0) k_edge_grad<T, VEC, 4><<<grid, 256, 0, st>>>(a);
    else if (units % 2 == 0) k_edge_grad<T, VEC, 2><<<grid, 256, 0, st>>>(a);
    else k_edge_grad<T, VEC, 1><<<grid, 256, 0, st>>>(a);
}

// Row of every stored entry (one warp per row, lanes strided over the row's entries).
__global__ void __launch_bounds__(256) k_entry_rows(int64_t n, const int64_t* row_ptr, int32_t* entry_row)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x / 32);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); r < n; r += nw)
        for (int64_t e = row_ptr[r] + lane; e < row_ptr[r + 1]; e += 32) entry_row[e] = (int32_t)r;
}

void launch_entry_rows(int grid, cudaStream_t st, int64_t n, const int64_t* row_ptr, int32_t* entry_row)
{
    k_entry_rows<<<grid, 256, 0, st>>>(n, row_ptr, entry_row);
}

void launch_edge_grad_f32(int grid, cudaStream_t st, const EdgeGradArgs<float>& a) { launch_eg<float>(grid, st, a); }
void launch_edge_grad_f64(int grid, cudaStream_t st, const EdgeGradArgs<double>& a) { launch_eg<double>(grid, st, a); }

// ------------------------------------------------- potentials and flows, pair-major
// Bound by the output, 4 bytes per item and pair (and, for flows, the gathers of phi[col]). A block
// takes kPmItems consecutive items: their rows of phi are read along the columns in 16-byte
// units, the values pass through a tile in shared memory, and each pair's run of items is
// written out whole. Read per output element instead (a stride of ld between lanes, every
// 32-byte sector fetched for 4 of its bytes), the flows of 16 pairs over 3.9M entries took
// 285 us, against 38 us for their 250 MB alone.
constexpr int kPmItems = 128, kPmCols = 32;

template <typename T, int V>
__global__ void __launch_bounds__(256) k_pair_major(const PairMajorArgs a)
{
    __shared__ float tile[kPmCols][kPmItems + 1];
    const int64_t i0 = (int64_t)blockIdx.x * kPmItems;
    const int ni = (int)(a.items - i0 < kPmItems ? a.items - i0 : kPmItems);
    const T* phi = static_cast<const T*>(a.phi);
    for (int c0 = 0; c0 < a.npairs; c0 += kPmCols) {
        const int nc = a.npairs - c0 < kPmCols ? a.npairs - c0 : kPmCols;
        const int units = (nc + V - 1) / V;  // ld is a multiple of V, so the last unit is whole in memory
        for (int k = threadIdx.x; k < ni * units; k += 256) {
            const int i = k / units, cu = (k - i * units) * V;
            T x[V];
            if (a.row) {
                T y[V];
                ld_gather<T, V>(x, phi + (int64_t)__ldg(a.row + i0 + i) * a.ld + c0 + cu);
                ld_gather<T, V>(y, phi + (int64_t)__ldg(a.col + i0 + i) * a.ld + c0 + cu);
#pragma unroll
                for (int v = 0; v < V; ++v) x[v] -= y[v];
            } else {
                ld_gather<T, V>(x, phi + (i0 + i) * a.ld + c0 + cu);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) tile[cu + v][i] = (float)x[v];
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nc * kPmItems; k += 256) {
            const int i = k % kPmItems, p = k / kPmItems;
            if (i < ni) {
                const int64_t o = a.keep_idx ? a.keep_idx[i0 + i] : i0 + i;
                __stcs(a.out + (int64_t)(c0 + p) * a.out_stride + o, tile[p][i]);
            }
        }
        __syncthreads();
    }
}

template <typename T>
static void launch_pm(cudaStream_t st, const PairMajorArgs& a)
{
    constexpr int V = 16 / (int)sizeof(T);
    const int64_t grid = (a.items + kPmItems - 1) / kPmItems;
    if (grid == 0 || a.npairs == 0) return;
    if (a.ld % V == 0) k_pair_major<T, V><<<(unsigned)grid, 256, 0, st>>>(a);
    else k_pair_major<T, 1><<<(unsigned)grid, 256, 0, st>>>(a);
}

void launch_pair_major(cudaStream_t st, bool fp64, const PairMajorArgs& a)
{
    if (fp64) launch_pm<double>(st, a);
    else launch_pm<float>(st, a);
}

// --------------------------------------------------------------- compaction
// Slot map of the still-active pairs, in slot order (one block, chunked block scan), and
// the coefficients of the next step moved to the new slots.
template <typename T>
__global__ void __launch_bounds__(1024) k_compact_map(const CompactArgs a)
{
    __shared__ int warp_tot[32];
    __shared__ int base_s;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) base_s = 0;
    __syncthreads();
    for (int64_t c0 = 0; c0 < a.ld_old; c0 += blockDim.x) {
        const int64_t slot = c0 + tid;
        int p = -1;
        if (slot < a.ld_old) p = a.slot_pair_old ? a.slot_pair_old[slot] : (slot < a.npairs ? (int)slot : -1);
        const int keep = (p >= 0 && a.active[p]) ? 1 : 0;
        // block-wide exclusive scan of keep
        unsigned bal = __ballot_sync(0xffffffffu, keep);
        const int in_warp = __popc(bal & ((1u << lane) - 1u));
        if (lane == 0) warp_tot[w] = __popc(bal);
        __syncthreads();
        int before = 0;
        for (int i = 0; i < w; ++i) before += warp_tot[i];
        int chunk_total = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) chunk_total += warp_tot[i];
        const int dst = base_s + before + in_warp;
        if (keep && dst < a.ld_new) {
            a.slot_pair_new[dst] = p;
            a.old_slot[dst] = (int)slot;
        }
        __syncthreads();
        if (tid == 0) base_s += chunk_total;
        __syncthreads();
    }
    const int kept = base_s;
    const T* cfo = static_cast<const T*>(a.cf_old);
    T* cfn = static_cast<T*>(a.cf_new);
    for (int64_t d = tid; d < a.ld_new; d += blockDim.x) {
        if (d >= kept) {
            a.slot_pair_new[d] = -1;
            a.old_slot[d] = -1;
        }
    }
    __syncthreads();
    for (int64_t d = tid; d < a.ld_new; d += blockDim.x) {
        const int o = a.old_slot[d];
#pragma unroll
        for (int q = 0; q < 4; ++q) cfn[q * a.ld_new + d] = o >= 0 ? cfo[q * a.ld_old + o] : T(0);
    }
}

// q blocks copied column-wise into the compact layout (empty slots zero), any ld_new.
template <typename T>
__global__ void __launch_bounds__(256) k_compact_cols(const CompactArgs a)
{
    const int64_t total = a.n * a.ld_new;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const T* s0 = static_cast<const T*>(a.q_src0);
    const T* s1 = static_cast<const T*>(a.q_src1);
    T* d0 = static_cast<T*>(a.q_dst0);
    T* d1 = static_cast<T*>(a.q_dst1);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        const int64_t u = i / a.ld_new, c = i % a.ld_new;
        const int o = a.old_slot[c];
        d0[i] = o >= 0 ? s0[u * a.ld_old + o] : T(0);
        d1[i] = o >= 0 ? s1[u * a.ld_old + o] : T(0);
    }
}

// The same when ld_new is a multiple of the 16-byte unit V: thread t keeps one column unit
// (its V source slots in registers) and walks the rows t / units, + rows_per_pass, ...;
// each new row unit is one 16-byte store per block, and no index division runs per element.
template <typename T>
__global__ void __launch_bounds__(256) k_compact_cols_v(const CompactArgs a)
{
    constexpr int V = 16 / (int)sizeof(T);
    const int64_t units = a.ld_new / V;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t rows_per_pass = (int64_t)gridDim.x * blockDim.x / units;
    const int64_t r0 = t / units;
    if (r0 >= rows_per_pass) return;  // threads past the last whole group of units
    const int64_t cu = t % units;
    int o[V];
#pragma unroll
    for (int i = 0; i < V; ++i) o[i] = a.old_slot[cu * V + i];
    const T* s0 = static_cast<const T*>(a.q_src0);
    const T* s1 = static_cast<const T*>(a.q_src1);
    T* d0 = static_cast<T*>(a.q_dst0);
    T* d1 = static_cast<T*>(a.q_dst1);
    for (int64_t u = r0; u < a.n; u += rows_per_pass) {
        T x0[V], x1[V];
        const T* r0p = s0 + u * a.ld_old;
        const T* r1p = s1 + u * a.ld_old;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            x0[i] = o[i] >= 0 ? r0p[o[i]] : T(0);
            x1[i] = o[i] >= 0 ? r1p[o[i]] : T(0);
        }
        st_plain<T, V>(d0 + u * a.ld_new + cu * V, x0);
        st_plain<T, V>(d1 + u * a.ld_new + cu * V, x1);
    }
}

void launch_compact_map(cudaStream_t st, const CompactArgs& a)
{
    if (a.elem_size == 8) k_compact_map<double><<<1, 1024, 0, st>>>(a);
    else k_compact_map<float><<<1, 1024, 0, st>>>(a);
}

void launch_compact(cudaStream_t st, int grid, const CompactArgs& a)
{
    // the unit kernel needs whole 16-byte units per row and at least one row per pass
    const int64_t v = 16 / a.elem_size;
    const bool unit = a.ld_new % v == 0 && (int64_t)grid * 256 >= a.ld_new / v;
    if (a.elem_size == 8) {
        k_compact_map<double><<<1, 1024, 0, st>>>(a);
        if (unit) k_compact_cols_v<double><<<grid, 256, 0, st>>>(a);
        else k_compact_cols<double><<<grid, 256, 0, st>>>(a);
    } else {
        k_compact_map<float><<<1, 1024, 0, st>>>(a);
        if (unit) k_compact_cols_v<float><<<grid, 256, 0, st>>>(a);
        else k_compact_cols<float><<<grid, 256, 0, st>>>(a);
    }
}

// ---------------------------------------------------------- Power Method
template <typename T>
__global__ void k_pm_init(const PmArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.npairs) return;
    const int32_t s = a.s[p], t = a.t[p];
    if (s < 0 || (int64_t)s >= a.n || t < 0 || (int64_t)t >= a.n) {
        atomicOr(a.err_flag, 1);
        return;
    }
    a.rbar[p] = 0.0;
    if (s == t) return;
    T* y = static_cast<T*>(a.y);
    y[(int64_t)s * a.ld + p] = (T)(1.0 / a.deg64[s]);
    y[(int64_t)t * a.ld + p] = (T)(-1.0 / a.deg64[t]);
}

template <typename T>
__global__ void k_pm_accum(const PmArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.npairs) return;
    const int32_t s = a.s[p], t = a.t[p];
    if (s == t) {
        if (a.hist) a.hist[(int64_t)a.step * a.npairs + p] = 0.0;
        return;
    }
    const T* y = static_cast<const T*>(a.y);
    const double r = a.rbar[p] + 0.5 * ((double)y[(int64_t)s * a.ld + p] - (double)y[(int64_t)t * a.ld + p]);
    a.rbar[p] = r;
    if (a.hist) a.hist[(int64_t)a.step * a.npairs + p] = r;
}

void launch_pm_init(cudaStream_t st, const PmArgs& a)
{
    const int nb = (a.npairs + 127) / 128;
    if (a.elem_size == 8) k_pm_init<double><<<nb, 128, 0, st>>>(a);
    else k_pm_init<float><<<nb, 128, 0, st>>>(a);
}

void launch_pm_accum(cudaStream_t st, const PmArgs& a)
{
    const int nb = (a.npairs + 127) / 128;
    if (a.elem_size == 8) k_pm_accum<double><<<nb, 128, 0, st>>>(a);
    else k_pm_accum<float><<<nb, 128, 0, st>>>(a);
}

// ------------------------------------------------------------- on chip
// One pair per CTA, every step in one launch: SpMV from shared memory (one thread per light
// row, one warp per row above heavy_thr), three FP64 block sums in a fixed order, the same
// per-pair update as k_finalize (pair_core) by thread 0, normalisation in shared memory.
constexpr int kOnchipThreads = 1024;

size_t onchip_smem_bytes(int64_t n, int elem_size) { return (size_t)3 * (size_t)n * (size_t)elem_size + 64; }

// The pair's state across the steps of a whole-recurrence kernel, and its results.
struct OnchipPair {
    PairScalars s;
    double r = 0.0, est = 1.0;
    int k = 0, status = RD_OK;
};

// Above this many pairs one launch looks the ids over (k_check_ids) instead of every block. A scan by
// every block grows with the square of the pairs; 25 vertices, 4 steps: 4,096 pairs 225 us with the
// scan and 253 with the launch, 16,384 743 and 768, 65,536 3,861 and 2,813, 2^20 519,307 and 43,638.
constexpr int kScanPairs = 16384;

__device__ __forceinline__ bool bad_ids(const OnchipArgs& a, int i)
{
    const int32_t s = a.s[i], t = a.t[i];
    return s < 0 || s >= a.n || t < 0 || t >= a.n;
}

__global__ void k_check_ids(const OnchipArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.npairs && bad_ids(a, i)) atomicOr(&a.summary[2], 1);
}

// Start of a whole-recurrence kernel for pair p: true when its recurrence runs. A call with a bad id
// writes nothing but the flag, so every block first looks all ids over, or at what k_check_ids found; a
// pair that needs no recurrence is answered at once (`writer`: the thread that stores).
template <int NT>
__device__ __forceinline__ bool onchip_start(const OnchipArgs& a, int p, bool writer)
{
    int bad = 0;
    if (a.npairs > kScanPairs) bad = a.summary[2];
    else
        for (int i = threadIdx.x; i < a.npairs; i += NT) bad |= bad_ids(a, i);
    if (__syncthreads_or(bad)) {
        if (writer) a.summary[2] = 1;
        return false;
    }
    if (p >= a.npairs) return false;
    const int32_t s = a.s[p], t = a.t[p];
    const bool apart = a.comp && a.comp[s] != a.comp[t];
    if (s != t && !apart) return true;
    if (writer) {
        a.r_out[p] = apart ? INFINITY : 0.0;
        a.iters_out[p] = 0;
        a.err_out[p] = 0.0;
        a.status_out[p] = apart ? RD_ERR_DISCONNECTED : RD_OK;
    }
    return false;
}

// Step j's scalar update of the pair; when it ends the pair and `writer` is set, its results.
__device__ __forceinline__ bool onchip_update(const OnchipArgs& a, OnchipPair& q, int p, int j, const StepCoef& k,
                                              bool writer)
{
    PairStepOut o;
    const bool stop = pair_core(a.fin, q.s, j, k, o);
    if (o.ok) {
        q.r = o.r;
        q.est = o.est;
        q.k = j + 1;
        if (o.warn_not_converged) q.status = RD_WARN_NOT_CONVERGED;
    } else {
        q.status = RD_ERR_NUMERIC;  // the last good estimate stands
    }
    if (stop && writer) {
        a.r_out[p] = q.r;
        a.iters_out[p] = q.k;
        a.err_out[p] = q.est;
        a.status_out[p] = q.status;
        if (q.status == RD_WARN_NOT_CONVERGED) atomicOr(&a.summary[0], 1);
        if (q.status == RD_ERR_NUMERIC) atomicOr(&a.summary[1], 1);
    }
    return stop;
}

__device__ __forceinline__ OnchipPair onchip_pair(const OnchipArgs& a, int p)
{
    OnchipPair q;
    q.s = PairScalars{};
    q.s.b2 = 1.0 / a.deg64[a.s[p]] + 1.0 / a.deg64[a.t[p]];
    return q;
}

template <typename T, bool WEIGHTED, bool BY4>
__global__ void __launch_bounds__(kOnchipThreads) k_lanczos_onchip(const OnchipArgs a)
{
    extern __shared__ __align__(16) unsigned char onchip_raw[];
    __shared__ double red[3][kOnchipThreads / 32];
    __shared__ double coef[4], isd;
    __shared__ int stop_s;
    const int p = blockIdx.x;
    if (!onchip_start<kOnchipThreads>(a, p, threadIdx.x == 0)) return;  // uniform over the block
    const int64_t n = a.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthr = blockDim.x, nwarps = nthr >> 5;
    T* buf[3];
    buf[0] = reinterpret_cast<T*>(onchip_raw);
    buf[1] = buf[0] + n;
    buf[2] = buf[1] + n;
    int iprev = 0, icur = 1, iw = 2;
    for (int64_t u = tid; u < 3 * n; u += nthr) buf[0][u] = T(0);
    __syncthreads();
    OnchipPair pr;
    if (tid == 0) {
        isd = __ldg(a.fin.inv_sumdeg);
        pr = onchip_pair(a, p);
        const int32_t s = a.s[p], t = a.t[p];
        const double ds = a.deg64[s], dt = a.deg64[t];
        const double bn = sqrt(pr.s.b2);
        buf[icur][s] = (T)(1.0 / (ds * bn));
        buf[icur][t] = (T)(-1.0 / (dt * bn));
    }
    __syncthreads();
    T bt = T(0);
    for (int j = 0; j < a.fin.k_max; ++j) {
        const T* qp = buf[iprev];
        const T* qc = buf[icur];
        T* W = buf[iw];
        double pa = 0.0, pb = 0.0, pc = 0.0;
        for (int64_t u = tid; u < n; u += nthr) {
            const int64_t e0 = a.row_ptr[u], e1 = a.row_ptr[u + 1];
            if (e1 - e0 > a.heavy_thr) continue;
            T acc = T(0);
            int64_t e = e0;
            // BY4: four entries at a time, asked for while their lines are in the L1 (10,000 weighted FP32
            // vertices, rows of 28, 100 pairs: 4,685 us for 30 steps one at a time, 3,845 so; 7,000
            // unweighted FP64 vertices 3,842 and 3,386). Long rows of FP32 without weights go
            // one at a time while the L1 holds them (10,000 vertices, rows of 56: 4,253 us, 4,630 with
            // four; 16,000: 9,606 and 8,702)
            for (; BY4 && e + 4 <= e1; e += 4) {
                int v[4];
                float we[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    v[k] = __ldg(a.col + e + k);
                    if constexpr (WEIGHTED) we[k] = __ldg(a.w + e + k);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (WEIGHTED) acc += (T)we[k] * qc[v[k]];
                    else acc += qc[v[k]];
                }
            }
            for (; e < e1; ++e) {
                if constexpr (WEIGHTED) acc += (T)__ldg(a.w + e) * qc[__ldg(a.col + e)];
                else acc += qc[__ldg(a.col + e)];
            }
            const T invd = sizeof(T) == 8 ? (T)a.invdeg64[u] : (T)a.invdeg32[u];
            const T du = sizeof(T) == 8 ? (T)a.deg64[u] : (T)a.deg32[u];
            const T wv = invd * acc - bt * qp[u];
            W[u] = wv;
            const T dw = du * wv;
            pa += (double)(dw * qc[u]);
            pb += (double)(dw * wv);
            pc += (double)dw;
        }
        for (int64_t h = warp; h < a.n_heavy_rows; h += nwarps) {
            const int64_t u = a.heavy_rows[h];
            T acc = T(0);
            for (int64_t e = a.row_ptr[u] + lane; e < a.row_ptr[u + 1]; e += 32) {
                if constexpr (WEIGHTED) acc += (T)__ldg(a.w + e) * qc[__ldg(a.col + e)];
                else acc += qc[__ldg(a.col + e)];
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (lane == 0) {
                const T invd = sizeof(T) == 8 ? (T)a.invdeg64[u] : (T)a.invdeg32[u];
                const T du = sizeof(T) == 8 ? (T)a.deg64[u] : (T)a.deg32[u];
                const T wv = invd * acc - bt * qp[u];
                W[u] = wv;
                const T dw = du * wv;
                pa += (double)(dw * qc[u]);
                pb += (double)(dw * wv);
                pc += (double)dw;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            pa += __shfl_xor_sync(0xffffffffu, pa, off);
            pb += __shfl_xor_sync(0xffffffffu, pb, off);
            pc += __shfl_xor_sync(0xffffffffu, pc, off);
        }
        if (lane == 0) {
            red[0][warp] = pa;
            red[1][warp] = pb;
            red[2][warp] = pc;
        }
        __syncthreads();
        if (tid == 0) {
            double A = 0.0, B = 0.0, C = 0.0;
            for (int w = 0; w < nwarps; ++w) {
                A += red[0][w];
                B += red[1][w];
                C += red[2][w];
            }
            const StepCoef k = step_coef(a.fin, isd, A, B, C);
            stop_s = onchip_update(a, pr, p, j, k, true) ? 1 : 0;
            coef[0] = k.alpha;
            coef[1] = k.cdef;
            coef[2] = k.beta;
            coef[3] = k.inv_beta;
        }
        __syncthreads();
        if (stop_s) break;
        const T al = (T)coef[0], cd = (T)coef[1], ib = (T)coef[3];
        for (int64_t u = tid; u < n; u += nthr) W[u] = (W[u] - al * qc[u] - cd) * ib;
        bt = (T)coef[2];
        const int old_prev = iprev;
        iprev = icur;
        icur = iw;
        iw = old_prev;
        __syncthreads();
    }
}

// ---------------------------------------------------- on chip, one cluster per pair
// The whole recurrence of one pair on a thread-block cluster of C CTAs (C = 1..16): CTA r holds
// rows [r R, (r+1) R) of q_{i-1}, q_i and W, of d and 1/d, and (where they fit) of the CSR in its
// shared memory. Per step: every CTA's three FP64 block sums are written into every CTA of the
// cluster, a cluster barrier, every CTA sums the C partials in rank order and forms the same
// coefficients and normalises its rows, and a second cluster barrier publishes the vector.
//
// A product reads q_i[col] in one of two ways. COPY: every CTA holds a whole copy of q_i, and the
// normalise pass writes its rows into all C copies (whole segments, n (C - 1) / C elements into
// each SM). Otherwise: each entry's column is kept as the 32-bit address of its element in the
// owning CTA's shared memory and loaded through distributed shared memory (nnz / C single
// elements into each SM). An element costs about half a cycle either way (measured on a first
// form of the kernel: 64x64 grid, FP64, C = 16, 4.1 us a step with gathers and 5.3 with copies;
// 1,000 vertices, 13,800 entries, FP32, C = 2, a query of 64 pairs x 20 steps 341 us with
// gathers and 297 with copies), so the copies are
// taken when n (C - 1) <= nnz.
//
// What bounds a step is the FP64 unit: an FP64 instruction of one warp occupies a quarter SM for
// about 64 cycles (19 of the SM's) whatever the number of active lanes, an add has 57 cycles of
// latency, a reciprocal 365, a square root 610 (measured). So the chain from the sums to the
// next vector is kept to what it needs:
//  - each of the three block sums is taken by one warp on its own quarter of the SM, and the
//    C x 3 partials of the cluster by one warp (eight lanes a sum);
//  - only alpha, c, beta and 1/beta are formed before the next vector (step_coef); the LDL^T
//    update, the estimate and the stop test of step j - 1 (pair_core, three divisions) run in a
//    fourth warp beside the sums of step j, so a pair stops one product late;
// 64x64 grid, FP64, 16 CTAs: 8.0 us a step before (every partial and division on one thread's
// chain, 39 FP64 instructions for the block sums, the CSR read from global memory), 4.0 us now:
// 2,500 cycles for the product, 1,650 for the block sums, 1,300 and 950 for the barriers, 1,650
// for the coefficients, 700 for the normalise pass. 64 pairs x 20 steps on 1,000 vertices, FP32:
// 233 us before, 95 us now.
constexpr int kClusterMax = 16;
constexpr size_t kClusterSmemMax = 200 * 1024;  // of the 227 KB a block may have
constexpr size_t kClusterSmemMin = 116 * 1024;  // one CTA of a cluster per SM

struct ClusterLayout {
    int C;            // CTAs per pair
    int R;            // rows per CTA
    uint32_t inv_R;   // 2^32 / R rounded up: v / R = (v inv_R) >> 32 for v < 2^16
    int nnz_cap;      // entries of the CSR a CTA can hold in shared memory
};

// What a CTA keeps beside its rows of the three vectors: a copy of q_i (see above), or none
// (gathers); and d, 1/d and the row offsets, or, lean, not even those.
enum ClusterForm { kGather = 0, kCopy = 1, kLean = 2 };

__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, int rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(local), "r"(rank));
    return d;
}
__device__ __forceinline__ float cluster_ld(uint32_t a, float)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ double cluster_ld(uint32_t a, double)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void cluster_st(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_st(uint32_t a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Bytes of shared memory before the entries: the copy of q_i, a CTA's rows of three vectors, d and 1/d,
// and its row offsets.
__host__ __device__ inline size_t cluster_base_bytes(ClusterForm form, int64_t n, int R, int elem)
{
    if (form == kLean) return ((size_t)3 * R * elem + 15) & ~(size_t)15;
    return ((((size_t)(form == kCopy ? n : 0) + 5 * (size_t)R) * elem + (size_t)4 * (R + 1)) + 15) & ~(size_t)15;
}

// Blocks per SM the kernel is compiled for: two of 512 threads (64 registers) where single CTAs share an
// SM; gathers, which run in clusters alone, and FP64 vectors on small blocks get more registers (at
// 64 they spill: 951 FP64 vertices on 16 CTAs, 30 steps, 436 for 300 us).
template <typename T, ClusterForm FORM, int NT>
inline constexpr int kClusterMinBlocks = FORM == kGather ? (NT == 256 ? 3 : 1)
                                         : FORM == kCopy && NT == 256 ? (sizeof(T) == 8 ? 3 : 0) : 1024 / NT;

template <typename T, bool WEIGHTED, ClusterForm FORM, int NT>
__global__ void __launch_bounds__(NT, (kClusterMinBlocks<T, FORM, NT>)) k_lanczos_cluster(const OnchipArgs a, const ClusterLayout L)
{
    constexpr bool COPY = FORM == kCopy, LEAN = FORM == kLean;
    extern __shared__ __align__(16) unsigned char cl_raw[];
    __shared__ double part[3][kClusterMax];       // every CTA's sums of the step, by rank
    __shared__ double tpart[3][NT];               // per-thread partial sums of the step
    __shared__ StepCoef coef;                     // of the step last summed
    __shared__ double isd;                        // 1 / sum of the degrees
    __shared__ T next[4];                         // its 1/beta, alpha, c and beta as vector elements
    __shared__ int stop_s;
    __shared__ uint32_t rbase[kClusterMax];       // address of every rank's vectors
    const int C = L.C, R = L.R;
    const int rank = C > 1 ? blockIdx.x % C : 0;  // clusters are runs of C blocks along x
    const int p = blockIdx.x / C;
    if (!onchip_start<NT>(a, p, rank == 0 && threadIdx.x == 0)) return;  // uniform over the cluster
    const int n = (int)a.n;
    const int row0 = rank * R;
    const int nrow = row0 >= n ? 0 : (n - row0 < R ? n - row0 : R);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nthr = NT, nwarps = NT / 32;
    constexpr uint32_t E = sizeof(T);
    const int ncopy = COPY ? n : 0;
    T* full = reinterpret_cast<T*>(cl_raw);  // q_i, every row (COPY)
    T* buf0 = full + ncopy;
    T* s_invd = buf0 + 3 * R;
    T* s_deg = s_invd + R;
    int* s_rp = reinterpret_cast<int*>(s_deg + R);
    // the entries: weights, then the column (COPY) or the address of its element in buffer 0
    using Col = typename std::conditional<COPY, uint16_t, uint32_t>::type;
    float* s_w = reinterpret_cast<float*>(cl_raw + cluster_base_bytes(FORM, n, R, (int)E));
    Col* s_col = reinterpret_cast<Col*>(WEIGHTED ? s_w + L.nnz_cap : s_w);
    if (tid < C) rbase[tid] = cluster_addr(smem_addr(full), tid);  // buf0 where there is no copy
    for (int u = tid; u < ncopy + 3 * R; u += nthr) full[u] = T(0);
    const int64_t ebase = nrow > 0 ? a.row_ptr[row0] : 0;
    auto g_rp = [&](int u) { return nrow > 0 ? (int)(a.row_ptr[row0 + u] - ebase) : 0; };
    auto g_invd = [&](int u) { return E == 8 ? (T)a.invdeg64[row0 + u] : (T)a.invdeg32[row0 + u]; };
    auto g_deg = [&](int u) { return E == 8 ? (T)a.deg64[row0 + u] : (T)a.deg32[row0 + u]; };
    if constexpr (!LEAN) {
        for (int u = tid; u <= nrow; u += nthr) s_rp[u] = g_rp(u);
        for (int u = tid; u < nrow; u += nthr) {
            s_invd[u] = g_invd(u);
            s_deg[u] = g_deg(u);
        }
    }
    auto rp = [&](int u) {
        if constexpr (LEAN) return g_rp(u);
        else return s_rp[u];
    };
    if (tid == 0) {
        stop_s = 0;
        isd = __ldg(a.fin.inv_sumdeg);
    }
    __syncthreads();
    const int nent = rp(nrow);
    const bool cached = !LEAN && nent <= L.nnz_cap;
    auto locate = [&](int e) -> uint32_t {
        const int v = __ldg(a.col + ebase + e);
        if constexpr (COPY) return (uint32_t)v;
        const int r = (int)__umulhi((uint32_t)v, L.inv_R);
        return rbase[r] + (uint32_t)(v - r * R) * E;
    };
    if (cached)
        for (int e = tid; e < nent; e += nthr) {
            s_col[e] = (Col)locate(e);
            if constexpr (WEIGHTED) s_w[e] = __ldg(a.w + ebase + e);
        }
    OnchipPair pr;
    if (tid == 96) pr = onchip_pair(a, p);
    if (tid == 0) {
        const int32_t s = a.s[p], t = a.t[p];
        const double bn = sqrt(1.0 / a.deg64[s] + 1.0 / a.deg64[t]);
        const T qs = (T)(1.0 / (a.deg64[s] * bn)), qt = (T)(-1.0 / (a.deg64[t] * bn));
        if constexpr (COPY) {
            full[s] = qs;
            full[t] = qt;
        }
        if (s >= row0 && s < row0 + nrow) buf0[R + (s - row0)] = qs;
        if (t >= row0 && t < row0 + nrow) buf0[R + (t - row0)] = qt;
    }
    cluster_arrive();
    cluster_wait();  // q_1 is in place, and every CTA of the cluster runs
    int iprev = 0, icur = 1, iw = 2;
    T bt = T(0);
    // the scalar update of step j (thread 96), its results stored by rank 0
    auto update = [&](int j, const StepCoef& k) { return onchip_update(a, pr, p, j, k, rank == 0); };
    for (int j = 0;; ++j) {
        if (j == a.fin.k_max) {  // the last step's update (it stops there)
            if (tid == 96) update(j - 1, coef);
            break;
        }
        const T* qp = buf0 + iprev * R;
        const T* qc = buf0 + icur * R;
        T* W = buf0 + iw * R;
        double pa = 0.0, pb = 0.0, pc = 0.0;
        bool first = true;
        auto close_row = [&](int ul, T acc) {
            const T wv = (LEAN ? g_invd(ul) : s_invd[ul]) * acc - bt * qp[ul];
            W[ul] = wv;
            const T dw = (LEAN ? g_deg(ul) : s_deg[ul]) * wv;
            if (first) {  // no FP64 addition to zero
                pa = (double)(dw * qc[ul]);
                pb = (double)(dw * wv);
                pc = (double)dw;
                first = false;
            } else {
                pa += (double)(dw * qc[ul]);
                pb += (double)(dw * wv);
                pc += (double)dw;
            }
        };
        const uint32_t cur = (uint32_t)(icur * R) * E;
        auto fetch = [&](uint32_t at) {
            if constexpr (COPY) return full[at];
            else return cluster_ld(at + cur, T(0));
        };
        // the rows' products; `held`: the CTA's entries are in shared memory (a branch per entry
        // would cost more than the loads)
        auto product = [&](auto held) {
            auto where = [&](int e) -> uint32_t {
                if constexpr (decltype(held)::value) return s_col[e];
                else return locate(e);
            };
            auto weight = [&](int e) {
                if constexpr (decltype(held)::value) return s_w[e];
                else return __ldg(a.w + ebase + e);
            };
            for (int ul = tid; ul < nrow; ul += nthr) {
                int e = rp(ul);
                const int e1 = rp(ul + 1);
                if (e1 - e > a.heavy_thr) continue;
                T acc = T(0);
                // gathers in flight four at a time, added in order; the first is not added to zero
                auto four = [&](bool open) {
                    uint32_t at[4];
                    float we[4];
                    T x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        at[u] = where(e + u);
                        if constexpr (WEIGHTED && !decltype(held)::value) we[u] = weight(e + u);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[u] = fetch(at[u]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if constexpr (WEIGHTED) {
                            if constexpr (decltype(held)::value) we[u] = weight(e + u);
                            if (open && u == 0) acc = (T)we[0] * x[0];
                            else acc += (T)we[u] * x[u];
                        } else {
                            if (open && u == 0) acc = x[0];
                            else acc += x[u];
                        }
                    }
                    e += 4;
                };
                if (e + 4 <= e1) four(true);
                while (e + 4 <= e1) four(false);
                for (; e < e1; ++e) {
                    const T x = fetch(where(e));
                    if constexpr (WEIGHTED) acc += (T)weight(e) * x;
                    else acc += x;
                }
                close_row(ul, acc);
            }
            for (int64_t h = warp; h < a.n_heavy_rows; h += nwarps) {
                const int ul = a.heavy_rows[h] - row0;
                if (ul < 0 || ul >= nrow) continue;
                T acc = T(0);
                const int e1 = rp(ul + 1);
                for (int e = rp(ul) + lane; e < e1; e += 32) {
                    const T x = fetch(where(e));
                    if constexpr (WEIGHTED) acc += (T)weight(e) * x;
                    else acc += x;
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) acc += shfl_xor_t(0xffffffffu, acc, off);
                if (lane == 0) close_row(ul, acc);
            }
        };
        if (cached) product(std::true_type{});
        else product(std::false_type{});
        tpart[0][tid] = pa;
        tpart[1][tid] = pb;
        tpart[2][tid] = pc;
        __syncthreads();
        // one warp a sum, each on its own quarter of the SM: lane l adds threads l, l+32, ... in
        // order, then a fixed xor tree; lane r < C writes it into slot `rank` of CTA r
        const bool updates = warp == 3 && j > 0;
        StepCoef kprev;
        if (warp < 3) {
            double s = tpart[warp][lane];
#pragma unroll
            for (int w = 1; w < nwarps; ++w) s += tpart[warp][w * 32 + lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane < C) cluster_st(cluster_addr(smem_addr(&part[warp][rank]), lane), s);
        } else if (updates) {
            kprev = coef;  // rewritten behind the barrier
        }
        __syncwarp();
        cluster_arrive();
        if (updates && lane == 0) stop_s = update(j - 1, kprev) ? 1 : 0;
        __syncwarp();
        cluster_wait();  // all partial sums have arrived
        if (warp == 0) {
            // eight lanes a sum: partials i and i + 8, then a fixed xor tree
            const int q = lane >> 3, i = lane & 7;
            double s = 0.0;
            if (q < 3 && i < C) s = part[q][i];
            if (C > 8) s += q < 3 ? part[q][i + 8] : 0.0;
            for (int off = (C < 8 ? C : 8) >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            const double A = __shfl_sync(0xffffffffu, s, 0), B = __shfl_sync(0xffffffffu, s, 8);
            const double Cs = __shfl_sync(0xffffffffu, s, 16);
            const StepCoef k = step_coef(a.fin, isd, A, B, Cs);
            if (lane == 0) {
                coef = k;
                next[0] = (T)k.inv_beta;
                next[1] = (T)k.alpha;
                next[2] = (T)k.cdef;
                next[3] = (T)k.beta;
            }
        }
        __syncthreads();
        if (stop_s) break;  // step j - 1 ended the pair: the same decision in every CTA of the cluster
        const T ib = next[0], al = next[1], cd = next[2];
        bt = next[3];
        for (int ul = tid; ul < nrow; ul += nthr) {
            const T x = (W[ul] - al * qc[ul] - cd) * ib;
            W[ul] = x;
            if constexpr (COPY)
                for (int r = 0; r < C; ++r) cluster_st(rbase[r] + (uint32_t)(row0 + ul) * E, x);
        }
        const int old_prev = iprev;
        iprev = icur;
        icur = iw;
        iw = old_prev;
        cluster_arrive();
        cluster_wait();  // the new q_i is complete in every CTA before the next product reads it
    }
    cluster_arrive();
    cluster_wait();  // no CTA leaves while another may still address its shared memory
}

// Cluster size for the whole-recurrence kernel: as many CTAs per pair as keep every pair's
// cluster resident at once (npairs * C <= SMs), at least 64 rows per CTA, at most 16.
static int cluster_size(const OnchipArgs& a)
{
    if (!a.allow_cluster || a.n_heavy_rows > 64) return 1;
    int C = 1;
    while (C < kClusterMax && (int64_t)a.npairs * C * 2 <= a.sm_count && a.n >= (int64_t)64 * C) C <<= 1;
    return C;
}

// Rows per CTA, even so that what follows them stays 8-byte aligned.
static int cluster_rows(const OnchipArgs& a, int C) { return (int)(((a.n + C - 1) / C + 1) & ~1ll); }

// Threads per CTA: a row each up to 512 rows: the products wait on shared-memory latency, and more
// warps hide it (1,000 vertices on 2 CTAs, FP32: 10,300 cycles a step with two rows a thread).
static int cluster_threads(const OnchipArgs& a, int C) { return cluster_rows(a, C) <= 256 ? 256 : 512; }

static size_t cluster_entry_bytes(const OnchipArgs& a, ClusterForm form)
{
    return (a.weighted ? 4 : 0) + (form == kCopy ? 2 : 4);
}

// Entries a CTA of this form has room for (whole words, within the limit); -1 if its rows do not fit.
static int64_t cluster_room(const OnchipArgs& a, int C, ClusterForm form)
{
    const size_t base = cluster_base_bytes(form, a.n, cluster_rows(a, C), a.elem_size);
    if (base > kClusterSmemMax || a.n > 65535) return -1;
    return form == kLean ? 0 : (int64_t)((kClusterSmemMax - base) / cluster_entry_bytes(a, form)) & ~(int64_t)1;
}

// KB of an SM's 256 that shared memory takes when `bytes` of it are in use; the L1 has the rest.
static int smem_split(size_t bytes)
{
    for (int kb : {8, 16, 32, 64, 100, 132, 164, 196})
        if (bytes <= (size_t)kb * 1024) return kb;
    return 228;
}

// How far over the L1 the lines are that the threads of an SM read entries from (12 KB of it left to
// the rest): a thread walks its row in order, so until it leaves a 128-byte line the line has to
// stay. `blocks` of `smem` bytes and `threads` threads are resident.
static double l1_pressure(const OnchipArgs& a, int blocks, int threads, size_t smem)
{
    const double row = a.n > 0 ? 4.0 * (double)a.nnz / (double)a.n : 0.0;
    return blocks * threads * std::min(row, 128.0) * (a.weighted ? 2 : 1) / (1024.0 * (244 - smem_split(blocks * smem)));
}

// Bytes of an SM that one block takes.
static size_t cluster_footprint(const OnchipArgs& a, int C, size_t dynamic)
{
    return dynamic + 24 * (size_t)cluster_threads(a, C) + 512 + 1024;  // tpart, the rest, the system's
}

// Blocks of `smem` bytes that share an SM, at most `most` (by their registers).
static int resident_blocks(const OnchipArgs& a, size_t smem, int64_t most)
{
    const int64_t want = ((int64_t)a.npairs + a.sm_count - 1) / a.sm_count, fit = (int64_t)(228 * 1024 / smem);
    return (int)std::max<int64_t>(1, std::min({want, fit, most}));
}

// Launches the kernel with C CTAs per pair; 0 if it does not fit. Where the entries fit on average, for
// C > 1 they get all the shared memory that is left (one CTA of a cluster then occupies an SM: the
// FP64 rate per SM is what a cluster multiplies), and for C = 1 what the graph needs, so that several
// pairs share an SM. Where they do not, they are read from global memory and the space is left to
// the L1 cache, but for what keeps a cluster's CTAs on SMs of their own: 64 pairs, weighted, rows
// of 28 entries, FP32, 4,000 vertices: 2,351 us with all of it reserved, 934 now (8,000: 4,469 and 2,045).
template <typename T, bool WEIGHTED, ClusterForm FORM, int NT>
static int launch_cluster_t(cudaStream_t st, const OnchipArgs& a, int C)
{
    auto k = k_lanczos_cluster<T, WEIGHTED, FORM, NT>;
    ClusterLayout L;
    L.C = C;
    L.R = cluster_rows(a, C);
    L.inv_R = (uint32_t)(((1ull << 32) + L.R - 1) / L.R);
    const int64_t room = cluster_room(a, C, FORM);
    if (room < 0) return 0;
    const bool held = a.nnz <= room * C;
    L.nnz_cap = !held ? 0 : (int)(C > 1 ? room : (a.nnz + 1) & ~(int64_t)1);
    size_t sm = cluster_base_bytes(FORM, a.n, L.R, (int)sizeof(T)) + L.nnz_cap * cluster_entry_bytes(a, FORM);
    if (C > 1) sm = std::max(sm, kClusterSmemMin);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmemMax) != cudaSuccess)
        return 0;
    if (C > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    // no more of the SM than the resident blocks take (100 FP64 pairs of 4,000 weighted vertices, rows of
    // 56 entries, lean: 10,108 us with the default split, 5,454 so)
    int carve = cudaSharedmemCarveoutDefault;
    if (!held) {
        const size_t foot = cluster_footprint(a, C, sm);
        carve = 100 * smem_split((C > 1 ? 1 : resident_blocks(a, foot, 2)) * foot) / 228;
    }
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, carve);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.npairs * C), 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (C > 1 && (cudaOccupancyMaxActiveClusters(&nclusters, k, &cfg) != cudaSuccess || nclusters < 1)) {
        cudaGetLastError();
        return 0;
    }
    if (cudaLaunchKernelEx(&cfg, k, a, L) != cudaSuccess) {
        cudaGetLastError();  // a refused configuration is not sticky: try a smaller cluster
        return 0;
    }
    return C;
}

template <typename T, bool WEIGHTED, ClusterForm FORM>
static int launch_cluster_n(cudaStream_t st, const OnchipArgs& a, int C)
{
    return cluster_threads(a, C) == 256 ? launch_cluster_t<T, WEIGHTED, FORM, 256>(st, a, C)
                                        : launch_cluster_t<T, WEIGHTED, FORM, 512>(st, a, C);
}

template <typename T, bool WEIGHTED>
static int launch_cluster_f(cudaStream_t st, const OnchipArgs& a, int C, ClusterForm form)
{
    return form == kCopy ? launch_cluster_n<T, WEIGHTED, kCopy>(st, a, C)
           : form == kGather ? launch_cluster_n<T, WEIGHTED, kGather>(st, a, C)
                             : launch_cluster_n<T, WEIGHTED, kLean>(st, a, C);
}

static int launch_cluster(cudaStream_t st, const OnchipArgs& a, int C, ClusterForm form)
{
    if (a.elem_size == 8)
        return a.weighted ? launch_cluster_f<double, true>(st, a, C, form) : launch_cluster_f<double, false>(st, a, C, form);
    return a.weighted ? launch_cluster_f<float, true>(st, a, C, form) : launch_cluster_f<float, false>(st, a, C, form);
}

// The form for C CTAs per pair, or kOneBlock: k_lanczos_onchip on one CTA. Where the entries fit, copies
// where a pair's CTAs write fewer elements than they would gather (see above). Where they do not, an
// SM's L1 decides. 30 fixed steps, us, FP32 (unweighted | weighted), pressures in brackets:
//  - one CTA, 100 pairs, copies against kOneBlock: 4,000 vertices, rows of 56: 1,729 | 3,072 (0.6 | 1.2)
//    and 1,875 | 3,315; 7,000 vertices, rows of 14: 1,188 | 1,557 (1.8 | 3.6) and 969 | 1,266, of 28: 2,528 |
//    7,246 and 1,585 | 2,715; 300 pairs, two on an SM, 2,500 vertices, rows of 28: 1,047 | 1,957 (1.4 |
//    2.9) and 1,571 | 2,151, of 56: 1,919 | 4,349 (1.6 | 3.3) and 2,523 | 4,060;
//  - kOneBlock against lean: 100 pairs, 13,000 weighted vertices, rows of 28: 5,170 (2.9) and 5,786; 8,400
//    FP64 vertices, rows of 56: 9,575 (8.2) and 6,713; on two CTAs, 64 pairs, 18,000 vertices, rows of 14:
//    2,165 | 4,877 (3.6 | 7.2) and 3,036 | 3,120. FP64 steps are bound by the SM's FP64 unit, of which two
//    CTAs always have twice as much;
//  - two CTAs, 64 pairs, copies against lean: 12,000 vertices, rows of 28: 2,381 | 4,144 (3.6 | 7.2) and
//    3,957 | 4,113, of 56: 6,136 | 10,746 (4.1 | 8.2) and 7,396 | 7,790.
enum { kOneBlock = -1, kNoForm = -2 };
static int cluster_form(const OnchipArgs& a, int C)
{
    const ClusterForm wish = a.n * (C - 1) <= a.nnz ? kCopy : kGather;
    const int64_t room = cluster_room(a, C, wish);
    if (room >= 0 && a.nnz <= room * C) return wish;
    int resident = 1;
    auto pressure = [&](ClusterForm f) {
        if (cluster_room(a, C, f) < 0) return 1e30;
        size_t sm = cluster_base_bytes(f, a.n, cluster_rows(a, C), a.elem_size);
        if (C > 1) sm = std::max(sm, kClusterSmemMin);
        const size_t foot = cluster_footprint(a, C, sm);
        resident = C > 1 ? 1 : resident_blocks(a, foot, 2);
        return l1_pressure(a, resident, cluster_threads(a, C), foot);
    };
    const double lean = pressure(kLean), copy = pressure(kCopy);
    if (copy <= (C > 1 ? 6.0 : (resident > 1 ? 3.1 : (a.elem_size == 8 ? 2.0 : 1.4)))) return kCopy;
    const size_t one = onchip_smem_bytes(a.n, a.elem_size) + 2048;
    const double block = one > 222 * 1024 ? 1e30 : l1_pressure(a, 1, kOnchipThreads, one);
    if (block <= (C > 1 && a.weighted ? 2.0 : 4.0) && (C == 1 || a.elem_size == 4)) return kOneBlock;
    if (lean < block || (C > 1 && lean < 1e30)) return kLean;
    return block < 1e30 ? kOneBlock : kNoForm;
}

bool launch_check_ids(cudaStream_t st, const OnchipArgs& a)
{
    if (a.npairs <= kScanPairs) return false;
    k_check_ids<<<(a.npairs + 255) / 256, 256, 0, st>>>(a);
    return true;
}

int launch_onchip(cudaStream_t st, const OnchipArgs& a)
{
    for (int C = cluster_size(a); C >= 1; C >>= 1) {
        const int form = cluster_form(a, C);
        if (form == kOneBlock) break;
        const int used = form == kNoForm ? 0 : launch_cluster(st, a, C, (ClusterForm)form);
        if (used) return used;
    }
    // kOneBlock, and graphs whose three vectors fit in one SM but nothing beside them
    const size_t sm = onchip_smem_bytes(a.n, a.elem_size);
    if (sm > 220 * 1024) return 0;
    auto launch = [&](auto k) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k<<<a.npairs, kOnchipThreads, sm, st>>>(a);
    };
    if (a.elem_size == 8) {
        launch(a.weighted ? k_lanczos_onchip<double, true, true> : k_lanczos_onchip<double, false, true>);
    } else if (a.weighted) {
        launch(k_lanczos_onchip<float, true, true>);
    } else {
        const bool by4 = a.nnz <= 40 * a.n || l1_pressure(a, 1, kOnchipThreads, sm + 2048) > 2.0;
        launch(by4 ? k_lanczos_onchip<float, false, true> : k_lanczos_onchip<float, false, false>);
    }
    return 1;
}

}  // namespace rd
