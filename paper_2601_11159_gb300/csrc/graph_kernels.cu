// Graph ingest kernels: CSR validation and degrees (Section 2.1: d_u = sum of the
// weights of u's edges; Section 2.2: the D^{-1/2} scaling of Ahat, applied here as
// 1/d_u per row because vectors are kept as q = D^{-1/2} v).
#include <math.h>

#include <algorithm>

#include "rd_internal.cuh"

namespace rd {

struct CheckFlags {
    int32_t bad_rowptr;
    int32_t bad_col;
    int32_t bad_weight;
    int32_t zero_degree;
    int32_t asymmetric;
    uint32_t ticket;              // k_degrees: blocks done
    unsigned long long self_loops;
    double sumdeg, inv_sumdeg;    // sum of the degrees and its reciprocal (0 if there is none)
};

static_assert(sizeof(CheckFlags) <= kCheckFlagsBytes, "CheckFlags has its own scratch");

__global__ void k_check_csr(int64_t n, int64_t nnz, const int64_t* rp, const int32_t* col, const float* w,
                            CheckFlags* f)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t u = tid; u < n; u += stride) {
        const int64_t a = rp[u], b = rp[u + 1];
        if (a > b || a < 0 || b > nnz) atomicOr(&f->bad_rowptr, 1);
    }
    if (tid == 0 && (rp[0] != 0 || rp[n] != nnz)) atomicOr(&f->bad_rowptr, 1);
    for (int64_t e = tid; e < nnz; e += stride) {
        const int32_t c = col[e];
        if (c < 0 || (int64_t)c >= n) atomicOr(&f->bad_col, 1);
        if (w) {
            const float x = w[e];
            if (!(x > 0.0f) || !isfinite(x)) atomicOr(&f->bad_weight, 1);
        }
    }
}

// Flags a CSR whose rows are not strictly increasing in column, or which is not symmetric
// entry for entry (row v holds u with the same weight bits as row u holds v): the sparse
// first Lanczos step reads row s's weights in place of row u's.
// `mirror` (nullable) receives the index of entry (v, u) for every entry (u, v).
__global__ void k_rows_not_sorted_symmetric(int64_t n, const int64_t* rp, const int32_t* col, const float* w,
                                            int32_t* mirror, int32_t* flag)
{
    // one warp per row, lanes over its entries
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < n; u += nwarps) {
        const int64_t beg = rp[u], end = rp[u + 1];
        bool bad = false;
        for (int64_t e = beg + lane; e < end && !bad; e += 32) {
            const int32_t v = col[e];
            if (e > beg && v <= col[e - 1]) {
                bad = true;
                break;
            }
            const int64_t vend = rp[v + 1];
            int64_t lo = rp[v], hi = vend;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (col[mid] < (int32_t)u) lo = mid + 1; else hi = mid;
            }
            bad = lo >= vend || col[lo] != (int32_t)u ||
                  (w != nullptr && __float_as_uint(w[lo]) != __float_as_uint(w[e]));
            if (mirror) mirror[e] = (int32_t)lo;
        }
        if (bad) atomicOr(flag, 1);
    }
}

// Self-loops need the row of each entry: one thread per row.
__global__ void k_count_self_loops(int64_t n, const int64_t* rp, const int32_t* col, CheckFlags* f)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
        unsigned long long c = 0;
        for (int64_t e = rp[u]; e < rp[u + 1]; ++e) c += (col[e] == (int32_t)u);
        if (c) atomicAdd(&f->self_loops, c);
    }
}

// Degrees in FP64 and their derived copies, the sum of the degrees (per-block partials, added
// by the last block in a fixed order) and, for new weights, the checks that weights can fail: every one
// finite and positive, and both stored copies of an edge equal (`mirror`, nullable: the index of
// each entry's mirror; entries compare with theirs when it is stored after them). Bound by the
// reads of w and mirror and the gather of w[mirror]. Eight lanes sum a light row and the block a
// heavy one (a row of 4,472 entries took one thread 90 us); the reciprocals are taken afterwards
// by one thread a row, since an FP64 instruction costs the same for 1 lane as for 32. With one
// thread a row, a binary search of every mirror and four launches with four waits, new weights
// for 2M entries took 461 us of kernels (186 for the degrees, 166 for the search); a training step
// on 100,000 vertices, which sets them twice, went from 4.99 to 3.31 ms with one launch and wait.
struct DegArgs {
    int64_t n;
    const int64_t* rp;
    const float* w;               // nullable (unweighted)
    const int32_t* mirror;        // nullable
    int64_t n_heavy_rows;
    int heavy_thr;
    const int32_t* heavy_rows;
    double* deg64;
    double* invdeg64;
    float* deg32;
    float* invdeg32;
    double* block_sum;
    CheckFlags* f;
};

__device__ __forceinline__ void deg_store(const DegArgs& a, int64_t u, double d)
{
    a.deg64[u] = d;
    a.deg32[u] = (float)d;
    const double inv = d > 0.0 ? 1.0 / d : 0.0;
    a.invdeg64[u] = inv;
    a.invdeg32[u] = (float)inv;
    if (!(d > 0.0)) atomicOr(&a.f->zero_degree, 1);
}

// Sum of the weights of entries first, first + step, ... < end, checking each.
__device__ __forceinline__ double deg_sum(const DegArgs& a, int64_t first, int64_t end, int step)
{
    double d = 0.0;
    bool bad = false, asym = false;
#pragma unroll 4
    for (int64_t e = first; e < end; e += step) {
        const float x = __ldg(a.w + e);
        d += (double)x;
        bad |= !(x > 0.0f) || !isfinite(x);
        if (a.mirror) {
            const int64_t m = __ldg(a.mirror + e);
            if (m > e) asym |= __float_as_uint(__ldg(a.w + m)) != __float_as_uint(x);
        }
    }
    if (bad) atomicOr(&a.f->bad_weight, 1);
    if (asym) atomicOr(&a.f->asymmetric, 1);
    return d;
}

__global__ void __launch_bounds__(256) k_degrees(const DegArgs a)
{
    constexpr int L = 8;  // lanes per light row
    __shared__ double sd[256];
    const int tid = threadIdx.x;
    double local = 0.0;
    // 256 rows at a time, in octets dealt round the blocks: the long rows of a graph often have
    // neighbouring ids, and a block of 256 of them would hold up the rest
    auto row_of = [&](int64_t it, int k) { return ((it * 32 + k / 8) * gridDim.x + blockIdx.x) * 8 + k % 8; };
    for (int64_t it = 0; row_of(it, 0) < a.n; ++it) {
        if (a.w) {
            for (int k = tid / L; k < 256; k += 256 / L) {
                const int64_t u = row_of(it, k);
                int64_t beg = 0, end = 0;
                if (u < a.n) {
                    beg = a.rp[u];
                    end = a.rp[u + 1];
                }
                const bool light = end - beg <= a.heavy_thr;
                double d = light ? deg_sum(a, beg + tid % L, end, L) : 0.0;
                __syncwarp();
#pragma unroll
                for (int off = L / 2; off >= 1; off >>= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
                if (tid % L == 0) sd[k] = light ? d : -1.0;
            }
            __syncthreads();
        }
        const int64_t u = row_of(it, tid);
        if (u < a.n) {
            const double d = a.w ? sd[tid] : (double)(a.rp[u + 1] - a.rp[u]);
            if (d != -1.0) {  // heavy rows below
                deg_store(a, u, d);
                local += d;
            }
        }
        __syncthreads();
    }
    if (a.w)
        for (int64_t h = blockIdx.x; h < a.n_heavy_rows; h += gridDim.x) {
            const int64_t u = a.heavy_rows[h];
            if (a.rp[u + 1] - a.rp[u] <= a.heavy_thr) continue;  // summed above
            sd[tid] = deg_sum(a, a.rp[u] + tid, a.rp[u + 1], 256);
            __syncthreads();
            for (int s = 128; s > 0; s >>= 1) {
                if (tid < s) sd[tid] += sd[tid + s];
                __syncthreads();
            }
            if (tid == 0) {
                deg_store(a, u, sd[0]);
                local += sd[0];
            }
            __syncthreads();
        }
    sd[tid] = local;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (tid < s) sd[tid] += sd[tid + s];
        __syncthreads();
    }
    __shared__ bool last;
    if (tid == 0) {
        a.block_sum[blockIdx.x] = sd[0];
        __threadfence();
        last = atomicAdd(&a.f->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double sum = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += 256) sum += __ldcg(a.block_sum + b);
    sd[tid] = sum;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (tid < s) sd[tid] += sd[tid + s];
        __syncthreads();
    }
    if (tid == 0) {
        a.f->sumdeg = sd[0];
        a.f->inv_sumdeg = sd[0] > 0.0 ? 1.0 / sd[0] : 0.0;
    }
}

static int grid_for(int64_t work, int sm)
{
    int64_t g = (work + 255) / 256;
    const int64_t cap = (int64_t)sm * 8;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// Whether the rows are strictly increasing in column and the entries symmetric
// (g->rows_sorted_sym); for a weighted graph also keeps each entry's mirror, against which later
// weights are compared.
rd_status rows_sorted_symmetric(rd_graph* g, cudaStream_t st)
{
    int32_t* f = &static_cast<CheckFlags*>(g->check_scratch)->asymmetric;
    // without memory for the mirrors later weights are searched
    if (g->w && !g->mirror && g->keep_mirror &&
        cudaMalloc((void**)&g->mirror, sizeof(int32_t) * (g->nnz > 0 ? g->nnz : 1)) != cudaSuccess) {
        g->mirror = nullptr;
        cudaGetLastError();
    }
    RD_CUDA(cudaMemsetAsync(f, 0, sizeof(int32_t), st));
    if (g->n > 0)
        k_rows_not_sorted_symmetric<<<grid_for(g->n, g->sm_count), 256, 0, st>>>(g->n, g->row_ptr, g->col, g->w,
                                                                                 g->mirror, f);
    int32_t h = 0;
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    g->rows_sorted_sym = h == 0;
    // the search stops at a row's first fault, so the mirrors are whole only without one
    g->mirror_ok = g->rows_sorted_sym && g->mirror != nullptr;
    return RD_OK;
}

rd_status check_csr(rd_graph* g, cudaStream_t st, int64_t* self_loops)
{
    CheckFlags* f = nullptr;
    RD_CUDA(cudaMallocAsync((void**)&f, sizeof(CheckFlags), st));
    RD_CUDA(cudaMemsetAsync(f, 0, sizeof(CheckFlags), st));
    k_check_csr<<<grid_for(g->nnz > g->n ? g->nnz : g->n, g->sm_count), 256, 0, st>>>(g->n, g->nnz, g->row_ptr,
                                                                                       g->col, g->w, f);
    CheckFlags h{};
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(CheckFlags), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    if (h.bad_rowptr) {
        cudaFreeAsync(f, st);
        set_error("row_ptr must start at 0, be non-decreasing and end at nnz");
        return RD_ERR_INVALID_ARG;
    }
    if (h.bad_col) {
        cudaFreeAsync(f, st);
        set_error("a column index is outside [0, n)");
        return RD_ERR_INVALID_ARG;
    }
    if (h.bad_weight) {
        cudaFreeAsync(f, st);
        set_error("edge weights must be finite and > 0");
        return RD_ERR_INVALID_ARG;
    }
    k_count_self_loops<<<grid_for(g->n, g->sm_count), 256, 0, st>>>(g->n, g->row_ptr, g->col, f);
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(CheckFlags), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaFreeAsync(f, st));
    RD_CUDA(cudaStreamSynchronize(st));
    *self_loops = (int64_t)h.self_loops;
    return RD_OK;
}

int degree_grid(const rd_graph* g) { return grid_for(g->n, g->sm_count); }

// Degrees (and, with check_weights, the weight checks of rd_graph_set_weights) with one launch and
// one wait; `flags_dev` holds a CheckFlags, in which the kernels of a step find the degrees' sum from
// then on, and `block_sums_dev` degree_grid(g) doubles.
rd_status compute_degrees(rd_graph* g, cudaStream_t st, void* flags_dev, double* block_sums_dev, bool check_weights)
{
    CheckFlags* f = static_cast<CheckFlags*>(flags_dev);
    RD_CUDA(cudaMemsetAsync(f, 0, sizeof(CheckFlags), st));
    DegArgs a{};
    a.n = g->n;
    a.rp = g->row_ptr;
    a.w = g->w;
    a.mirror = check_weights && g->mirror_ok ? g->mirror : nullptr;
    a.n_heavy_rows = g->n_heavy_rows;
    a.heavy_thr = std::max(g->heavy_thr, 256);
    a.heavy_rows = g->heavy_rows;
    a.deg64 = g->deg64;
    a.invdeg64 = g->invdeg64;
    a.deg32 = g->deg32;
    a.invdeg32 = g->invdeg32;
    a.block_sum = block_sums_dev;
    a.f = f;
    k_degrees<<<degree_grid(g), 256, 0, st>>>(a);
    RD_CUDA(cudaGetLastError());
    CheckFlags h{};
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(CheckFlags), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    if (check_weights && h.bad_weight) {
        set_error("edge weights must be finite and > 0");
        return RD_ERR_INVALID_ARG;
    }
    g->inv_sumdeg = &f->inv_sumdeg;
    g->mean_deg = g->n ? h.sumdeg / (double)g->n : 0.0;
    if (a.mirror) g->rows_sorted_sym = h.asymmetric == 0;
    if (h.zero_degree && g->n > 1) {
        set_error("a vertex has degree 0 (isolated vertex)");
        return RD_ERR_ZERO_DEGREE;
    }
    return RD_OK;
}

}  // namespace rd

namespace rd {

// Variant of check_csr for callers that cannot allocate: the flag block lives in
// caller-provided device scratch.
rd_status check_csr_scratch(rd_graph* g, cudaStream_t st, void* flags_dev, int64_t* self_loops)
{
    CheckFlags* f = static_cast<CheckFlags*>(flags_dev);
    CheckFlags h{};
    RD_CUDA(cudaMemsetAsync(f, 0, sizeof(CheckFlags), st));
    k_check_csr<<<grid_for(g->nnz > g->n ? g->nnz : g->n, g->sm_count), 256, 0, st>>>(g->n, g->nnz, g->row_ptr,
                                                                                       g->col, g->w, f);
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(CheckFlags), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    if (h.bad_rowptr) {
        set_error("row_ptr must start at 0, be non-decreasing and end at nnz");
        return RD_ERR_INVALID_ARG;
    }
    if (h.bad_col) {
        set_error("a column index is outside [0, n)");
        return RD_ERR_INVALID_ARG;
    }
    if (h.bad_weight) {
        set_error("edge weights must be finite and > 0");
        return RD_ERR_INVALID_ARG;
    }
    k_count_self_loops<<<grid_for(g->n, g->sm_count), 256, 0, st>>>(g->n, g->row_ptr, g->col, f);
    RD_CUDA(cudaMemcpyAsync(&h, f, sizeof(CheckFlags), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    *self_loops = (int64_t)h.self_loops;
    return RD_OK;
}

}  // namespace rd

namespace rd {

// Triangle-count weights (the weighted setting of the paper's Exp-2): for stored entry
// e = (u, v), w(e) = |N(u) & N(v)| (the triangles through edge uv), or 1 when that is 0.
// One thread per entry: every element of the shorter adjacency list is looked up in the
// longer one by binary search (rows must be sorted by column).
__global__ void k_triangle_weights(int64_t n, const int64_t* rp, const int32_t* col, float* w_out, int32_t* unsorted)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
        const int64_t a0 = rp[u], a1 = rp[u + 1];
        for (int64_t e = a0; e < a1; ++e) {
            if (e > a0 && col[e] <= col[e - 1]) atomicOr(unsorted, 1);
            const int64_t v = col[e];
            const int64_t b0 = rp[v], b1 = rp[v + 1];
            int64_t s0 = a0, s1 = a1, l0 = b0, l1 = b1;  // shorter list [s0,s1), longer [l0,l1)
            if (a1 - a0 > b1 - b0) {
                s0 = b0; s1 = b1; l0 = a0; l1 = a1;
            }
            int64_t cnt = 0;
            for (int64_t i = s0; i < s1; ++i) {
                const int32_t x = col[i];
                int64_t lo = l0, hi = l1;
                while (lo < hi) {
                    const int64_t mid = (lo + hi) >> 1;
                    if (col[mid] < x) lo = mid + 1; else hi = mid;
                }
                cnt += (lo < l1 && col[lo] == x);
            }
            w_out[e] = cnt > 0 ? (float)cnt : 1.0f;
        }
    }
}

rd_status triangle_weights(int64_t n, const int64_t* rp, const int32_t* col, float* w_out, int sm_count,
                           cudaStream_t st, int32_t* flag_dev)
{
    RD_CUDA(cudaMemsetAsync(flag_dev, 0, sizeof(int32_t), st));
    k_triangle_weights<<<grid_for(n, sm_count), 256, 0, st>>>(n, rp, col, w_out, flag_dev);
    int32_t h = 0;
    RD_CUDA(cudaMemcpyAsync(&h, flag_dev, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    RD_CUDA(cudaStreamSynchronize(st));
    if (h) {
        set_error("triangle weights need every row's columns sorted increasingly and without duplicates");
        return RD_ERR_INVALID_ARG;
    }
    return RD_OK;
}

}  // namespace rd
