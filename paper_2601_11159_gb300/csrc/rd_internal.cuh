// Internal declarations of librd: graph object, workspace, kernel argument
// blocks and the launcher table. Not part of the public ABI (see include/rd.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/rd.h"
#include "df64.cuh"

namespace rd {

// ----------------------------------------------------------------- errors
void set_error(const std::string& msg);
rd_status cuda_status(cudaError_t e, const char* what);

#define RD_CUDA(call)                                                   \
    do {                                                                \
        cudaError_t _e = (call);                                        \
        if (_e != cudaSuccess) return ::rd::cuda_status(_e, #call);     \
    } while (0)

#define RD_TRY(call)                                                    \
    do {                                                                \
        rd_status _s = (call);                                          \
        if (_s < 0) return _s;                                          \
    } while (0)

// ------------------------------------------------------- SpMM configuration
// One warp is split into row groups of GS*NZL lanes. GS lanes span the
// right-hand-side tile (VEC elements each, so the tile is TP = VEC*GS
// columns); NZL lanes share the nonzeros of one row; RPW = 32/(GS*NZL) rows
// are in flight per warp.
// kind 0: row-group kernel (k_spmm, grid-stride over rows); kind 1: row-stream kernel
// (k_spmm_rows, grid-stride over tasks of consecutive rows; nzl must be 1); kind 2:
// warp-per-task SpMV (one column); kind 3: row-stream kernel with cp.async gathers into a
// shared-memory ring (k_spmm_async, FP32 vectors, vec 4, nzl 1); kind 4: row pipeline for short
// rows (k_spmm_pipe, one 16-byte unit of columns per lane, nzl 1).
struct SpmmCfg {
    int vec = 4, gs = 32, nzl = 1, kind = 0;
    int order = 0;  // row-group kernel: 1 = visit rows by decreasing degree (rd_graph::row_order)
    int tp() const { return vec * gs; }
    int rpw() const { return 32 / (gs * nzl); }
    bool operator==(const SpmmCfg& o) const
    {
        return vec == o.vec && gs == o.gs && nzl == o.nzl && kind == o.kind && order == o.order;
    }
};

// Configuration of the heavy-row pre-pass that goes with a step configuration: the same
// column tile, one whole warp per chunk of a heavy row (GS column lanes x 32/GS nonzero
// lanes), so that a chunk's gathers are spread over the warp instead of one row group.
// The async kernel (kind 3) has its own pre-pass with one row group per chunk.
inline SpmmCfg heavy_cfg(const SpmmCfg& c)
{
    SpmmCfg h;
    h.vec = c.vec;
    h.gs = c.gs;
    h.nzl = c.kind == 3 ? 1 : 32 / c.gs;
    h.kind = c.kind == 3 ? 3 : 0;
    return h;
}

constexpr int kBlock = 256;        // threads per block of the SpMM kernels
constexpr int kWarps = kBlock / 32;
constexpr int kRing = 4;           // increments kept for the delayed error estimate

// Argument block of one Lanczos step's SpMM (q-space: q = D^{-1/2} v).
// The row-stream and async kernels count entries in a signed 32-bit number and step (or look) up to this far
// past a row's end: graphs of more entries than 2^31 - 1 less this take the row-group kernel, whose
// counter has no sign, in their place. (Counting without a sign, from the middle of the range, or by what is
// left costs those two 3-5%: a gradient over 79.8M entries 17.2 -> 17.7 ms.)
constexpr int64_t kStreamReach = 1024;
constexpr int64_t kStreamEntries = (int64_t(1) << 31) - 1 - kStreamReach;
// They hold the offset of a gathered row as 32 bits of the lane's VEC elements: blocks of more units (64 GB at
// 16 bytes a lane) take the row-group kernel as well, whose offsets have 64 bits.
constexpr int64_t kStreamUnits = int64_t(1) << 32;

template <typename T>
struct StepArgs {
    int64_t n, ld;                 // rows, padded columns (row stride of vector blocks)
    const int64_t* row_ptr;
    const int32_t* col;
    const float* w;                // nullable (unweighted)
    const T* invdeg;               // 1/d_u
    const T* deg;                  // d_u
    const T* qcur;                 // q_i  (n x ld)
    const T* qprev;                // q_{i-1}
    T* w_out;                      // W = D^{-1} W_adj q_i - beta_i q_{i-1} (may be qprev's block)
    const T* cf_beta;              // beta_i per column (ld)
    // heavy rows (degree > heavy_thr): chunk partial sums made by the heavy kernel
    int heavy_thr;
    int64_t n_heavy_rows, n_chunks;
    const int32_t* heavy_rows;     // sorted row ids
    const int32_t* heavy_first;    // n_heavy_rows + 1 chunk offsets
    const int32_t* chunk_beg;      // nnz range of each chunk
    const int32_t* chunk_end;
    T* heavy_part;                 // n_chunks x ld
    int64_t hot_rows;              // gathers of rows below this id keep L2 priority (the rest evict first)
    int64_t ntasks;                // row-stream tasks: rows [task_row[i], task_row[i+1])
    const int32_t* task_row;
    double* block_part;            // [slab][block][3][TP]
    const int32_t* active_prev;    // early exit when *active_prev == 0 (nullable)
    int do_reduce;
    int lazy_walk;                 // Power Method step: W = (1/2) q + (1/2) D^{-1} W_adj q (no recurrence)
    // Step index read from device memory (graph replay; nullable): then the step j's
    // beta_i row is cf_beta + j * cf_stride and the early-exit count is act_count[j].
    const int32_t* step_dev;
    int64_t cf_stride;
    const int32_t* act_count;
    // row-group kernel: visiting order of the rows (nullable = 0 .. n-1); rows of equal
    // degree are adjacent, so the row groups of a warp finish their rows together
    const int32_t* row_order;
};

// Step-dependent operands of a StepArgs launch (fixed pointers, or derived from the step
// index in device memory when the launch is replayed from a CUDA graph).
template <typename T>
__device__ __forceinline__ const T* step_cf_beta(const StepArgs<T>& a)
{
    return a.step_dev ? a.cf_beta + (int64_t)(*a.step_dev) * a.cf_stride : a.cf_beta;
}

template <typename T>
__device__ __forceinline__ bool step_inactive(const StepArgs<T>& a)
{
    const int32_t* p = a.step_dev ? a.act_count + *a.step_dev : a.active_prev;
    return p != nullptr && *p == 0;
}

template <typename T>
struct NormArgs {
    int64_t n, ld;
    T* w_to_qnext;                 // in: W, out: q_{i+1} (in place)
    const T* qcur;
    const T* cf;                   // [4][ld]: beta_i, alpha_i, c_i, 1/beta_{i+1}
    T* phi;                        // nullable: phi += coef * q_i (replay pass)
    const T* coef;                 // ld, with phi
    const int32_t* active_prev;
    const int32_t* step_dev;       // as StepArgs: cf + j * cf_stride, act_count[j]
    int64_t cf_stride;
    const int32_t* act_count;
    // potential accumulated during the forward pass (nullable pvec: off)
    T* pvec;                       // p_{i-1} in, p_i out
    T* xvec;                       // x += mu_i p_i
    const T* xcf;                  // [2][ld]: lambda_i, mu_i (+ j * xcf_stride with step_dev)
    int64_t xcf_stride;
};

// End of a pass of up to `m` steps whose vectors were kept (k_potential_pass). Blocks of n x ld
// elements, `stride` elements apart: block 0 holds W of the pass's last step, block 1 + i the
// vector q of its step i.
constexpr int kPotSteps = 8;
template <typename T>
struct PotPassArgs {
    int64_t n, ld, stride;
    int m, k_max;
    T* blocks;
    T* pvec;                      // p of the last step before the pass in, of its last step out
    T* xvec;                      // x += sum over the pass's steps of mu_i p_i
    const T* cf;                  // [k_max + 1][4][ld] coefficients by step
    const T* xcf;                 // [k_max][2][ld]: lambda_i, mu_i by step
    const int32_t* act_count;
    int32_t* base;                // first step of the pass; advanced by m at its end
    int32_t* ticket;              // blocks done (0 between launches)
};

// Normalise pass fused with a column compaction (k_normalize_pack).
template <typename T>
struct NormPackArgs {
    int64_t n, ld_old, ld_new;
    const T* w;                    // W, old layout
    const T* qcur;                 // q_i, old layout
    const T* cf;                   // [4][ld_old]: beta_i, alpha_i, c_i, 1/beta_{i+1} of the step
    const int32_t* old_slot;       // [ld_new]: source column of each packed column, -1 none
    T* qnext_new;                  // q_{i+1}, packed (n x ld_new)
    T* qcur_new;                   // q_i, packed (n x ld_new)
};

// Per-pair FP64 state of the running LDL^T factorisation of I - T_k.
struct PairState {
    double* b2;        // ||b||^2 = 1/d_s + 1/d_t
    double* bnorm;     // ||b||
    double* delta;     // last pivot
    double* inv_delta; // 1 / delta
    double* g;         // last entry of L^{-1} e_1
    double* S;         // e_1^T (I - T_k)^{-1} e_1
    double* beta;      // beta_{k+1}
    double* ring;      // kRing x ld increments
    double* r;         // b2 * S
    double* err;       // estimated relative error
    int32_t* k;        // steps done
    int32_t* status;   // rd_status per pair
    int32_t* active;   // 1 while iterating
    double* hist_alpha;   // k_max x ld
    double* hist_beta;    // (k_max + 1) x ld: beta_1 .. beta_{k_max+1}
    int32_t* act_count;   // k_max + 1 counters: active pairs entering step j
};

struct FinArgs {
    int64_t ld;
    int npairs, tp, nblocks, step;      // step: 0-based index of the step just reduced
    int k_max, deflate, fixed_k, fp64;
    double rel_tol, resid_tol;
    const double* inv_sumdeg;           // 1 / sum of the degrees, on the device: new weights leave the
                                        // arguments, and with them the captured graphs, as they are
    int est_delayed;                    // 1: delayed-sum error estimate (RD_Q_EST_DELAYED)
    const double* block_part;
    PairState st;
    int64_t pstride;                    // stride of the per-pair [k][pair] arrays (original ld)
    const int32_t* slot_pair;           // column slot -> pair (-1: empty); NULL = identity
    void* cf_step;                      // T [4][ld]: rows 1..3 receive alpha_i, c_i, 1/beta_{i+1}
    void* cf_next;                      // T [4][ld]: row 0 receives beta_{i+1} for the next step
    int elem_size;
    const int32_t* step_dev;            // nullable: step index from device memory (graph replay);
    int64_t cf_stride;                  // then cf_step/cf_next advance by j * cf_stride
    int df;                             // 1: coefficients are stored as double-float pairs
    void* xcf;                          // nullable T [k_max][2][ld]: step j receives lambda_i, mu_i
                                        // of the potential's direct update (identity slot map only)
    // device-resident step loop (see k_finalize and k_loop_entry)
    int loop;                           // 1: this launch is in the loop's body; 2: it only advances
                                        // loop_step and loop_norm (no conditional node)
    int loop_compact, loop_lag;         // test for a column compaction, on the count `lag` steps back
    unsigned long long loop_handle;     // the while node's cudaGraphConditionalHandle
    int32_t* loop_step;                 // step index of the body's pre-pass, SpMM and finalize
    int32_t* loop_norm;                 // step index of the body's normalise pass
    int32_t* loop_ticket;               // finalize blocks done (0 between steps)
    int32_t* loop_saved;                // [4]: where the loop stopped
    const int32_t* loop_cfrom;          // first step at which a compaction is tested for
};

// Whole recurrence of one pair per CTA with q_{i-1}, q_i and W in shared memory (graphs
// small enough); reads the CSR from global memory (L1/L2 resident).
struct OnchipArgs {
    int64_t n, nnz;
    int npairs;
    const int64_t* row_ptr;
    const int32_t* col;
    const float* w;
    const double* deg64;
    const double* invdeg64;
    const float* deg32;
    const float* invdeg32;
    const int32_t* s;
    const int32_t* t;
    int heavy_thr;
    int64_t n_heavy_rows;
    const int32_t* heavy_rows;
    FinArgs fin;                  // stop rule, tolerances, per-pair state
    int elem_size, weighted;
    int sm_count;                 // SMs of the device (cluster size choice)
    int allow_cluster;            // 0: one CTA per pair (RD_Q_NO_CLUSTER)
    const int32_t* comp;          // nullable: component of each vertex
    // results per pair, and the call's flags (zero on entry): [0] a pair did not converge, [1] a
    // pair ended RD_ERR_NUMERIC, [2] a pair id is out of range (then nothing else is written)
    double* r_out;
    int32_t* iters_out;
    double* err_out;
    int32_t* status_out;
    int32_t* summary;
};
size_t onchip_smem_bytes(int64_t n, int elem_size);
// Launches the whole-recurrence kernel; returns the CTAs per pair used (1: one CTA per pair,
// 2..16: a thread-block cluster per pair), or 0 if the graph does not fit.
int launch_onchip(cudaStream_t st, const OnchipArgs& a);
// The kernel that looks a large batch's ids over before launch_onchip; false if the batch needs none.
bool launch_check_ids(cudaStream_t st, const OnchipArgs& a);

// Column compaction: keep the slots whose pair is still active, in slot order.
struct CompactArgs {
    int64_t n, ld_old, ld_new;
    const int32_t* slot_pair_old;       // NULL = identity over npairs
    int npairs;
    int32_t* slot_pair_new;             // ld_new
    int32_t* old_slot;                  // ld_new: source slot or -1
    const int32_t* active;              // per pair
    const void* cf_old;                 // T [4][ld_old]
    void* cf_new;                       // T [4][ld_new]
    const void* q_src0;                 // T n x ld_old
    const void* q_src1;
    void* q_dst0;                       // T n x ld_new
    void* q_dst1;
    int elem_size;
};
void launch_compact(cudaStream_t st, int grid, const CompactArgs& a);
// the slot maps and the packed coefficients only (the q blocks packed by the caller)
void launch_compact_map(cudaStream_t st, const CompactArgs& a);

// Power Method (Algorithm 1) in y = D^{-1} r: start y = D^{-1}(e_s - e_t), accumulate
// rbar += (y_s - y_t)/2 per step (r(s)/(2 d_s) - r(t)/(2 d_t) of Algorithm 1).
struct PmArgs {
    int64_t n, ld;
    int npairs;
    const int32_t* s;
    const int32_t* t;
    const double* deg64;
    void* y;                      // T n x ld
    double* rbar;                 // npairs
    double* hist;                 // nullable: [step][npairs]
    int step, elem_size;
    int32_t* err_flag;
};
void launch_pm_init(cudaStream_t st, const PmArgs& a);
void launch_pm_accum(cudaStream_t st, const PmArgs& a);

constexpr int kStagePairs = 2048;

// Whether kernels on `device` may use a caller's array at p in place: memory of that device (a peer's
// is reached by copies alone) or managed memory, aligned to its elements as the kernels' loads
// and stores need it (a copy takes any address).
inline bool usable_in_place(cudaMemoryType type, int mem_device, int device, const void* p, size_t align)
{
    if (type != cudaMemoryTypeManaged && !(type == cudaMemoryTypeDevice && mem_device == device)) return false;
    return reinterpret_cast<uintptr_t>(p) % align == 0;
}

inline bool ranges_overlap(const void* a, size_t na, const void* b, size_t nb)
{
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return a && b && x < y + nb && y < x + na;
}

// --------------------------------------------------------------- graph
struct Workspace {
    void* base = nullptr;
    size_t bytes = 0;
};

}  // namespace rd

struct rd_graph {
    int device = 0, sm_count = 0;
    int64_t n = 0, nnz = 0, nnz_in = 0;
    bool weighted = false;
    int64_t* row_ptr = nullptr;
    int32_t* col = nullptr;
    float* w = nullptr;
    int64_t* keep_idx = nullptr;      // internal entry -> original entry (only if self-loops dropped)
    double* deg64 = nullptr;
    double* invdeg64 = nullptr;
    float* deg32 = nullptr;
    float* invdeg32 = nullptr;
    rd::df64* degdf = nullptr;        // double-float copies (built on first use)
    rd::df64* invdegdf = nullptr;
    const double* inv_sumdeg = nullptr;  // 1 / sum of the degrees (device, in compute_degrees' flags)
    int32_t* mirror = nullptr;        // weighted graphs: entry (v, u) of each entry (u, v)
    bool mirror_ok = false;           // rows sorted and the structure symmetric: mirror is whole
    bool keep_mirror = true;          // false: given back for a workspace that did not fit beside it
    void* check_scratch = nullptr;    // flags and block sums of compute_degrees
    int32_t* comp = nullptr;
    int32_t ncomp = 0;
    // heavy-row chunks
    int heavy_thr = 256;
    int64_t n_heavy_rows = 0, n_chunks = 0;
    int32_t* heavy_rows = nullptr;
    int32_t* heavy_first = nullptr;
    int32_t* chunk_beg = nullptr;
    int32_t* chunk_end = nullptr;
    // row-stream tasks: consecutive rows with at most task_length() nonzeros, heavy rows alone; the
    // one-column SpMV has its own of at most 512
    int64_t ntasks = 0, n_spmv_tasks = 0;
    int32_t* task_row = nullptr;
    int32_t* spmv_task_row = nullptr;
    // rows by decreasing degree (stable: equal degrees in row order)
    int32_t* row_order = nullptr;
    // row of every stored entry (built on first use by the per-entry kernels)
    int32_t* entry_row = nullptr;

    bool rows_sorted_sym = false;     // rows strictly increasing in column, entries symmetric
    double mean_deg = 0.0;
    rd::Workspace ws;
    rd_call_stats stats{};
    int* h_pinned = nullptr;          // small pinned host buffer for polls (16 ints)
    int32_t* h_stage = nullptr;       // behind it, pinned: ids of up to kStagePairs pairs on their way in
    int64_t l2_bytes = 0;             // device L2 size
    // SpMM configurations chosen by the autotuner on this graph, per width class
    struct TunedCfg {
        int prec = 0, single = 0;     // element precision (0 FP32, 1 FP64, 2 double-float); one column or many
        int64_t width = 0;            // width class (power-of-two tile holding the pairs; 1 if single)
        // every candidate with the measured time of one SpMM launch pair at `width` columns
        std::vector<std::pair<rd::SpmmCfg, float>> times;
    };
    std::vector<TunedCfg> tuned;
    // instantiated CUDA graphs of two Lanczos steps, keyed by the bytes of their launch
    // arguments (oldest evicted first), and the stream they are captured on
    std::vector<std::pair<std::string, cudaGraphExec_t>> graphs;
    cudaStream_t capture_stream = nullptr;
};

namespace rd {

// Launchers (defined in the kernel translation units).
// Returns false if the configuration is not instantiated.
bool launch_spmm_f32(const SpmmCfg& c, bool weighted, bool heavy, int grid, cudaStream_t st,
                     const StepArgs<float>& a);
bool launch_spmm_df64(const SpmmCfg& c, bool weighted, bool heavy, int grid, cudaStream_t st,
                      const StepArgs<df64>& a);
bool launch_spmm_f64(const SpmmCfg& c, bool weighted, bool heavy, int grid, cudaStream_t st,
                     const StepArgs<double>& a);
// prec: 0 FP32 vectors, 1 FP64, 2 double-float
int spmm_blocks_per_sm(const SpmmCfg& c, bool weighted, bool heavy, int prec);
std::vector<SpmmCfg> spmm_configs(bool fp64);

void launch_potential_pass_f32(int grid, cudaStream_t st, const PotPassArgs<float>& a);
void launch_potential_pass_f64(int grid, cudaStream_t st, const PotPassArgs<double>& a);
void launch_normalize_f32(int grid, cudaStream_t st, const NormArgs<float>& a);
void launch_normalize_f64(int grid, cudaStream_t st, const NormArgs<double>& a);
void launch_normalize_df64(int grid, cudaStream_t st, const NormArgs<df64>& a);
// false when the packed layout has no whole 16-byte units (the caller then packs separately)
bool launch_normalize_pack_f32(int grid, cudaStream_t st, const NormPackArgs<float>& a);
bool launch_normalize_pack_f64(int grid, cudaStream_t st, const NormPackArgs<double>& a);
bool launch_normalize_pack_df64(int grid, cudaStream_t st, const NormPackArgs<df64>& a);
void launch_split_df(cudaStream_t st, int grid, int64_t n, const double* src, df64* dst);
void launch_finalize(cudaStream_t st, const FinArgs& a);
// Advance the device step index by one, saturating at `limit` (end of a replayed step).
void launch_step_advance(cudaStream_t st, int32_t* step, int limit);
// Entry condition of the device-resident step loop, on its finalize launch's arguments.
void launch_loop_entry(cudaStream_t st, const FinArgs& a);

struct InitArgs {
    int64_t n, ld;
    int npairs, k_max, elem_size;
    int df;                       // 1: vectors are double-float pairs (elem_size 8)
    const int32_t* s;
    const int32_t* t;
    const double* deg64;
    const int32_t* comp;          // nullable
    void* qcur;                   // T n x ld (zeroed before)
    PairState st;
    int32_t* err_flag;
    int replay;                   // 1: only rebuild q_1 (the per-pair state is left untouched)
};
void launch_init(cudaStream_t st, const InitArgs& a);

struct OutArgs {
    int npairs;
    int64_t ld;
    PairState st;
    double* r_out;
    int32_t* iters_out;
    double* err_out;
    int32_t* status_out;
    int32_t* summary;            // [0]: any not converged, [1]: any numeric
    const int32_t* err_flag;     // set: a pair id is out of range, and nothing is written
};
void launch_output(cudaStream_t st, const OutArgs& a);

struct ZsolveArgs {
    int npairs;
    int64_t ld;
    int k_max;
    PairState st;
    const double* grad_r;         // nullable (ones)
    void* coef_hist;              // T [k_max][ld]: sqrt(b2) * z_j (0 beyond k_p)
    void* gbar;                   // T [ld]: upstream gradient per column (0 if unused)
    double* zscratch;             // [k_max][2][ld]
    int elem_size;
};
void launch_zsolve(cudaStream_t st, const ZsolveArgs& a);

template <typename T>
struct EdgeGradArgs {
    int64_t n, ld, nnz;
    int npairs;
    const int64_t* row_ptr;
    const int32_t* col;
    const int32_t* entry_row;     // row of each stored entry (nnz)
    const T* phi;                 // n x ld
    const T* gbar;                // ld
    float* grad_out;              // internal entries
};
void launch_edge_grad_f32(int grid, cudaStream_t st, const EdgeGradArgs<float>& a);
void launch_edge_grad_f64(int grid, cudaStream_t st, const EdgeGradArgs<double>& a);
void launch_entry_rows(int grid, cudaStream_t st, int64_t n, const int64_t* row_ptr, int32_t* entry_row);


// Pair-major float output of the potential block: out[p][i] = phi[i][p] of vertex i (potentials),
// or, with `row`, phi[row[i]][p] - phi[col[i]][p] of entry i, stored at keep_idx[i] (flows).
struct PairMajorArgs {
    int64_t items, ld, out_stride;
    int npairs;
    const void* phi;              // T n x ld
    const int32_t* row;           // nullable
    const int32_t* col;
    const int64_t* keep_idx;      // nullable: identity
    float* out;
};
void launch_pair_major(cudaStream_t st, bool fp64, const PairMajorArgs& a);

// First Lanczos step from the sparse start vector (two nonzeros per column).
template <typename T>
struct Step0Args {
    int64_t n, ld;
    int npairs;
    int tp;                       // column tile of the plan (layout of block_part)
    const int64_t* row_ptr;
    const int32_t* col;
    const float* w;               // nullable
    const T* invdeg;
    const double* deg64;
    const int32_t* s;
    const int32_t* t;
    const T* q1;                  // q_1 block (n x ld)
    T* wout;                      // W, written over the zeroed q_0 block
    double* block_part;           // [slab][1][3][TP]: each column's sums as one block (nullable)
};
// Step 0's normalise pass after the sparse first step, in two parts: the rows of
// N(s) ∪ N(t) ∪ {s, t} of each column (k_normalize_step0, marking them in `mask`), then every
// other entry (k_normalize_step0_fill), where W_1 and q_1 are zero.
template <typename T>
struct Step0NormArgs {
    int64_t n, ld;
    int npairs;
    const int64_t* row_ptr;
    const int32_t* col;
    const int32_t* s;
    const int32_t* t;
    const T* q1;                  // q_1 block
    T* w;                         // in: W_1 on those rows (k_step0_sparse's output), out: q_2
    const T* cf;                  // [4][ld]: beta_1, alpha_1, c_1, 1/beta_2
    uint32_t* mask;               // n x ld bits, zero on entry: the entries the first part wrote
};
void launch_normalize_step0_f32(int grid, cudaStream_t st, const Step0NormArgs<float>& a);
void launch_normalize_step0_f64(int grid, cudaStream_t st, const Step0NormArgs<double>& a);
void launch_normalize_step0_df64(int grid, cudaStream_t st, const Step0NormArgs<df64>& a);
void launch_step0_f32(cudaStream_t st, const Step0Args<float>& a);
void launch_step0_f64(cudaStream_t st, const Step0Args<double>& a);
void launch_step0_df64(cudaStream_t st, const Step0Args<df64>& a);

// Graph preparation kernels.
constexpr size_t kCheckFlagsBytes = 64;
rd_status rows_sorted_symmetric(rd_graph* g, cudaStream_t st);
int degree_grid(const rd_graph* g);
rd_status compute_degrees(rd_graph* g, cudaStream_t st, void* flags_dev, double* block_sums_dev, bool check_weights);

}  // namespace rd
