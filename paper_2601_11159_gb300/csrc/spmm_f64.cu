// FP64 instantiations of the SpMM step (FP64 vectors and sums).
#include "spmm.cuh"

namespace rd {

#define RD_F64_ROWS(X) \
    X(2, 4) \
    X(2, 8) \
    X(2, 16) \
    X(2, 32) \
    X(4, 32) \
    X(1, 1)

#define RD_F64_CONFIGS(X) \
    X(1, 1, 4)            \
    X(1, 1, 8)            \
    X(1, 1, 16)           \
    X(1, 1, 32)           \
    X(2, 4, 8)            \
    X(2, 8, 4)            \
    X(2, 16, 2)           \
    X(2, 4, 1)            \
    X(2, 8, 1)            \
    X(2, 16, 1)           \
    X(2, 32, 1)           \
    X(4, 32, 1)

// async row-stream (kind 3): two 8-byte elements per 16-byte lane slot, slabs of 16 to 64 columns
#define RD_F64_ASYNC(X) \
    X(8)                \
    X(16)               \
    X(32)

bool launch_spmm_f64(const SpmmCfg& c, bool weighted, bool heavy, int grid, cudaStream_t st,
                     const StepArgs<double>& a)
{
    if (c.kind == 3) {
        if (c.vec != 2 || c.nzl != 1) return false;
#define X(G) \
    if (c.gs == G) return launch_async_cfg<double, G>(weighted, heavy, grid, st, a);
        RD_F64_ASYNC(X)
#undef X
        return false;
    }
    if (c.kind == 4 && !heavy) {
        if (c.vec != 2 || c.nzl != 1) return false;
#define X(G) \
    if (c.gs == G) return launch_pipe_cfg<double, G>(weighted, grid, st, a);
        RD_F64_ASYNC(X)
#undef X
        return false;
    }
    if (c.kind == 2 && !heavy) return launch_spmv_tasks<double>(weighted, grid, st, a);
    if (c.kind == 1 && !heavy) {
#define X(V, G) \
    if (c.vec == V && c.gs == G && c.nzl == 1) return launch_rows_cfg<double, V, G>(weighted, grid, st, a);
        RD_F64_ROWS(X)
#undef X
        return false;
    }
    // the heavy-row pre-pass runs the row-group heavy kernel with the same column tile and
    // one warp per chunk (heavy_cfg)
    const int zl = heavy ? heavy_cfg(c).nzl : c.nzl;
#define X(V, G, Z) \
    if (c.vec == V && c.gs == G && zl == Z) return launch_cfg<double, V, G, Z>(weighted, heavy, grid, st, a);
    RD_F64_CONFIGS(X)
#undef X
    return false;
}

int spmm_blocks_per_sm_f64(const SpmmCfg& c, bool weighted, bool heavy)
{
    if (c.kind == 3) {
        if (c.vec != 2 || c.nzl != 1) return 0;
#define X(G) \
    if (c.gs == G) return occupancy_async_cfg<double, G>(weighted, heavy);
        RD_F64_ASYNC(X)
#undef X
        return 0;
    }
    if (c.kind == 4 && !heavy) {
        if (c.vec != 2 || c.nzl != 1) return 0;
#define X(G) \
    if (c.gs == G) return occupancy_pipe_cfg<double, G>(weighted);
        RD_F64_ASYNC(X)
#undef X
        return 0;
    }
    if (c.kind == 2 && !heavy) return occupancy_spmv_tasks<double>(weighted);
    if (c.kind == 1 && !heavy) {
#define X(V, G) \
    if (c.vec == V && c.gs == G && c.nzl == 1) return occupancy_rows_cfg<double, V, G>(weighted);
        RD_F64_ROWS(X)
#undef X
        return 0;
    }
    const int zl = heavy ? heavy_cfg(c).nzl : c.nzl;
#define X(V, G, Z) \
    if (c.vec == V && c.gs == G && zl == Z) return occupancy_cfg<double, V, G, Z>(weighted, heavy);
    RD_F64_CONFIGS(X)
#undef X
    return 0;
}

std::vector<SpmmCfg> spmm_configs_f64()
{
    std::vector<SpmmCfg> v;
#define X(V, G, Z) v.push_back(SpmmCfg{V, G, Z, 0});
    RD_F64_CONFIGS(X)
#undef X
    v.push_back(SpmmCfg{1, 1, 1, 2});
#define X(V, G) v.push_back(SpmmCfg{V, G, 1, 1});
    RD_F64_ROWS(X)
#undef X
#define X(G) v.push_back(SpmmCfg{2, G, 1, 3}), v.push_back(SpmmCfg{2, G, 1, 4});
    RD_F64_ASYNC(X)
#undef X
    return v;
}

}  // namespace rd
