// pairs.cu -- host launcher of the small problems' kernels (k_pairs.cuh).
#include "host_common.h"
#include "k_pairs.cuh"

namespace domagg {

template <int M, class Op, int WT, bool F32>
static void launch_one(Launcher& L, const PairCall& C, unsigned blocks, bool beside) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(PAIR_THREADS);
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = beside ? 1 : 0;  // beside k_pair_stats, which it does not read from
    cudaLaunchKernelEx(&cfg, k_pairs<M, Op, WT, F32>, C);
}

template <int M, bool F32, int ITEMS, int T>
static void launch_stats(Launcher& L, const PairStatCall& C, unsigned jobs, unsigned cluster) {
    constexpr size_t smem = pstat_smem<ITEMS, T>();
    cudaFuncSetAttribute(k_pair_stats<M, F32, ITEMS, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(jobs * cluster);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_pair_stats<M, F32, ITEMS, T>, C);
}

template <int M, bool F32>
static void launch_mf(Launcher& L, PairOp op, const PairCall& C, unsigned blocks, const PairStatCall* st,
                      unsigned st_jobs, u32 st_points, double bytes) {
    const bool beside = M >= 2 && st && st_jobs > 0;
    if constexpr (M >= 2) {
        if (beside) {
            L.start(KIND_SMALL, 0.0);
            if (!st->tab) {  // a single problem: a cluster per coordinate
                const unsigned cl = PSTAT_CLUSTER;
                if (st_points <= 4u * cl * PSTAT_FEW_THREADS) launch_stats<M, F32, 4, PSTAT_FEW_THREADS>(L, *st, st_jobs, cl);
                else launch_stats<M, F32, 3, PSTAT_THREADS>(L, *st, st_jobs, cl);
            } else if (st_points <= 2u * PSTAT_THREADS) {
                launch_stats<M, F32, 2, PSTAT_THREADS>(L, *st, st_jobs, 1);
            } else if (st_points <= 8u * PSTAT_THREADS) {
                launch_stats<M, F32, 8, PSTAT_THREADS>(L, *st, st_jobs, 1);
            } else {
                launch_stats<M, F32, 24, PSTAT_THREADS>(L, *st, st_jobs, 1);
            }
            L.stop();
        }
    }
    L.start(KIND_PAIRS, bytes);
    switch (op) {
        case PAIR_SUM_F32: launch_one<M, OpSumF32, 2, F32>(L, C, blocks, beside); break;
        case PAIR_SUM_I64: launch_one<M, OpSumI64, 1, F32>(L, C, blocks, beside); break;
        case PAIR_MAX_I32: launch_one<M, OpMaxI32, 0, F32>(L, C, blocks, beside); break;
        case PAIR_MAX_F32: launch_one<M, OpMaxF32, 2, F32>(L, C, blocks, beside); break;
        case PAIR_MIN_I32: launch_one<M, OpMinI32, 0, F32>(L, C, blocks, beside); break;
        case PAIR_MIN_F32: launch_one<M, OpMinF32, 2, F32>(L, C, blocks, beside); break;
        case PAIR_COUNT: launch_one<M, OpCount, 3, F32>(L, C, blocks, beside); break;
    }
    L.stop();
}

void pairs_launch(Launcher& L, int m, PairOp op, bool f32, const PairCall& C, unsigned blocks,
                  const PairStatCall* st, unsigned st_jobs, u32 st_points, double bytes) {
#define DOMAGG_PAIRS(MM)                                                      \
    if (f32) launch_mf<MM, true>(L, op, C, blocks, st, st_jobs, st_points, bytes);     \
    else launch_mf<MM, false>(L, op, C, blocks, st, st_jobs, st_points, bytes);        \
    break
    switch (m) {
        case 1: DOMAGG_PAIRS(1);
        case 2: DOMAGG_PAIRS(2);
        case 3: DOMAGG_PAIRS(3);
        default: DOMAGG_PAIRS(4);
    }
#undef DOMAGG_PAIRS
}

u32 bounds_site_pairs(bool clear) {
#ifdef DOMAGG_CHECKED
    u32 hit = 0, site = 0;
    cudaMemcpyFromSymbol(&hit, g_bounds_hit, sizeof(u32));
    cudaMemcpyFromSymbol(&site, g_bounds_site, sizeof(u32));
    if (clear && hit) {
        const u32 z = 0;
        cudaMemcpyToSymbol(g_bounds_hit, &z, sizeof(u32));
    }
    cudaGetLastError();
    return hit ? (site ? site : 1u) : 0u;
#else
    (void)clear;
    return 0u;
#endif
}

}  // namespace domagg
