// cr_tail.cu -- the coarse levels of a short FP64 system in one launch per sweep
// direction: a cluster of CTAs runs level after level, with the cluster's
// barrier where the per-level kernels have a launch.
//
// Why.  A coarse level keeps a few SMs busy for 5 to 10 us (a chain of pivots
// and dependent products), and a launch, its wait and the arrival counters of
// the CTA boundaries cost as much again.  A CTA holds as many odd blocks as its
// warps run side by side (tail_blocks), so that the level takes about as long as
// with a block per CTA.  Chunks, formulas and their order are those of the
// level kernels, so results are bit-identical.
//
// The even block on a chunk boundary: after the cluster's barrier the CTA on its
// right subtracts its own part (read through L2, as another SM wrote the
// other), as the fix-up kernels do, and a second barrier ends the level.
#include "cr_launch.h"
#include "cr_core.cuh"

namespace crs {

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The forms of a block size: kSplit by tiles on the tensor cores, else the wide
// FMA forms (few blocks per CTA).
template <int MT, bool kSplit>
__global__ void __launch_bounds__(256) k_factor_tail(const __grid_constant__ TailArgs ta) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    level_begin();
    const int64_t c = blockIdx.x;
    for (int i = 0; i < ta.n; ++i) {
        const LevelArgs &a = ta.lev[i];
        const int64_t nc = crs_num_ctas(a.no, a.nb);
        if (c < nc) {
            if constexpr (kSplit) factor_split<MT, false>(a, c, smem_raw);
            else factor_chunk<MT, double, true>(a, c, smem_raw);
        }
        cluster_sync();
        if (nc > 1) {
            if (c >= 1 && c < nc)
                for (int e = threadIdx.x; e < a.m * (a.m + 1) / 2; e += blockDim.x) factor_fix_entry<double, true>(a, c, e);
            cluster_sync();
        }
    }
}

// Columns blockIdx.y * kc .. of every level: the down sweep to the last level,
// then the up sweep.
template <int MT, bool kSplit>
__global__ void __launch_bounds__(256) k_solve_tail(const __grid_constant__ TailArgs ta) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    level_begin();
    const int64_t c = blockIdx.x;
    const int cc = blockIdx.y;
    for (int i = 0; i < ta.n; ++i) {
        const LevelArgs &a = ta.lev[i];
        const int64_t nc = crs_num_ctas(a.no, a.nb);
        if (c < nc) {
            if constexpr (kSplit) solve_down_split<MT, false>(a, c, cc, smem_raw);
            else solve_down_chunk<MT, double, true>(a, c, cc, smem_raw);
        }
        cluster_sync();
        if (nc > 1) {
            const int kw = min(a.kc, a.k - cc * a.kc);
            if (c >= 1 && c < nc)
                for (int e = threadIdx.x; e < a.m * kw; e += blockDim.x)
                    solve_down_fix_entry<double, true>(a, c, (e / kw) * a.k + cc * a.kc + e % kw);
            cluster_sync();
        }
    }
    for (int i = ta.n - 1; i >= 0; --i) {
        const LevelArgs &a = ta.lev[i];
        if (c < crs_num_ctas(a.no, a.nb)) {
            if constexpr (kSplit) solve_up_split<MT, false>(a, c, cc, smem_raw);
            else solve_up_chunk<MT, double, true>(a, c, cc, smem_raw);
        }
        cluster_sync();
    }
}

// Above m = 32 a level is long enough for its launch not to matter, and the level
// kernels take more threads.
int tail_blocks(int m) { return m <= 4 ? 8 : (m <= 8 ? 4 : (m <= 16 ? 2 : (m <= 32 ? 1 : 0))); }

static cudaError_t launch_tail(void (*kernel)(TailArgs), dim3 grid, size_t smem, const TailArgs &ta, cudaStream_t s) {
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kTailCtas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, ta);
}

#define CRS_TAIL(kernel, mt, split)                                              \
    switch (mt) {                                                                \
        case 4: k = kernel<4, false>; break;                                     \
        case 8: k = split ? kernel<8, true> : kernel<8, false>; break;           \
        case 16: k = split ? kernel<16, true> : kernel<16, false>; break;        \
        case 32: k = kernel<32, true>; break;                                    \
        default: return cudaErrorInvalidValue;                                   \
    }

cudaError_t prepare_tail(int m, int smem_optin) {
    if (tail_blocks(m) == 0) return cudaSuccess;
    const int mt = pick_mt(m);
    const bool split = split_form(m, 8);
    void (*k)(TailArgs) = nullptr;
    CRS_TAIL(k_factor_tail, mt, split)
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
    if (e != cudaSuccess) return e;
    CRS_TAIL(k_solve_tail, mt, split)
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
}

cudaError_t launch_factor_tail(const TailArgs &ta, cudaStream_t s) {
    const int m = ta.lev[0].m, mt = pick_mt(m), nb = ta.lev[0].nb;
    const bool split = split_form(m, 8);
    void (*k)(TailArgs) = nullptr;
    CRS_TAIL(k_factor_tail, mt, split)
    return launch_tail(k, dim3(kTailCtas), split ? nb * factor64_entries(mt) * sizeof(z2) : factor_smem_bytes(mt, nb, 8), ta, s);
}

cudaError_t launch_solve_tail(const TailArgs &ta, cudaStream_t s) {
    const LevelArgs &a = ta.lev[0];
    const int mt = pick_mt(a.m);
    const bool split = split_form(a.m, 8);
    void (*k)(TailArgs) = nullptr;
    CRS_TAIL(k_solve_tail, mt, split)
    const size_t smem = split ? (size_t)a.nb * mt * a.kc * 2 * sizeof(z2) : solve_smem_bytes(mt, a.nb, a.kc, 3, 8);
    return launch_tail(k, dim3(kTailCtas, (unsigned)((a.k + a.kc - 1) / a.kc)), smem, ta, s);
}

}  // namespace crs
