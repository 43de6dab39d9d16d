// cr_batch.cuh -- the persistent kernel of the batched form (see cr_batched.cu for
// its design), instantiated per thread count in translation units of their
// own (cr_batched.cu, cr_batched512.cu), which compile side by side.
#pragma once
#include <cstdint>

#include "cr_launch.h"

namespace crs {

struct SysDesc {
    int64_t N, offA, offB, offY;  // element offsets into the packed A, B, y / x
    int32_t m, k, mt, pad;
};

struct BatchTiles {
    int nbf[5], nbs[5], kc[5];
};

struct BatchArgs {
    const SysDesc *sys;
    const int32_t *order;
    int32_t nsys;
    int32_t *counter;
    const z2 *A, *B, *y;
    z2 *x;
    char *slots;
    int64_t slot_bytes;
    unsigned long long *status;  // [nsys]
    BatchTiles tiles;
    unsigned long long *dbg;     // bounds-checked builds: first out-of-range access
};

__host__ __device__ inline int64_t al16(int64_t b) { return (b + 15) & ~(int64_t)15; }

__host__ __device__ inline int num_levels(int64_t N) {
    int n = 1;
    while (N > 1) { N /= 2; ++n; }
    return n;
}

// Bytes of level l's stored factor region: L [no][m][m], Z [no][m][2m],
// r [no][m][k] (complex) and 1/diag(L) [no][m] (double).
__host__ __device__ inline int64_t level_region(int64_t no, int m, int k) {
    return no * (int64_t)(3 * m * m + m * k) * 16 + al16(no * (int64_t)m * 8);
}

// Slot layout of a system: the levels' factor regions, then the ping-pong
// buffers: system buffers S[p] (A then B, capacity cap[p] blocks) and vector
// buffers Y[p] (capacity cap[p] blocks of m x k), p = parity of the level
// they hold (levels 1, 3, ... in p = 1 with cap N_1; 2, 4, ... in p = 0 with cap N_2).
struct SlotLevel {
    int64_t Nl, no, ne, off;           // level sizes and the offset of its factor region
    int64_t sysbuf[2], vecbuf[2], cap[2];
};

__host__ __device__ inline int64_t slot_layout(int64_t N, int m, int k, int want, SlotLevel *out) {
    int64_t off = 0, Nl = N, N1 = N / 2, N2 = N / 4;
    const int nlev = num_levels(N);
    for (int l = 0; l < nlev; ++l) {
        const int64_t no = (Nl + 1) / 2;
        if (out && l == want) { out->Nl = Nl; out->no = no; out->ne = Nl / 2; out->off = off; }
        off += level_region(no, m, k);
        Nl /= 2;
    }
    int64_t cap[2] = {N2, N1};
    int64_t sb[2], vb[2];
    for (int p = 0; p < 2; ++p) {
        sb[p] = off;
        off += cap[p] * 2 * (int64_t)m * m * 16;
        vb[p] = off;
        off += cap[p] * (int64_t)m * k * 16;
    }
    if (out)
        for (int p = 0; p < 2; ++p) { out->sysbuf[p] = sb[p]; out->vecbuf[p] = vb[p]; out->cap[p] = cap[p]; }
    return (off + 255) & ~(int64_t)255;
}

// Level l's arguments for system d in slot `slot` (same for every thread).
__device__ inline void make_level_args(LevelArgs &a, const BatchArgs &ba, const SysDesc &d, int32_t sid, char *slot,
                                       int l) {
    const int m = d.m, k = d.k, mm = m * m, mk = m * k;
    SlotLevel sl;
    slot_layout(d.N, m, k, l, &sl);
    a = LevelArgs{};
    a.Nl = sl.Nl; a.no = sl.no; a.ne = sl.ne; a.m = m; a.k = k; a.level = l; a.inline_fix = 1;
    const int p = l & 1, q = (l + 1) & 1;
    char *reg = slot + sl.off;
    a.L = reinterpret_cast<z2 *>(reg);
    a.Z = a.L + sl.no * mm;
    a.r = a.Z + sl.no * 2 * mm;
    a.inv = reinterpret_cast<double *>(a.r + sl.no * mk);
    z2 *Sp = reinterpret_cast<z2 *>(slot + sl.sysbuf[p]), *Sq = reinterpret_cast<z2 *>(slot + sl.sysbuf[q]);
    z2 *Yp = reinterpret_cast<z2 *>(slot + sl.vecbuf[p]), *Yq = reinterpret_cast<z2 *>(slot + sl.vecbuf[q]);
    a.A = l == 0 ? ba.A + d.offA : Sp;
    a.B = l == 0 ? ba.B + d.offB : Sp + sl.cap[p] * mm;
    a.An = Sq;
    a.Bn = Sq + sl.cap[q] * mm;
    a.y = l == 0 ? ba.y + d.offY : Yp;
    a.yn = Yq;
    a.x = l == 0 ? ba.x + d.offY : Yp;
    a.xn = Yq;
    a.status = ba.status + sid;
    a.dbg = ba.dbg;
}

// One chunk in the form of its block size (the form the level kernels take); a
// function each, which keeps the kernel quick to compile.
template <int MT>
__device__ __noinline__ void factor_of(const LevelArgs &a, int64_t c, unsigned char *smem) {
    if constexpr (Forms<MT, double>::fma) {
        if (!split_form(a.m, 8)) return factor_chunk<MT, double>(a, c, smem);
    }
    if constexpr (Forms<MT, double>::split) factor_chunk_split<MT>(a, c, smem);
}
template <int MT>
__device__ __noinline__ void solve_down_of(const LevelArgs &a, int64_t c, int cc, unsigned char *smem) {
    if constexpr (Forms<MT, double>::fma) {
        if (!split_form(a.m, 8)) return solve_down_chunk<MT, double>(a, c, cc, smem);
    }
    if constexpr (Forms<MT, double>::split) solve_down_chunk_split<MT>(a, c, cc, smem);
}
template <int MT>
__device__ __noinline__ void solve_up_of(const LevelArgs &a, int64_t c, int cc, unsigned char *smem) {
    if constexpr (Forms<MT, double>::fma) {
        if (!split_form(a.m, 8)) return solve_up_chunk<MT, double>(a, c, cc, smem);
    }
    if constexpr (Forms<MT, double>::split) solve_up_chunk_split<MT>(a, c, cc, smem);
}

// The whole classic cyclic reduction of one system, run by one CTA.  The
// level arguments live in shared memory (sa) so that they do not hold
// registers across the chunk loops.
template <int MT>
__device__ __noinline__ void run_system(const BatchArgs &ba, const SysDesc &d, int32_t sid, char *slot,
                                        unsigned char *smem, LevelArgs &sa) {
    const int k = d.k;
    const int nlev = num_levels(d.N);
    const int ti = MT == 4 ? 0 : MT == 8 ? 1 : MT == 16 ? 2 : MT == 32 ? 3 : 4;
    const int nbf = ba.tiles.nbf[ti], nbs = ba.tiles.nbs[ti], kcm = ba.tiles.kc[ti];
    // down: factor level l, then reduce its right-hand side
    for (int l = 0; l < nlev; ++l) {
        if (threadIdx.x == 0) {
            make_level_args(sa, ba, d, sid, slot, l);
            sa.nb = (int)min((int64_t)nbf, sa.no);
        }
        __syncthreads();
        for (int64_t c = 0, nc = crs_num_ctas(sa.no, sa.nb); c < nc; ++c) {
            factor_of<MT>(sa, c, smem);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            sa.nb = (int)min((int64_t)nbs, sa.no);
            sa.kc = min(kcm, k);
        }
        __syncthreads();
        const int ncc = (k + sa.kc - 1) / sa.kc;
        for (int64_t c = 0, nc = crs_num_ctas(sa.no, sa.nb); c < nc; ++c)
            for (int cc = 0; cc < ncc; ++cc) {
                solve_down_of<MT>(sa, c, cc, smem);
                __syncthreads();
            }
    }
    // up: coarsest level first
    for (int l = nlev - 1; l >= 0; --l) {
        if (threadIdx.x == 0) {
            make_level_args(sa, ba, d, sid, slot, l);
            sa.nb = (int)min((int64_t)nbs, sa.no);
            sa.kc = min(kcm, k);
        }
        __syncthreads();
        const int ncc = (k + sa.kc - 1) / sa.kc;
        for (int64_t c = 0, nc = crs_num_ctas(sa.no, sa.nb); c < nc; ++c)
            for (int cc = 0; cc < ncc; ++cc) {
                solve_up_of<MT>(sa, c, cc, smem);
                __syncthreads();
            }
    }
}

// TH threads: 256 with two CTAs per SM, or 512 with one where the batch lasts as
// long as its largest system (see crsolve_batch_create).
template <int TH>
__global__ void __launch_bounds__(TH, 512 / TH) k_batch(BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int32_t s_next;
    __shared__ LevelArgs s_args;
    char *slot = ba.slots + (int64_t)blockIdx.x * ba.slot_bytes;
    for (;;) {
        if (threadIdx.x == 0) s_next = atomicAdd(ba.counter, 1);
        __syncthreads();
        const int32_t i = s_next;
        __syncthreads();
        if (i >= ba.nsys) return;
        const int32_t sid = ba.order[i];
        const SysDesc d = ba.sys[sid];
        switch (d.mt) {
            case 4: run_system<4>(ba, d, sid, slot, smem_raw, s_args); break;
            case 8: run_system<8>(ba, d, sid, slot, smem_raw, s_args); break;
            case 16: run_system<16>(ba, d, sid, slot, smem_raw, s_args); break;
            case 32: run_system<32>(ba, d, sid, slot, smem_raw, s_args); break;
            default: run_system<64>(ba, d, sid, slot, smem_raw, s_args); break;
        }
        __syncthreads();
    }
}

// k_batch<512>, from cr_batched512.cu
void (*batch_kernel512())(BatchArgs);

}  // namespace crs
