// Entry points to the pieces of cr_split.cuh for the tests that compare them
// with exact integer and rational arithmetic.
#include "cr_launch.h"
#include "cr_split.cuh"

using namespace crs;

// split_value of seven digit sums over ks K-steps, on the host.
extern "C" double split_value_host(int ks, const int *sums) {
    int s[kSplitDigits];
    for (int d = 0; d < kSplitDigits; ++d) s[d] = ks == 1 ? (int)((unsigned)sums[d] + (unsigned)kSplitMagic) : sums[d];
    switch (ks) {
        case 1: return split_value<1>(s);
        case 2: return split_value<2>(s);
        case 4: return split_value<4>(s);
        case 8: return split_value<8>(s);
        default: return split_value<16>(s);
    }
}

// One tile by one warp: out[g][c] of a [8][8 KS] and b [8][8 KS].
template <SplitKind KIND, bool kJoint, int KS>
__global__ void k_tile(const z2 *a, const z2 *b, z2 *out) {
    z2 v[2];
    int e[2];
    split_tile<KIND, kJoint, KS>(KS, [=](int i, int k) { return a[i * 8 * KS + k]; }, [=](int i, int k) { return b[i * 8 * KS + k]; }, {8, 8, kFull},
                                 false, v, e);
    const int g = threadIdx.x >> 2, t = threadIdx.x & 3;
    for (int j = 0; j < 2; ++j) out[8 * g + 2 * t + j] = zmk(split_scaled(v[j].x, e[j]), split_scaled(v[j].y, e[j]));
}

template <SplitKind KIND, bool kJoint>
static int tile_ks(int ks, const z2 *a, const z2 *b, z2 *out) {
    switch (ks) {
        case 1: k_tile<KIND, kJoint, 1><<<1, 32>>>(a, b, out); break;
        case 2: k_tile<KIND, kJoint, 2><<<1, 32>>>(a, b, out); break;
        case 4: k_tile<KIND, kJoint, 4><<<1, 32>>>(a, b, out); break;
        case 8: k_tile<KIND, kJoint, 8><<<1, 32>>>(a, b, out); break;
        default: k_tile<KIND, kJoint, 16><<<1, 32>>>(a, b, out);
    }
    return (int)cudaDeviceSynchronize();
}

// kind: 0 conj(a) b on separate grids, 1 a b and 2 a conj(b) on the joint grid;
// device pointers.
extern "C" int split_tile_device(int kind, int ks, const void *a, const void *b, void *out) {
    const z2 *pa = static_cast<const z2 *>(a), *pb = static_cast<const z2 *>(b);
    z2 *po = static_cast<z2 *>(out);
    if (kind == 0) return tile_ks<kConjA, false>(ks, pa, pb, po);
    if (kind == 1) return tile_ks<kPlain, true>(ks, pa, pb, po);
    return tile_ks<kConjB, true>(ks, pa, pb, po);
}

// r[i] = fast_rcp(d[i]) where it takes d[i], else 0; device pointers.
__global__ void k_rcp(const double *d, double *r, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = fast_rcp_takes(d[i]) ? fast_rcp(d[i]) : 0.0;
}
extern "C" int fast_rcp_device(const void *d, void *r, int n) {
    k_rcp<<<(n + 255) / 256, 256>>>(static_cast<const double *>(d), static_cast<double *>(r), n);
    return (int)cudaDeviceSynchronize();
}

extern "C" double mixed_step_cost_host(int m, int k, int split) { return mixed_step_cost(m, k, split != 0); }
