// cr_core64.cuh -- the FP64 level steps of the blocks of split_form,
// run by one CTA on one chunk of a level, with every product on the tensor
// cores (cr_split.cuh).
//
// The factor keeps X = L^{-1} of every odd block in place of L, so that all
// triangular solves are products: Z = X [B_l | B_r^H], r = X y, x = X^H w.  With
// FP64 FMAs the solves, Z^H Z and the sweeps' products were 95% of the FP64
// instructions of a step, on a pipe of 2 FMA per clock per SM; here FP64
// instructions are left in the Cholesky factorisation with its inverse and in
// one rounding per result.
//
// An inverse of L is as good as substitution where it is multiplied exactly:
// the rounding errors of X are those of the substitution on the unit vectors
// (L X = I + E, |E| <= m u |L| |X|), and a product with X adds one rounding of
// its result where a substitution adds one per term.
//
// Tiles are 8 x 8; blocks whose m is no multiple of 8 are padded with zeros in
// registers.  Every result depends on the block's data alone, not on the chunk
// size, the threads or the right-hand-side chunk, so the level kernels, the
// batched kernel and the allocation-free path agree bit for bit.
#pragma once
#include "cr_split.cuh"

namespace crs {

// Which blocks take these forms: those that fill their tiles well enough.  A
// block of m <= 4 would fill a quarter of a fragment; at m = 5 the padding to
// 8 x 8 costs more than the FMAs (factor and solve at N = 100003, k = 3: 815 + 1076
// against 595 + 800 us), and so does that of m = 9 and 10 to 16 x 16 (factor at
// m = 10, N = 48000: about 1900 against 1733 us; at m = 11, N = 36062: 1574 against
// 1652, solve with k = 4 1009 against 1436, before small results took FMAs; with
// them, and on banded systems, the factor is 1.45 times the FMA form's and the
// solve 0.77 of it).
__host__ __device__ constexpr bool split_form(int m, size_t rsize) { return rsize == 8 && (m >= 11 || m == 7 || m == 8); }
// The classes that have blocks of either kind.
template <int MT, class R> struct Forms {
    static constexpr bool split = sizeof(R) == 8 && MT >= 8;
    static constexpr bool fma = sizeof(R) == 4 || MT <= 16;
};

// Shared memory of a chunk, in complex entries per odd block.  Odd strides
// keep the accesses of consecutive blocks and rows in different banks.
template <int MT> struct Split64 {
    static constexpr int LDZ = 2 * MT + 1;          // row of Z
    static constexpr int SL = Tri<MT>::n | 1;       // packed triangle
    // scratch: two columns of an 8 x 8 diagonal block (chol_inv8) or, not at
    // the same time, one row of blocks U (inverse_chunk)
    static constexpr int SC = MT > 8 ? 8 * MT + 1 : 17;
};
__host__ __device__ constexpr size_t factor64_entries(int mt) {
    return (size_t)(((mt * (mt + 1) / 2) | 1) + mt * (2 * mt + 1) + (mt > 8 ? 8 * mt + 1 : 17));
}

// Row of entry f of a packed 8 x 8 lower triangle.
__device__ __forceinline__ int tri8_row(int f) {
    constexpr unsigned kStarts = 1u << 1 | 1u << 3 | 1u << 6 | 1u << 10 | 1u << 15 | 1u << 21 | 1u << 28;
    return f >= 28 ? 7 : __popc(kStarts & ((2u << f) - 1u));
}

// The breakdown test of pivot d of block b, and 1 / d (fast_rcp).  Pivots in
// fast_rcp's range are told by their high word, as a comparison in FP64 would
// take as long as a step of the reciprocal.  0 for the others, whose
// reciprocal need not be a normal number: pivot_scale divides by them.
__device__ __forceinline__ double pivot_rcp(const LevelArgs &a, int64_t block, double d) {
    if (!fast_rcp_takes(d)) {
        if (!(d > 0.0)) report_fail(a.status, a.level, report_index(a, 2 * block));
        return 0.0;
    }
    return fast_rcp(d);
}

// v / d for pivot d with reciprocal s (pivot_rcp).
__device__ __forceinline__ z2 pivot_scale(z2 v, double d, double s) {
    return __double2hiint(s) != 0 ? zscale(v, s) : zmk(v.x / d, v.y / d);
}

// X = L^{-1} of the diagonal blocks o .. o + w - 1 (w <= 8) of A_b = L L^H (packed
// lower in sL, in place) for the blocks b < nbh of a chunk, with the breakdown
// test of every pivot.  Right-looking elimination A = M D M^H: with pivot d_c
// final, every later row r takes t_r = A_rc / d_c times (the conjugate of) column
// c off its trailing entries and t_r times row c of M^{-1} off its entries of
// M^{-1}; column c of A is not needed after that, so -t_r, the new entry of M^{-1},
// takes its place (a Gauss-Jordan step).  At the end X = D^{-1/2} M^{-1}: the
// square roots are off the chain of pivots, which on GB300 costs 64 clocks per
// FP64 instruction of a warp whatever its lanes (measured).  Two forms with the
// same operations on every entry, so the same numbers:
//  - up to 4 blocks (coarse levels; also what a CTA of m > 32 holds): a warp per
//    block, two entries per lane, pivots and columns by shuffles;
//  - else: one entry per thread, consecutive threads on consecutive blocks, two
//    barriers per column (t and the column copied; the updates, and meanwhile
//    in a warp of its own the next pivot), which takes a tenth of the FP64
//    instructions.
// Ends with __syncthreads().
template <int MT>
__device__ __forceinline__ void chol_inv8(const LevelArgs &a, int64_t t0, z2 *sL, z2 *sC, int nbh, int o, int w) {
    constexpr int SL = Split64<MT>::SL, SC = Split64<MT>::SC;
    const int NT = blockDim.x, tid = threadIdx.x;
    auto at = [&](int r, int c) { return tri(o + r, o + c); };
    if (nbh <= 4) {
        constexpr unsigned kAll = 0xffffffffu;
        const int lane = tid & 31, r = lane >> 2, q = lane & 3, nw = NT >> 5;
        for (int b = tid >> 5; b < nbh; b += nw) {
            z2 *Lb = sL + b * SL;
            z2 e[2];
            double dr = 1.0;
#pragma unroll
            for (int h = 0; h < 2; ++h) e[h] = (r < w && 2 * q + h <= r) ? Lb[at(r, 2 * q + h)] : zmk(0.0, 0.0);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c >= w) break;
                const z2 col = e[c & 1];    // entry (r, c) in lane 4 r + c / 2
                const double d = __shfl_sync(kAll, col.x, 4 * c + (c >> 1));
                if (r == c) dr = d;
                const double s = pivot_rcp(a, t0 + b, d);
                if (c + 1 >= w) break;
                z2 t, wv[2];
                t.x = __shfl_sync(kAll, col.x, 4 * r + (c >> 1));
                t.y = __shfl_sync(kAll, col.y, 4 * r + (c >> 1));
                t = pivot_scale(t, d, s);
                const z2 cc = zconj(col);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // conj(A_jc) from row j > c, the entry of M^{-1} from row c
                    const int j = 2 * q + h, src = j > c ? 4 * j + (c >> 1) : 4 * c + q;
                    const z2 v = r == c ? e[h] : cc;
                    wv[h].x = __shfl_sync(kAll, v.x, src);
                    wv[h].y = __shfl_sync(kAll, v.y, src);
                    if (j == c) wv[h] = zmk(1.0, 0.0);
                }
                if (r > c) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (2 * q + h == c) e[h] = zmk(0.0, 0.0);
                        zmsub(e[h], t, wv[h]);
                    }
                }
            }
            const double iv = rsq(dr);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = 2 * q + h;
                if (r < w && j <= r) Lb[at(r, j)] = j == r ? zmk(iv, 0.0) : zscale(e[h], iv);
            }
        }
        __syncthreads();
        return;
    }
    const int npiv = NT >= 64 ? 32 : 0;       // threads kept for the pivots
    // a pivot is kept with its reciprocal
    auto pivot = [&](int b, int c, double d) { sL[b * SL + at(c, c)] = zmk(d, pivot_rcp(a, t0 + b, d)); };
    const int pstep = npiv ? npiv : NT;
    const bool piv = tid < pstep;
    if (piv)
        for (int b = tid; b < nbh; b += pstep) pivot(b, 0, sL[b * SL + at(0, 0)].x);
    const int q1 = min(nbh, NT), b1 = tid % q1, f1 = tid / q1, s1 = NT / q1;
    const int nu = NT - npiv, q2 = min(nbh, nu), ut = tid - npiv, b2 = ut % q2, f2 = ut / q2, s2 = nu / q2;
    const int ntri = w * (w + 1) / 2;
    for (int c = 0; c + 1 < w; ++c) {
        __syncthreads();
        if (f1 < s1 && f1 < w)
            for (int b = b1; b < nbh; b += q1) {
                const z2 *Lb = sL + b * SL;
                z2 *Cb = sC + b * SC;
                const z2 p = Lb[at(c, c)];
                for (int i = f1; i < w; i += s1) {
                    if (i <= c) continue;
                    const z2 v = Lb[at(i, c)];
                    Cb[i] = pivot_scale(v, p.x, p.y);
                    Cb[8 + i] = v;
                }
            }
        __syncthreads();
        if (piv)
            for (int b = tid; b < nbh; b += pstep) {
                const z2 t = sC[b * SC + c + 1], v = sC[b * SC + 8 + c + 1];
                double d = sL[b * SL + at(c + 1, c + 1)].x;
                d = fma(-t.x, v.x, d);
                d = fma(-t.y, v.y, d);
                pivot(b, c + 1, d);
            }
        if (ut >= 0 && f2 < s2)
            for (int b = b2; b < nbh; b += q2) {
                z2 *Lb = sL + b * SL;
                const z2 *Cb = sC + b * SC;
                for (int f = tri(c + 1, 0) + f2; f < ntri; f += s2) {
                    const int r = tri8_row(f), j = f - tri(r, 0);
                    if (j == c + 1 && r == c + 1) continue;             // the next pivot
                    const z2 t = Cb[r];
                    z2 y = j > c ? zconj(Cb[8 + j]) : Lb[at(c, j)], u = Lb[at(r, j)];
                    if (j == c) {
                        y = zmk(1.0, 0.0);
                        u = zmk(0.0, 0.0);
                    }
                    zmsub(u, t, y);
                    Lb[at(r, j)] = u;
                }
            }
    }
    __syncthreads();
    if (f1 < s1 && f1 < w)
        for (int b = b1; b < nbh; b += q1)
            for (int r = f1; r < w; r += s1) sC[b * SC + r].x = rsq(sL[b * SL + at(r, r)].x);
    __syncthreads();
    if (f1 < s1)
        for (int b = b1; b < nbh; b += q1)
            for (int f = f1; f < ntri; f += s1) {
                const int r = tri8_row(f), j = f - tri(r, 0);
                const double iv = sC[b * SC + r].x;
                z2 *u = sL + b * SL + at(r, j);
                *u = r == j ? zmk(iv, 0.0) : zscale(*u, iv);
            }
    __syncthreads();
}

// X_b = L_b^{-1} of A_b = L_b L_b^H (packed lower in sL, in place) for the blocks
// of a chunk, by 8 x 8 blocks: left-looking, one warp per block of
//   T_IJ = A_IJ - sum_{K<J} L_IK L_JK^H,  X_JJ from T_JJ (chol_inv8),
//   L_IJ = T_IJ X_JJ^H,  U_JK = sum_{K<=M<J} L_JM X_MK,  X_JK = -X_JJ U_JK,
// so that every block is rounded once per formula.  X_JK takes the place of
// L_JK one step after U_JK has read row J of L.  Ends with __syncthreads().
template <int MT, bool FULL>
__device__ __forceinline__ void inverse_chunk(const LevelArgs &a, int64_t t0, z2 *sL, z2 *sC, int nbh) {
    const int m = FULL ? MT : a.m;
    if constexpr (MT == 8) {
        chol_inv8<MT>(a, t0, sL, sC, nbh, 0, m);
        return;
    } else {
        constexpr int SL = Split64<MT>::SL, SU = Split64<MT>::SC, KS = MT / 8;
        z2 *sU = sC;
        const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, tq = lane & 3, warp = tid >> 5, nw = blockDim.x >> 5;
        const int g8 = FULL ? KS : (m + 7) >> 3;
        for (int J = 0; J <= g8; ++J) {
            // T_IJ for I >= J, and row J - 1 of X (J - 1 blocks)
            const int nT = J > 0 ? g8 - J : 0, nX = J > 1 ? J - 1 : 0, n1 = nT + nX;
            for (int e = warp; e < nbh * n1; e += nw) {
                const int b = e / n1, f = e - b * n1;
                z2 *Lb = sL + b * SL;
                z2 v[2];
                int ex[2];
                if (f < nT) {
                    const int I = J + f;
                    auto row = [=](int R) {
                        return [=](int i, int k) { return (FULL || 8 * R + i < m) ? Lb[tri(8 * R + i, k)] : zmk(0.0, 0.0); };
                    };
                    split_tile<kConjB, false, KS>(J, row(I), row(J), {m - 8 * I, m - 8 * J, I == J ? kGram : kFull}, I == J, v, ex);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int r = 8 * I + g, c = 8 * J + 2 * tq + j;
                        if ((!FULL && r >= m) || c > r) continue;
                        z2 &u = Lb[tri(r, c)];
                        const double sc = -split_scale(ex[j]);
                        u.x = fma(v[j].x, sc, u.x);
                        u.y = r == c ? 0.0 : fma(v[j].y, sc, u.y);
                    }
                } else {
                    const int I = J - 1, K = f - nT;
                    const z2 *Ub = sU + b * SU + 8 * K;
                    auto x = [=](int i, int k) { return (k <= i && (FULL || 8 * I + i < m)) ? Lb[tri(8 * I + i, 8 * I + k)] : zmk(0.0, 0.0); };
                    split_tile<kPlain, true, 1>(1, [=](int i, int k) { return (FULL || 8 * I + k < m) ? Ub[k * MT + i] : zmk(0.0, 0.0); }, x, {8, m - 8 * I, kFull}, false, v, ex);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int r = 8 * I + 2 * tq + j;
                        if (FULL || r < m)
                            Lb[tri(r, 8 * K + g)] = zmk(dneg_bits(split_scaled(v[j].x, ex[j])), dneg_bits(split_scaled(v[j].y, ex[j])));
                    }
                }
            }
            if (J == g8) break;
            __syncthreads();
            chol_inv8<MT>(a, t0, sL, sC, nbh, 8 * J, min(8, m - 8 * J));
            // L_IJ for I > J, and U_JK for K < J
            const int nL = g8 - 1 - J, n2 = nL + J;
            for (int e = warp; e < nbh * n2; e += nw) {
                const int b = e / n2, f = e - b * n2;
                z2 *Lb = sL + b * SL;
                z2 v[2];
                int ex[2];
                if (f < nL) {
                    const int I = J + 1 + f;
                    // block column J is complete (8 wide) as there is a row below it
                    split_tile<kConjB, true, 1>(1, [=](int i, int k) { return (FULL || 8 * I + i < m) ? Lb[tri(8 * I + i, 8 * J + k)] : zmk(0.0, 0.0); },
                                                [=](int i, int k) { return k <= i ? Lb[tri(8 * J + i, 8 * J + k)] : zmk(0.0, 0.0); }, {m - 8 * I, 8, kFull}, false, v, ex);
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (FULL || 8 * I + g < m)
                            Lb[tri(8 * I + g, 8 * J + 2 * tq + j)] = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
                } else {
                    const int K = f - nL;
                    split_tile<kPlain, false, KS>(
                        J - K,
                        [=](int i, int k) {     // column i of X
                            const int r = 8 * K + k, c = 8 * K + i;
                            return c <= r ? Lb[tri(r, c)] : zmk(0.0, 0.0);
                        },
                        [=](int i, int k) { return (FULL || 8 * J + i < m) ? Lb[tri(8 * J + i, 8 * K + k)] : zmk(0.0, 0.0); }, {8, m - 8 * J, kFull}, false, v, ex);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (FULL || 8 * J + 2 * tq + j < m)
                            sU[b * SU + (2 * tq + j) * MT + 8 * K + g] = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
                }
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

// One chunk of nb odd blocks of a factor level (see factor_chunk).
template <int MT, bool FULL>
__device__ __forceinline__ void factor_split(const LevelArgs &a, int64_t chunk, unsigned char *smem_raw) {
    [[maybe_unused]] const LevelArgs *const ap = &a;    // for bounds-checked loads in closures
    constexpr int LDZ = Split64<MT>::LDZ, SL = Split64<MT>::SL, KS = MT / 8;
    constexpr bool kOn = MT >= 32;
    const int m = FULL ? MT : a.m, nb = a.nb, NT = blockDim.x, tid = threadIdx.x;
    const int mm = m * m, m2 = 2 * m;
    const int64_t t0 = chunk * nb;
    const int nbh = (int)min((int64_t)nb, a.no - t0);
    z2 *sL = reinterpret_cast<z2 *>(smem_raw);              // [nb][SL] A_2t, then X, then P^H P
    z2 *sZ = sL + (size_t)nb * SL;                            // [nb][MT][LDZ] [B_l | B_r^H], then Z = [P | Q]
    z2 *sC = sZ + (size_t)nb * MT * LDZ;                      // [nb][SC]
    const z2 zero = zmk(0.0, 0.0);

    for (int e = tid; e < nbh * mm; e += NT) {
        const int b = e / mm, rem = e - b * mm, r = rem / m, c = rem - r * m;
        const int64_t pos = 2 * (t0 + b);
        if (r >= c) sL[b * SL + tri(r, c)] = CRS_IN(a, kDbgA, pos * mm + rem) ? a.A[pos * mm + rem] : zero;
        sZ[(b * MT + r) * LDZ + c] = (pos >= 1 && CRS_IN(a, kDbgB, (pos - 1) * mm + rem)) ? a.B[(pos - 1) * mm + rem] : zero;
        sZ[(b * MT + c) * LDZ + m + r] =
            (pos + 1 < a.Nl && CRS_IN(a, kDbgB, pos * mm + rem)) ? zconj(a.B[pos * mm + rem]) : zero;
    }
    __syncthreads();
    inverse_chunk<MT, FULL>(a, t0, sL, sC, nbh);

    const int lane = tid & 31, g = lane >> 2, tq = lane & 3, warp = tid >> 5, nw = NT >> 5;
    const int g8 = (FULL || KS == 1) ? KS : (m + 7) >> 3, ngrp = 2 * g8;
    z2 *sW = sL;    // P^H P
    const z2 zero_on = split_zero_on();

    // Z = X [B_l | B_r^H] of 8 columns of a block in place, by one warp, the rows
    // from the bottom up.  Column groups 0 .. g8-1 are P, the others Q.
    auto z_task = [&](int b, int cg) {
        const int64_t t = t0 + b;
        const bool inP = cg < g8;
        const int c0 = 8 * (inP ? cg : cg - g8), nc = m - c0, col = (inP ? c0 : m + c0) + g;
        z2 *Zb = sZ + b * MT * LDZ;
        const z2 *Xb = sL + b * SL;
        if (inP ? t >= 1 : 2 * t + 1 < a.Nl) {
            for (int R = g8 - 1; R >= 0; --R) {
                z2 v[2];
                int ex[2];
                const z2 *Zc = Zb + col - g, *XL = a.L;
                split_tile<kPlain, true, KS>(
                    R + 1, [=](int i, int k) { return (FULL || (i < nc && k < m)) ? Zc[k * LDZ + i] : zmk(0.0, 0.0); },
                    [=](int i, int k) {
                        if (!((FULL || 8 * R + i < m) && k <= 8 * R + i)) return zmk(0.0, 0.0);
                        if constexpr (!kOn) return Xb[tri(8 * R + i, k)];
                        const int64_t o = t * mm + (8 * R + i) * m + k;     // (sL has X on its grid)
                        return CRS_IN(*ap, kDbgL, o) ? XL[o] : zmk(0.0, 0.0);
                    },
                    {nc, m - 8 * R, kFull}, false, v, ex);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int r = 8 * R + 2 * tq + j;
                    if (FULL || (g < nc && r < m))
                        Zb[r * LDZ + col] = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
                }
                __syncwarp();
            }
        }
        // (a zero coupling leaves its half of Z zero)
        if (FULL || g < nc)
            for (int r = tq; r < m; r += 4) {
                const int64_t o = t * 2 * (int64_t)mm + r * m2 + col;
                if (CRS_IN(a, kDbgZ, o)) a.Z[o] = Zb[r * LDZ + col];
            }
    };

    // Entry (p, q), q <= p, of P^H P of block b: kept in sW for the left even block,
    // or for the chunk's first block given to the previous chunk.
    auto put_pp = [&](int b, int p, int q, z2 w) {
        const int64_t t = t0 + b;
        if (b > 0) {
            sW[b * SL + tri(p, q)] = w;
        } else if (a.inline_fix) {
            // the previous chunk (same CTA, earlier) left V = A - Q^H Q
            const int64_t o = (t - 1) * mm;
            if (CRS_IN(a, kDbgAn, o + p * m + q) && CRS_IN(a, kDbgAn, o + q * m + p)) {
                z2 u = zsub(a.An[o + p * m + q], w);
                if (p == q) u.y = 0.0;
                a.An[o + p * m + q] = u;
                if (p != q) a.An[o + q * m + p] = zconj(u);
            }
        } else if (CRS_IN(a, kDbgWbd, chunk * mm + p * m + q)) {
            a.Wbd[chunk * mm + p * m + q] = w;
        }
    };
    // Entry (p, q) of Q^H P = -F, the next level's B.
    auto put_qp = [&](int b, int p, int q, z2 w) {
        const int64_t o = (t0 + b - 1) * mm + p * m + q;
        if (CRS_IN(a, kDbgBn, o)) a.Bn[o] = zneg(w);
    };
    // A - Q^H Q at entry (p, q), q <= p, of block b's right even block (A loaded
    // ahead of the product)
    auto load_a = [&](int b, int p, int q) {
        const int64_t oa = (2 * (t0 + b) + 1) * mm + p * m + q;
        return (q <= p && (FULL || p < m) && 2 * (t0 + b) + 1 < a.Nl && CRS_IN(a, kDbgA, oa)) ? a.A[oa] : zero;
    };
    auto sub_qq = [&](z2 u, int p, int q, z2 v, int ex) {
        const double sc = -split_scale(ex);
        u.x = fma(v.x, sc, u.x);
        u.y = p == q ? 0.0 : fma(v.y, sc, u.y);
        return u;
    };
    // ... complete unless the right neighbour is in the next chunk
    auto put_v = [&](int b, int p, int q, z2 u) {
        const int64_t o = (t0 + b) * mm;
        if (b + 1 < nbh) u = zsub(u, sW[(b + 1) * SL + tri(p, q)]);
        if (CRS_IN(a, kDbgAn, o + p * m + q)) a.An[o + p * m + q] = u;
        if (p != q && CRS_IN(a, kDbgAn, o + q * m + p)) a.An[o + q * m + p] = zconj(u);
    };

    // Z^H Z by tiles (row group I >= column group J): pass 0 has P^H P and Q^H P,
    // pass 1 Q^H Q.
    const int ntri = g8 * (g8 + 1) / 2;
    //
    // kOn: the entries of X, B and Z are put on their grids once (see the end), with
    // the exponents of the block's columns in sE: those of X at 0, its rows at
    // MT, Z's at 2 MT (0: out of the split's range; the tile then takes Z as
    // stored), and at 4 MT and 5 MT whether X's and Z's columns have imaginary
    // parts.  Small results (split_needs) read the stored entries.  Pays from m > 16 on, where a tile's operands are read by many
    // tiles (level 0 of N = 4096, m = 64: 3335 -> 2884 us, m = 32: 448 -> 417;
    // N = 65536, m = 16: 1069 -> 1125).
    int *const sE = reinterpret_cast<int *>(sC);
    constexpr int SE = 4 * Split64<MT>::SC;    // ints per block
    auto h_task = [&](int b, int pass, int f) {
        const int64_t t = t0 + b;
        int I, J;
        const bool pJ = pass == 0, pI = pass == 0 && f < ntri;
        if (pI || !pJ) {
            I = tri_row(f);
            J = f - I * (I + 1) / 2;
        } else {
            I = (f - ntri) / g8;
            J = f - ntri - I * g8;
        }
        if ((pJ && t < 1) || (!pI && 2 * t + 1 >= a.Nl)) return;
        const z2 *Zb = sZ + b * MT * LDZ;
        const z2 *zi = Zb + 8 * I + (pI ? 0 : m), *zj = Zb + 8 * J + (pJ ? 0 : m);
        const int ni = m - 8 * I, nj = m - 8 * J;
        z2 v[2], u[2];
        int ex[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) u[j] = pJ ? zero : load_a(b, 8 * I + g, 8 * J + 2 * tq + j);
        if constexpr (!kOn) {
            split_tile<kConjA, false, KS>(
                g8, [=](int i, int k) { return (FULL || (i < ni && k < m)) ? zi[k * LDZ + i] : zmk(0.0, 0.0); },
                [=](int i, int k) { return (FULL || (i < nj && k < m)) ? zj[k * LDZ + i] : zmk(0.0, 0.0); }, {ni, nj, zi == zj ? kGram : kFull}, zi == zj, v, ex);
        } else {
            const int *ze = sE + b * SE + 2 * MT;
            const int ci = 8 * I + (pI ? 0 : m), cj = 8 * J + (pJ ? 0 : m);
            const int ei = (FULL || g < ni) ? ze[ci + g] : 1023, ej = (FULL || g < nj) ? ze[cj + g] : 1023;
            auto zg = [&](int c0, int nc) {
                const int64_t oz = t * m2 * m + c0;
                const z2 *Z = a.Z;
                return [=](int i, int k) {
                    const int64_t o = oz + k * m2 + i;
                    return ((FULL || (i < nc && k < m)) && CRS_IN(*ap, kDbgZ, o)) ? Z[o] : zmk(0.0, 0.0);
                };
            };
            auto zgi = zg(ci, ni), zgj = zg(cj, nj);
            if (__any_sync(0xffffffffu, ei < 600 || ej < 600)) {
                split_tile<kConjA, false, KS>(g8, zgi, zgj, {ni, nj, zi == zj ? kGram : kFull}, zi == zj, v, ex);
            } else {
                split_tile_on<kConjA, KS>(
                    g8, [&](int i, int k) { return (FULL || (i < ni && k < m)) ? zi[k * LDZ + i] : zero_on; },
                    [&](int i, int k) { return (FULL || (i < nj && k < m)) ? zj[k * LDZ + i] : zero_on; }, zi == zj, v);
#pragma unroll
                for (int j = 0; j < 2; ++j) ex[j] = ei + __shfl_sync(0xffffffffu, ej, 8 * tq + 4 * j);
                const int *zim = sE + b * SE + 5 * MT;
                const unsigned im = ((FULL || g < ni) ? zim[ci + g] : 0) | ((FULL || g < nj) ? zim[cj + g] : 0);
                split_recheck<kConjA, 4>(g8, zgi, zgj, {ni, nj, zi == zj ? kGram : kFull}, im, SplitGrid{ei, ej}, v, ex);
            }
        }
        const int p = 8 * I + g;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int q = 8 * J + 2 * tq + j;
            if (!FULL && (p >= m || q >= m)) continue;
            if (!pJ) {
                if (q <= p) put_v(b, p, q, sub_qq(u[j], p, q, v[j], ex[j]));
                continue;
            }
            z2 w = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
            if (!pI) {
                put_qp(b, p, q, w);
            } else if (q <= p) {
                if (p == q) w.y = 0.0;
                put_pp(b, p, q, w);
            }
        }
    };

    if constexpr (MT == 8) {
        // Blocks that fill at least half of the warps: one warp takes a block
        // through all five products, Z staying in registers (an entry of Z is
        // in the lane that needs it for Z^H Z, and X, P and Q are cut once).
        // Halves the integer work per block against the tasks below, which
        // spread a block over warps; the same numbers.
        if (2 * nbh > nw) {
            for (int b = warp; b < nbh; b += nw) {
                const int64_t t = t0 + b;
                const bool hasL = t >= 1, hasR = 2 * t + 1 < a.Nl;
                z2 *Zb = sZ + b * MT * LDZ;
                const z2 *Xb = sL + b * SL;
                auto xl = [=](int i, int k) { return ((FULL || i < m) && k <= i) ? Xb[tri(i, k)] : zmk(0.0, 0.0); };
                z2 x[2], z[2][2];
                SplitCut cx, cz[2];
                SplitJoint jt[2];
                unsigned mx[2], mz[2], im[2] = {0, 0};
                bool ok = true;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int k = 2 * tq + j;
                    x[j] = xl(g, k);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        z[h][j] = (FULL || (g < m && k < m)) ? Zb[k * LDZ + (h ? m : 0) + g] : zero;
                        im[h] |= im_bits(z[h][j]) | im_bits(x[j]);
                    }
                    const int64_t o = t * mm + g * m + k;
                    if ((FULL || (g < m && k < m)) && CRS_IN(a, kDbgL, o)) a.L[o] = x[j];
                }
                split_joint_exp(x[0], x[1], mx[0], mx[1]);
                const int c0 = split_exp(mx[0]), c1 = split_exp(mx[1]);
                split_cut(cx, x[0], x[1], c0, c1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    jt[h].term(split_mag(z[h][0]), mx[0]);
                    jt[h].term(split_mag(z[h][1]), mx[1]);
                    if (jt[h].finish() || jt[h].ea < kSplitSumTiny) ok = false;
                    split_cut(cz[h], z[h][0], z[h][1], jt[h].ea - c0, jt[h].ea - c1);
                    SplitAcc acc;
                    split_start(acc, kSplitStart);
                    split_mma<kPlain>(cz[h], cx, acc);
                    z2 v[2];
                    split_sums(acc, v);
                    const z2 *Bs = Zb + (h ? m : 0);
                    auto bl = [=](int i, int k) { return (FULL || (i < m && k < m)) ? Bs[k * LDZ + i] : zmk(0.0, 0.0); };
                    if (split_needs<1>(1, bl, xl, {m, m, kFull}, im[h], SplitGridJoint{jt[h].ea}, v)) ok = false;
#pragma unroll
                    for (int j = 0; j < 2; ++j) z[h][j] = zmk(split_scaled(v[j].x, jt[h].ea), split_scaled(v[j].y, jt[h].ea));
                    mz[h] = split_max4(max(split_mag(z[h][0]), split_mag(z[h][1])));
                    if (split_unsafe(mz[h])) ok = false;
                }
                const int ez[2] = {split_exp(mz[0]), split_exp(mz[1])};
                if (2 * min(ez[0], ez[1]) < kSplitSumTiny) ok = false;
                ok = __all_sync(0xffffffffu, ok);
                if (lane == 0) sC[b * Split64<MT>::SC].x = ok ? 1.0 : 0.0;
                __syncwarp();
                if (!ok) {      // out of the split's range, or a small entry of Z
                    z_task(b, 0);
                    z_task(b, 1);
                    __syncwarp();
                    h_task(b, 0, 0);
                    h_task(b, 0, 1);
                    continue;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int r = 2 * tq + j;
                        const int64_t o = t * 2 * (int64_t)mm + r * m2 + (h ? m : 0) + g;
                        if ((FULL || (g < m && r < m)) && CRS_IN(a, kDbgZ, o)) a.Z[o] = z[h][j];
                    }
                    split_cut(cz[h], z[h][0], z[h][1], ez[h], ez[h]);
                    im[h] = im_bits(z[h][0]) | im_bits(z[h][1]);
                }
                __syncwarp();       // Z is stored
                unsigned again = 0;     // products with small entries
                // P^H P, Q^H P, Q^H Q
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    const int hi = f > 0, hj = f > 1;
                    if ((!hj && !hasL) || (hi && !hasR)) continue;
                    SplitAcc acc;
                    split_start(acc, kSplitStart);
                    split_mma<kConjA>(cz[hi], cz[hj], acc);
                    z2 v[2];
                    int ex[2];
                    split_sums(acc, v);
#pragma unroll
                    for (int j = 0; j < 2; ++j) ex[j] = ez[hi] + __shfl_sync(0xffffffffu, ez[hj], 8 * tq + 4 * j);
                    const z2 *Z = a.Z + t * 2 * (int64_t)mm;
                    auto zl = [=](int h) {
                        return [=](int i, int k) {
                            return ((FULL || (i < m && k < m)) && CRS_IN(*ap, kDbgZ, t * 2 * (int64_t)mm + k * m2 + h * m + i)) ? Z[k * m2 + h * m + i]
                                                                                                                       : zmk(0.0, 0.0);
                        };
                    };
                    if (split_needs<1>(1, zl(hi), zl(hj), {m, m, f != 1 ? kGram : kFull}, im[hi] | im[hj],
                                       SplitGrid{ez[hi], ez[hj]}, v)) {
                        again |= 1u << f;
                        continue;
                    }
                    if (f == 2 && again) continue;      // (Q^H Q takes Z's place in sZ)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int p = g, q = 2 * tq + j;
                        if ((!FULL && (p >= m || q >= m)) || (f != 1 && q > p)) continue;
                        if (f == 2) {
                            Zb[p * LDZ + q] = sub_qq(load_a(b, p, q), p, q, v[j], ex[j]);
                        } else {
                            z2 w = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
                            if (f == 1) {
                                put_qp(b, p, q, w);
                            } else {
                                if (p == q) w.y = 0.0;
                                put_pp(b, p, q, w);
                            }
                        }
                    }
                }
                if (again) {        // by tasks, Q^H Q below
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const int r = 2 * tq + j;
                            const int64_t o = t * 2 * (int64_t)mm + r * m2 + (h ? m : 0) + g;
                            if (FULL || (g < m && r < m)) Zb[r * LDZ + (h ? m : 0) + g] = CRS_IN(a, kDbgZ, o) ? a.Z[o] : zero;
                        }
                    if (lane == 0) sC[b * Split64<MT>::SC].x = 0.0;
                    __syncwarp();
                    if (again & 1) h_task(b, 0, 0);
                    if (again & 2) h_task(b, 0, 1);
                }
            }
            __syncthreads();
            for (int b = warp; b < nbh; b += nw) {
                if (2 * (t0 + b) + 1 >= a.Nl) continue;
                if (sC[b * Split64<MT>::SC].x == 0.0) {
                    h_task(b, 1, 0);
                    continue;
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int p = g, q = 2 * tq + j;
                    if ((FULL || p < m) && q <= p) put_v(b, p, q, sZ[(b * MT + p) * LDZ + q]);
                }
            }
            __syncthreads();
        }
    }
    if constexpr (kOn) {
        // X is stored, and put on its grid in place where all of its columns are
        // in the split's range: column exponents, row exponents, entries.
        constexpr unsigned kAll = 0xffffffffu;
        for (int e = warp; e < nbh * m; e += nw) {
            const int b = e / m, k = e - b * m;
            unsigned mx = 0, im = 0;
            for (int r = k + lane; r < m; r += 32) {
                mx = max(mx, split_mag(sL[b * SL + tri(r, k)]));
                im |= im_bits(sL[b * SL + tri(r, k)]);
            }
            for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(kAll, mx, o));
            im = __any_sync(kAll, im != 0u);
            if (lane == 0) {
                sE[b * SE + k] = split_unsafe(mx) ? 0 : split_exp(mx);
                sE[b * SE + 4 * MT + k] = im;
            }
        }
        __syncthreads();
        for (int e = warp; e < nbh * m; e += nw) {
            const int b = e / m, r = e - b * m;
            int rho = -4096;
            for (int k = lane; k <= r; k += 32) {
                const unsigned n = split_mag(sL[b * SL + tri(r, k)]);
                if (n) rho = max(rho, (int)(n >> 20) - sE[b * SE + k]);
            }
            for (int o = 16; o; o >>= 1) rho = max(rho, __shfl_xor_sync(kAll, rho, o));
            if (lane == 0) sE[b * SE + MT + r] = max(rho, -40);     // keeps E - e above 58 for zeros
        }
        __syncthreads();
        for (int e = tid; e < nbh * mm; e += NT) {
            const int b = e / mm, rem = e - b * mm, r = rem / m, c = rem - r * m;
            z2 x = zero;
            if (r >= c) {
                z2 *p = sL + b * SL + tri(r, c);
                x = *p;
                *p = split_onto(x, sE[b * SE + c] + sE[b * SE + MT + r]);
            }
            if (CRS_IN(a, kDbgL, (t0 + b) * mm + rem)) a.L[(t0 + b) * mm + rem] = x;
        }
        __syncthreads();
        for (int e = warp; e < nbh * ngrp; e += nw) {
            const int b = e / ngrp, cg = e - b * ngrp;
            const int64_t t = t0 + b;
            const bool inP = cg < g8;
            const int c0 = 8 * (inP ? cg : cg - g8), nc = m - c0, col = (inP ? c0 : m + c0) + g;
            const int *xe = sE + b * SE;
            int *ze = sE + b * SE + 2 * MT;
            z2 *Zb = sZ + b * MT * LDZ;
            const z2 *Xb = sL + b * SL;
            auto zc = [&](int k) { return (FULL || (g < nc && k < m)) ? Zb[k * LDZ + col] : zero; };
            // B's columns onto the joint grid
            SplitJoint jt;
            bool xbad = false;
            unsigned im = 0;
            for (int s = 0; s < g8; ++s)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int k = 8 * s + 2 * tq + u, c = (FULL || k < m) ? xe[k] : 1023;
                    xbad |= c == 0;
                    im |= im_bits(zc(k)) | ((FULL || k < m) ? xe[4 * MT + k] : 0);
                    // (a column of X has its diagonal entry)
                    jt.term(split_mag(zc(k)), (unsigned)c << 20);
                }
            bool ok = !jt.finish() && !xbad && jt.ea - 40 >= kSplitSumTiny;
            ok = __all_sync(kAll, ok);
            if (!(inP ? t >= 1 : 2 * t + 1 < a.Nl)) {
                ok = false;     // no coupling: Z is zero, as staged
            } else if (!ok) {
                z_task(b, cg);
            } else {
                const z2 *BL = a.B, *XL = a.L;
                auto bg = [=](int i, int k) {       // the columns as the level has them
                    if (!FULL && (i >= nc || k >= m)) return zmk(0.0, 0.0);
                    const int64_t o = inP ? (2 * t - 1) * mm + k * m + c0 + i : 2 * t * mm + (c0 + i) * m + k;
                    if (!CRS_IN(*ap, kDbgB, o)) return zmk(0.0, 0.0);
                    return inP ? BL[o] : zconj(BL[o]);
                };
                for (int s = 0; s < g8; ++s)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int k = 8 * s + 2 * tq + u;
                        if (FULL || (g < nc && k < m)) Zb[k * LDZ + col] = split_onto(Zb[k * LDZ + col], jt.ea - xe[k]);
                    }
                __syncwarp();
                for (int R = g8 - 1; R >= 0; --R) {
                    z2 v[2];
                    int ex[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) ex[j] = jt.ea + ((FULL || 8 * R + 2 * tq + j < m) ? xe[MT + 8 * R + 2 * tq + j] : 0);
                    split_tile_on<kPlain, KS>(
                        R + 1, [&](int i, int k) { return (FULL || (i < nc && k < m)) ? Zb[k * LDZ + col - g + i] : zero_on; },
                        [&](int i, int k) { return ((FULL || 8 * R + i < m) && k <= 8 * R + i) ? Xb[tri(8 * R + i, k)] : zero_on; }, false, v);
                    auto xg = [=](int i, int k) {
                        const int64_t o = t * mm + (8 * R + i) * m + k;
                        return ((FULL || 8 * R + i < m) && k <= 8 * R + i && CRS_IN(*ap, kDbgL, o)) ? XL[o] : zmk(0.0, 0.0);
                    };
                    const int ea = jt.ea, er = (FULL || 8 * R + g < m) ? xe[MT + 8 * R + g] : 0;
                    auto grid = [=](int s, z2, z2, int (&ga)[2], int (&gb)[2]) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int k = 8 * s + 2 * tq + u, c = (FULL || k < m) ? xe[k] : 1023;
                            ga[u] = ea - c;
                            gb[u] = c + er;
                        }
                    };
                    split_recheck<kPlain, 4>(R + 1, bg, xg, {nc, m - 8 * R, kFull}, im, grid, v, ex);
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int r = 8 * R + 2 * tq + j;
                        if (FULL || (g < nc && r < m)) {
                            const int64_t o = t * m2 * m + r * m2 + col;
                            const z2 w = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
                            Zb[r * LDZ + col] = w;
                            if (CRS_IN(a, kDbgZ, o)) a.Z[o] = w;
                        }
                    }
                    __syncwarp();
                }
            }
            if (!ok && (FULL || g < nc))
                for (int r = tq; r < m; r += 4) {
                    const int64_t o = t * m2 * m + r * m2 + col;
                    if (CRS_IN(a, kDbgZ, o)) a.Z[o] = Zb[r * LDZ + col];
                }
            // Z's columns onto their own grid
            unsigned mx = 0;
            im = 0;
            for (int s = 0; s < g8; ++s)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const z2 z = zc(8 * s + 2 * tq + u);
                    mx = max(mx, split_mag(z));
                    im |= im_bits(z);
                }
            mx = split_max4(mx);
            im = split_max4(im);
            const int ez = split_unsafe(mx) ? 0 : split_exp(mx);
            if (FULL || g < nc) {
                if (tq == 0) {
                    ze[col] = ez;
                    ze[3 * MT + col] = im != 0u;
                }
                for (int s = 0; s < g8; ++s)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int k = 8 * s + 2 * tq + u;
                        if (FULL || k < m) Zb[k * LDZ + col] = split_onto(Zb[k * LDZ + col], ez);
                    }
            }
        }
        __syncthreads();
    } else if (MT > 8 || 2 * nbh <= nw) {
        for (int e = warp; e < nbh * ngrp; e += nw) z_task(e / ngrp, e % ngrp);
        // keep X
        for (int e = tid; e < nbh * mm; e += NT) {
            const int b = e / mm, rem = e - b * mm, r = rem / m, c = rem - r * m;
            if (CRS_IN(a, kDbgL, (t0 + b) * mm + rem)) a.L[(t0 + b) * mm + rem] = r >= c ? sL[b * SL + tri(r, c)] : zero;
        }
        __syncthreads();
    }
    if (MT > 8 || 2 * nbh <= nw) {
        for (int pass = 0; pass < 2; ++pass) {
            const int nt = pass == 0 ? ntri + g8 * g8 : ntri;
            for (int e = warp; e < nbh * nt; e += nw) h_task(e / nt, pass, e % nt);
            __syncthreads();
        }
    }
    if (a.bd_count) {
        const int nl = m * (m + 1) / 2;
        const int sec = bd_arrive(a.bd_count, chunk, crs_num_ctas(a.no, a.nb));
        for (int e = tid; e < ((sec & 1) ? nl : 0); e += NT) factor_fix_entry<double, true>(a, chunk, e);
        for (int e = tid; e < ((sec & 2) ? nl : 0); e += NT) factor_fix_entry<double, true>(a, chunk + 1, e);
    }
}

// One chunk of nb odd blocks and right-hand-side columns [cchunk*kc, +kc) of
// a down-sweep level: r = X y_odd, then P^H r, then v = (y_even - Q^H r) - P^H r.
// One warp per block, 8 rows and 8 columns.
template <int MT, bool FULL>
__device__ __forceinline__ void solve_down_split(const LevelArgs &a, int64_t chunk, int cchunk,
                                                       unsigned char *smem_raw) {
    [[maybe_unused]] const LevelArgs *const ap = &a;    // for bounds-checked loads in closures
    constexpr int KS = MT / 8;
    const int m = FULL ? MT : a.m, k = a.k, nb = a.nb, kc = a.kc, NT = blockDim.x, tid = threadIdx.x;
    const int mm = m * m, m2 = 2 * m, mk = m * k;
    const int cb = cchunk * kc, kw = min(kc, k - cb);
    const int64_t t0 = chunk * nb;
    const int nbh = (int)min((int64_t)nb, a.no - t0);
    z2 *sR = reinterpret_cast<z2 *>(smem_raw);              // [nb][MT][kc] r of odd t0 + b
    z2 *sW = sR + (size_t)nb * MT * kc;                       // [nb][MT][kc] P^H r of odd t0 + b
    const z2 zero = zmk(0.0, 0.0);
    const int lane = tid & 31, g = lane >> 2, tq = lane & 3, warp = tid >> 5, nw = NT >> 5;
    const int g8 = (FULL || KS == 1) ? KS : (m + 7) >> 3, ncg = (kw + 7) >> 3, per = g8 * ncg;

    // Operands of block b: columns n0 .. of y_odd, rows 8 R .. of X, columns 8 G ..
    // of P (h = 0) or Q.
    auto y_of = [&](int b, int n0) {
        const int64_t yo = 2 * (t0 + b) * mk + cb + n0;
        const z2 *y = a.y;
        const int nc = kw - n0;
        return [=](int i, int s) { return (i < nc && (FULL || s < m) && CRS_IN(*ap, kDbgY, yo + s * k + i)) ? y[yo + s * k + i] : zmk(0.0, 0.0); };
    };
    auto x_of = [&](int b, int R) {
        const int64_t xo = (t0 + b) * mm + 8 * R * m;
        const z2 *X = a.L;
        return [=](int i, int s) {
            return ((FULL || 8 * R + i < m) && s <= 8 * R + i && CRS_IN(*ap, kDbgL, xo + i * m + s)) ? X[xo + i * m + s] : zmk(0.0, 0.0);
        };
    };
    auto z_of = [&](int b, int h, int G) {
        const int64_t zo = (t0 + b) * m2 * m + (h ? m : 0) + 8 * G;
        const z2 *Z = a.Z;
        return [=](int i, int s) {
            return ((FULL || (8 * G + i < m && s < m)) && CRS_IN(*ap, kDbgZ, zo + s * m2 + i)) ? Z[zo + s * m2 + i] : zmk(0.0, 0.0);
        };
    };
    // r of rows 8 R .. and columns n0 .. of block b
    auto r_task = [&](int b, int R, int n0) {
        const int64_t t = t0 + b;
        const int nc = kw - n0;
        z2 v[2];
        int ex[2];
        split_tile<kPlain, true, KS>(R + 1, y_of(b, n0), x_of(b, R), {nc, m - 8 * R, kFull}, false, v, ex);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = 8 * R + 2 * tq + j;
            if (g >= nc || (!FULL && r >= m)) continue;
            const z2 w = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
            sR[(b * MT + r) * kc + n0 + g] = w;
            const int64_t o = t * mk + r * k + cb + n0 + g;
            if (CRS_IN(a, kDbgR, o)) a.r[o] = w;
        }
    };
    // Entry (p, n) of P^H r: kept in sW, or for the chunk's first block given to
    // the previous chunk.
    auto put_pr = [&](int b, int p, int n, z2 w) {
        const int64_t t = t0 + b, rem = (int64_t)p * k + cb + n;
        if (b > 0) {
            sW[(b * MT + p) * kc + n] = w;
        } else if (a.inline_fix) {
            const int64_t o = (t - 1) * mk + rem;
            if (CRS_IN(a, kDbgYn, o)) a.yn[o] = zsub(a.yn[o], w);
        } else if (CRS_IN(a, kDbgCbd, chunk * mk + rem)) {
            a.cbd[chunk * mk + rem] = w;
        }
    };
    // v from y_even - Q^H r
    auto put_v = [&](int b, int p, int n, z2 w) {
        const int64_t o = (t0 + b) * mk + (int64_t)p * k + cb + n;
        if (b + 1 < nbh) w = zsub(w, sW[((b + 1) * MT + p) * kc + n]);
        if (CRS_IN(a, kDbgYn, o)) a.yn[o] = w;
    };
    auto load_y = [&](int b, int p, int n) {     // y_even, ahead of the product
        const int64_t o = (2 * (t0 + b) + 1) * mk + (int64_t)p * k + cb + n;
        return ((FULL || p < m) && n < kw && 2 * (t0 + b) + 1 < a.Nl && CRS_IN(a, kDbgY, o)) ? a.y[o] : zero;
    };
    // rows 8 G .. of P^H r (pass 0) or Q^H r (pass 1); keep: y_even - Q^H r goes to
    // sR in the place of r
    auto u_task = [&](int b, int pass, int G, int n0, bool keep) {
            const int64_t t = t0 + b;
            if (pass ? 2 * t + 1 >= a.Nl : t < 1) return;
            const int nc = kw - n0, np = m - 8 * G;
            const z2 *Rb = sR + b * MT * kc + n0;
            z2 v[2], u[2];
            int ex[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) u[j] = pass ? load_y(b, 8 * G + g, n0 + 2 * tq + j) : zero;
            split_tile<kConjA, false, KS>(
                g8, z_of(b, pass, G),
                [=](int i, int s) { return (i < nc && (FULL || s < m)) ? Rb[s * kc + i] : zmk(0.0, 0.0); }, {np, nc, kFull}, false, v, ex);
            if (keep) __syncwarp();     // sR is read up to here
            const int p = 8 * G + g;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int n = 2 * tq + j;
                if ((!FULL && p >= m) || n >= nc) continue;
                if (pass == 0) {
                    put_pr(b, p, n0 + n, zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j])));
                } else {
                    const double sc = -split_scale(ex[j]);
                    const z2 w = zmk(fma(v[j].x, sc, u[j].x), fma(v[j].y, sc, u[j].y));
                    if (keep) sR[(b * MT + p) * kc + n0 + n] = w;
                    else put_v(b, p, n0 + n, w);
                }
            }
    };

    if constexpr (MT == 8) {
        // One warp per block and 8 columns: all operands loaded at once, r stays
        // in the lanes that need it for Z^H r; the same numbers as the tasks.
        constexpr unsigned kAll = 0xffffffffu;
        for (int e = warp; e < nbh * ncg; e += nw) {
            const int b = e / ncg, n0 = 8 * (e - b * ncg);
            const int64_t t = t0 + b;
            const bool hasL = t >= 1, hasR = 2 * t + 1 < a.Nl;
            const int nc = kw - n0;
            z2 x[2], y[2], z[2][2], u[2], r[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int s = 2 * tq + j;
                const int64_t oy = 2 * t * mk + (int64_t)s * k + cb + n0 + g, ox = t * mm + g * m + s, oz = t * m2 * m + s * m2 + g;
                y[j] = (g < nc && (FULL || s < m) && CRS_IN(a, kDbgY, oy)) ? a.y[oy] : zero;
                x[j] = ((FULL || g < m) && s <= g && CRS_IN(a, kDbgL, ox)) ? a.L[ox] : zero;
                z[0][j] = (hasL && (FULL || (g < m && s < m)) && CRS_IN(a, kDbgZ, oz)) ? a.Z[oz] : zero;
                z[1][j] = (hasR && (FULL || (g < m && s < m)) && CRS_IN(a, kDbgZ, oz + m)) ? a.Z[oz + m] : zero;
                u[j] = load_y(b, g, n0 + s);
            }
            unsigned mx[2], mz[2];
            unsigned im = im_bits(y[0]) | im_bits(y[1]) | im_bits(x[0]) | im_bits(x[1]);
            SplitJoint jt;
            split_joint_exp(x[0], x[1], mx[0], mx[1]);
            jt.term(split_mag(y[0]), mx[0]);
            jt.term(split_mag(y[1]), mx[1]);
            bool ok = !jt.finish() && jt.ea >= kSplitSumTiny;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                mz[h] = split_max4(max(split_mag(z[h][0]), split_mag(z[h][1])));
                if (split_unsafe(mz[h]) || split_exp(mz[h]) < kSplitSumTiny / 2) ok = false;
            }
            SplitCut c1, c2;
            SplitAcc acc;
            {
                const int e0 = split_exp(mx[0]), e1 = split_exp(mx[1]);
                split_cut(c1, y[0], y[1], jt.ea - e0, jt.ea - e1);
                split_cut(c2, x[0], x[1], e0, e1);
                split_start(acc, kSplitStart);
                split_mma<kPlain>(c1, c2, acc);
                split_sums(acc, r);
                if (split_needs<1>(1, y_of(b, n0), x_of(b, 0), {nc, m, kFull}, im, SplitGridJoint{jt.ea}, r)) ok = false;
#pragma unroll
                for (int j = 0; j < 2; ++j) r[j] = zmk(split_scaled(r[j].x, jt.ea), split_scaled(r[j].y, jt.ea));
            }
            const unsigned mr = split_max4(max(split_mag(r[0]), split_mag(r[1])));
            const int er = split_exp(mr);
            if (split_unsafe(mr) || er < kSplitSumTiny / 2) ok = false;
            if (!__all_sync(kAll, ok)) {        // out of the split's range, or a small entry of r
                r_task(b, 0, n0);
                __syncwarp();
                u_task(b, 0, 0, n0, false);
                __syncwarp();
                u_task(b, 1, 0, n0, true);
                continue;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int64_t o = t * mk + (int64_t)(2 * tq + j) * k + cb + n0 + g;
                if (g < nc && (FULL || 2 * tq + j < m) && CRS_IN(a, kDbgR, o)) a.r[o] = r[j];
            }
            split_cut(c2, r[0], r[1], er, er);
            const unsigned ir = im_bits(r[0]) | im_bits(r[1]);
            __syncwarp();       // r is stored
            unsigned again = 0;     // products with small entries
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h ? !hasR : !hasL) continue;
                const int ez = split_exp(mz[h]);
                split_cut(c1, z[h][0], z[h][1], ez, ez);
                split_start(acc, kSplitStart);
                split_mma<kConjA>(c1, c2, acc);
                z2 v[2];
                int ex[2];
                split_sums(acc, v);
#pragma unroll
                for (int j = 0; j < 2; ++j) ex[j] = ez + __shfl_sync(kAll, er, 8 * tq + 4 * j);
                const int64_t ro = t * mk + cb + n0;
                const z2 *Rg = a.r;
                auto rl = [=](int i, int s) {
                    return (i < nc && (FULL || s < m) && CRS_IN(*ap, kDbgR, ro + s * k + i)) ? Rg[ro + s * k + i] : zmk(0.0, 0.0);
                };
                if (split_needs<1>(1, z_of(b, h, 0), rl, {m, nc, kFull}, ir | im_bits(z[h][0]) | im_bits(z[h][1]),
                                   SplitGrid{ez, er}, v)) {
                    again |= 1u << h;
                    continue;
                }
                if (h == 1 && again) continue;      // (y - Q^H r takes the place of r in sR)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int n = 2 * tq + j;
                    if ((!FULL && g >= m) || n >= nc) continue;
                    if (h == 0) {
                        put_pr(b, g, n0 + n, zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j])));
                    } else {
                        const double sc = -split_scale(ex[j]);
                        sR[(b * MT + g) * kc + n0 + n] = zmk(fma(v[j].x, sc, u[j].x), fma(v[j].y, sc, u[j].y));
                    }
                }
            }
            if (again) {        // by tasks
                r_task(b, 0, n0);
                __syncwarp();
                if (again & 1) u_task(b, 0, 0, n0, false);
                __syncwarp();
                u_task(b, 1, 0, n0, true);
            }
        }
        __syncthreads();
        for (int e = warp; e < nbh * ncg; e += nw) {
            const int b = e / ncg, n0 = 8 * (e - b * ncg);
            if (2 * (t0 + b) + 1 >= a.Nl) continue;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int n = n0 + 2 * tq + j;
                if ((FULL || g < m) && n < kw) put_v(b, g, n, sR[(b * MT + g) * kc + n]);
            }
        }
        __syncthreads();
    } else {
        for (int e = warp; e < nbh * per; e += nw) {
            const int b = e / per, rem = e - b * per, R = rem / ncg;
            r_task(b, R, 8 * (rem - R * ncg));
        }
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {      // 0: P^H r, 1: Q^H r
            for (int e = warp; e < nbh * per; e += nw) {
                const int b = e / per, rem = e - b * per, G = rem / ncg;
                u_task(b, pass, G, 8 * (rem - G * ncg), false);
            }
            __syncthreads();
        }
    }
    if (a.bd_count) {
        // counters of this right-hand-side chunk: [cchunk][boundary]
        const int64_t ncta = crs_num_ctas(a.no, a.nb);
        const int sec = bd_arrive(a.bd_count + cchunk * ncta, chunk, ncta);
        for (int e = tid; e < ((sec & 1) ? m * kw : 0); e += NT)
            solve_down_fix_entry<double, true>(a, chunk, (e / kw) * k + cb + e % kw);
        for (int e = tid; e < ((sec & 2) ? m * kw : 0); e += NT)
            solve_down_fix_entry<double, true>(a, chunk + 1, (e / kw) * k + cb + e % kw);
    }
}

// One chunk of an up-sweep level: w = r - Z [x_left; x_right], x_odd = X^H w; the
// even unknowns are copied.
template <int MT, bool FULL>
__device__ __forceinline__ void solve_up_split(const LevelArgs &a, int64_t chunk, int cchunk,
                                                     unsigned char *smem_raw) {
    [[maybe_unused]] const LevelArgs *const ap = &a;    // for bounds-checked loads in closures
    constexpr int KS = MT / 8;
    const int m = FULL ? MT : a.m, k = a.k, nb = a.nb, kc = a.kc, NT = blockDim.x, tid = threadIdx.x;
    const int mm = m * m, m2 = 2 * m, mk = m * k;
    const int cb = cchunk * kc, kw = min(kc, k - cb);
    const int64_t t0 = chunk * nb;
    const int nbh = (int)min((int64_t)nb, a.no - t0);
    z2 *sW = reinterpret_cast<z2 *>(smem_raw);              // [nb][MT][kc]
    const z2 zero = zmk(0.0, 0.0);
    const int lane = tid & 31, g = lane >> 2, tq = lane & 3, warp = tid >> 5, nw = NT >> 5;
    const int g8 = (FULL || KS == 1) ? KS : (m + 7) >> 3, ncg = (kw + 7) >> 3, per = g8 * ncg;

    const bool failed = a.level == 0 && *a.status != CRS_NO_FAIL;   // the result is NaN
    // the even unknowns (MT = 8: below, with the lanes' operands)
    for (int e = tid; e < ((MT > 8 || failed) ? nbh * m * kw : 0); e += NT) {
        const int b = e / (m * kw), rem = e - b * (m * kw), r = rem / kw, c = rem - r * kw;
        const int64_t t = t0 + b, o = (int64_t)r * k + cb + c;
        if (failed && CRS_IN(a, kDbgX, 2 * t * mk + o)) a.x[2 * t * mk + o] = zmk(qnan(0.0), qnan(0.0));
        if (t < a.ne && CRS_IN(a, kDbgX, (2 * t + 1) * mk + o))
            a.x[(2 * t + 1) * mk + o] =
                failed ? zmk(qnan(0.0), qnan(0.0)) : (CRS_IN(a, kDbgXn, t * mk + o) ? a.xn[t * mk + o] : zero);
    }
    if (failed) return;

    // Operands of block b: columns n0 .. of [x_left; x_right] and rows 8 R .. of [P | Q]
    // (terms 0 .. 8 g8 - 1: P and x_left, 8 g8 .. : Q and x_right), columns 8 G .. of
    // X from row 8 G on (X[s][p] is zero for s < p).
    auto xn_of = [&](int b, int n0) {
        const int64_t t = t0 + b, xo = t * mk + cb + n0;
        const bool hasL = t >= 1, hasR = t < a.ne;
        const z2 *xn = a.xn;
        const int nc = kw - n0;
        return [=](int i, int s) {
            const bool right = s >= 8 * g8;
            const int q = right ? s - 8 * g8 : s;
            const int64_t o = xo + (right ? 0 : -mk) + q * k + i;
            return (i < nc && (FULL || q < m) && (right ? hasR : hasL) && CRS_IN(*ap, kDbgXn, o)) ? xn[o] : zmk(0.0, 0.0);
        };
    };
    auto z_of = [&](int b, int R) {
        const int64_t zo = (t0 + b) * m2 * m + 8 * R * m2;
        const z2 *Z = a.Z;
        return [=](int i, int s) {
            const bool right = s >= 8 * g8;
            const int q = right ? s - 8 * g8 : s;
            const int64_t o = zo + i * m2 + (right ? m : 0) + q;
            return ((FULL || (8 * R + i < m && q < m)) && CRS_IN(*ap, kDbgZ, o)) ? Z[o] : zmk(0.0, 0.0);
        };
    };
    auto x_of = [&](int b, int G) {
        const int64_t xo = (t0 + b) * mm + 8 * G * m + 8 * G;
        const int np = m - 8 * G;
        const z2 *X = a.L;
        return [=](int i, int s) {
            return ((FULL || (i < np && s < np)) && i <= s && CRS_IN(*ap, kDbgL, xo + s * m + i)) ? X[xo + s * m + i] : zmk(0.0, 0.0);
        };
    };
    auto w_task = [&](int b, int R, int n0) {
        const int64_t t = t0 + b;
        const int nc = kw - n0;
        z2 v[2], u[2];
        int ex[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {       // r, loaded ahead of the product
            const int64_t o = t * mk + (int64_t)(8 * R + 2 * tq + j) * k + cb + n0 + g;
            u[j] = (g < nc && (FULL || 8 * R + 2 * tq + j < m) && CRS_IN(a, kDbgR, o)) ? a.r[o] : zero;
        }
        split_tile<kPlain, true, 2 * KS>(2 * g8, xn_of(b, n0), z_of(b, R), {nc, m - 8 * R, kFull}, false, v, ex);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = 8 * R + 2 * tq + j;
            if (g >= nc || (!FULL && r >= m)) continue;
            z2 w = u[j];
            const double sc = -split_scale(ex[j]);
            w.x = fma(v[j].x, sc, w.x);
            w.y = fma(v[j].y, sc, w.y);
            sW[(b * MT + r) * kc + n0 + g] = w;
        }
    };
    auto x_task = [&](int b, int G, int n0) {
        const int64_t t = t0 + b;
        const int nc = kw - n0, np = m - 8 * G;
        const z2 *Wb = sW + (b * MT + 8 * G) * kc + n0;
        z2 v[2];
        int ex[2];
        split_tile<kConjA, false, KS>(
            g8 - G, x_of(b, G),
            [=](int i, int s) { return (i < nc && (FULL || s < np)) ? Wb[s * kc + i] : zmk(0.0, 0.0); }, {np, nc, kFull}, false, v, ex);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int p = 8 * G + g, n = 2 * tq + j;
            const int64_t o = 2 * t * mk + (int64_t)p * k + cb + n0 + n;
            if ((FULL || p < m) && n < nc && CRS_IN(a, kDbgX, o))
                a.x[o] = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
        }
    };

    if constexpr (MT == 8) {
        // One warp per block and 8 columns, as in the down sweep.
        constexpr unsigned kAll = 0xffffffffu;
        for (int e = warp; e < nbh * ncg; e += nw) {
            const int b = e / ncg, n0 = 8 * (e - b * ncg);
            const int64_t t = t0 + b;
            const int nc = kw - n0;
            z2 xn[2][2], z[2][2], x[2], w[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int s = 2 * tq + j;
                const bool in = FULL || (g < m && s < m);
                const int64_t o = t * mk + (int64_t)s * k + cb + n0 + g, oz = t * m2 * m + g * m2 + s, ox = t * mm + s * m + g;
                const bool col = g < nc && (FULL || s < m);
                xn[0][j] = (col && t >= 1 && CRS_IN(a, kDbgXn, o - mk)) ? a.xn[o - mk] : zero;
                xn[1][j] = (col && t < a.ne && CRS_IN(a, kDbgXn, o)) ? a.xn[o] : zero;
                w[j] = (col && CRS_IN(a, kDbgR, o)) ? a.r[o] : zero;
                z[0][j] = (in && CRS_IN(a, kDbgZ, oz)) ? a.Z[oz] : zero;
                z[1][j] = (in && CRS_IN(a, kDbgZ, oz + m)) ? a.Z[oz + m] : zero;
                x[j] = (in && g <= s && CRS_IN(a, kDbgL, ox)) ? a.L[ox] : zero;
                const int64_t oe = (2 * t + 1) * mk + (int64_t)s * k + cb + n0 + g;
                if (col && t < a.ne && CRS_IN(a, kDbgX, oe)) a.x[oe] = xn[1][j];
            }
            unsigned mx[2][2], im = 0;
            SplitJoint jt;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                split_joint_exp(z[h][0], z[h][1], mx[h][0], mx[h][1]);
                jt.term(split_mag(xn[h][0]), mx[h][0]);
                jt.term(split_mag(xn[h][1]), mx[h][1]);
                im |= im_bits(z[h][0]) | im_bits(z[h][1]) | im_bits(xn[h][0]) | im_bits(xn[h][1]);
            }
            bool ok = !jt.finish() && jt.ea >= kSplitSumTiny;
            const unsigned ml = split_max4(max(split_mag(x[0]), split_mag(x[1])));
            if (split_unsafe(ml) || split_exp(ml) < kSplitSumTiny / 2) ok = false;
            SplitCut c1, c2;
            SplitAcc acc;
            split_start(acc, 0.f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int e0 = split_exp(mx[h][0]), e1 = split_exp(mx[h][1]);
                split_cut(c1, xn[h][0], xn[h][1], jt.ea - e0, jt.ea - e1);
                split_cut(c2, z[h][0], z[h][1], e0, e1);
                split_mma<kPlain>(c1, c2, acc);
            }
            {
                z2 v[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int s0[kSplitDigits], s1[kSplitDigits];
#pragma unroll
                    for (int d = 0; d < kSplitDigits; ++d) {
                        s0[d] = __float2int_rn(acc[d][j]);
                        s1[d] = __float2int_rn(acc[d][j + 2]);
                    }
                    v[j] = zmk(split_value<2>(s0), split_value<2>(s1));
                }
                if (split_needs<2>(2, xn_of(b, n0), z_of(b, 0), {nc, m, kFull}, im, SplitGridJoint{jt.ea}, v)) ok = false;
                const double sc = -split_scale(jt.ea);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    w[j].x = fma(v[j].x, sc, w[j].x);
                    w[j].y = fma(v[j].y, sc, w[j].y);
                }
            }
            const unsigned mw = split_max4(max(split_mag(w[0]), split_mag(w[1])));
            const int ew = split_exp(mw), el = split_exp(ml);
            if (split_unsafe(mw) || ew < kSplitSumTiny / 2) ok = false;
            // by tasks: out of the split's range, or a small entry
            if (!__all_sync(kAll, ok)) {
                w_task(b, 0, n0);
                __syncwarp();
                x_task(b, 0, n0);
                continue;
            }
            split_cut(c1, x[0], x[1], el, el);
            split_cut(c2, w[0], w[1], ew, ew);
            split_start(acc, kSplitStart);
            split_mma<kConjA>(c1, c2, acc);
            z2 v[2];
            int ex[2];
            split_sums(acc, v);
#pragma unroll
            for (int j = 0; j < 2; ++j) ex[j] = el + __shfl_sync(kAll, ew, 8 * tq + 4 * j);
            const z2 *Wb = sW + b * MT * kc + n0;
            auto wl = [=](int i, int s) {       // (of the block, put into sW for this look)
                return (i < nc && (FULL || s < m)) ? Wb[s * kc + i] : zmk(0.0, 0.0);
            };
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (g < nc && (FULL || 2 * tq + j < m)) sW[(b * MT + 2 * tq + j) * kc + n0 + g] = w[j];
            __syncwarp();
            if (split_needs<1>(1, x_of(b, 0), wl, {m, nc, kFull}, im_bits(x[0]) | im_bits(x[1]) | im_bits(w[0]) | im_bits(w[1]),
                               SplitGrid{el, ew}, v)) {
                x_task(b, 0, n0);
                continue;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int n = 2 * tq + j;
                const int64_t o = 2 * t * mk + (int64_t)g * k + cb + n0 + n;
                if ((FULL || g < m) && n < nc && CRS_IN(a, kDbgX, o))
                    a.x[o] = zmk(split_scaled(v[j].x, ex[j]), split_scaled(v[j].y, ex[j]));
            }
        }
    } else {
        for (int e = warp; e < nbh * per; e += nw) {
            const int b = e / per, rem = e - b * per, R = rem / ncg;
            w_task(b, R, 8 * (rem - R * ncg));
        }
        __syncthreads();
        for (int e = warp; e < nbh * per; e += nw) {
            const int b = e / per, rem = e - b * per, G = rem / ncg;
            x_task(b, G, 8 * (rem - G * ncg));
        }
    }
}

}  // namespace crs
