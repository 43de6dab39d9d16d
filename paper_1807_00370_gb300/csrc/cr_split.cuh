// cr_split.cuh -- FP64 products of small complex blocks on the tensor cores by
// error-free splitting, one warp per 8 x 8 complex tile.
//
// Why.  GB300 has 2 FP64 FMA per clock per SM, and mma.sync m16n8k16 on FP16
// operands with FP32 accumulators does 1016 multiply-adds per clock per SM
// (both measured), so 28 of its instructions, which form one 8 x 8 x 8 complex
// product exactly from seven slices of each operand, take 56 clocks where the
// FP64 pipe takes 1024.  mma.sync and not tcgen05: the blocks are 8 to 64 wide,
// its fragments are 8 wide and live in registers, where the slices are cut.
//
// How (the splitting of Ozaki, Ogita, Oishi, Rump 2012).  Every column p of an
// operand has a binary exponent E_p, that of its largest entry.  An entry v
// becomes the integer n = trunc(|v| 2^(56 - E_p)) < 2^57: the column's largest
// entry keeps all of its 53 bits and any other entry is off by at most 2^-56 of
// the largest.  n is cut into seven digits, n = sum d_i 2^(8(6-i)) with
// 0 <= d_0 <= 512 and |d_i| <= 128, which FP16 holds exactly with v's sign.  The
// digit products with i + j <= 6 are accumulated per i + j: over 64 real terms
// (four K-steps of the instruction) these sums are at most 2^24, so FP32 holds
// them exactly.  The dropped digit products are below 2^-55 of the largest
// product and have either sign.  The sums are added up in 64-bit integers and
// rounded once.  The error is thus that of one rounding of the result plus
// about 2^-56 max|a| max|b| sqrt(K), where a chain of FP64 FMAs rounds K times.
//
// That second part is measured by the largest entries.  A result whose own terms
// are all much smaller (a localised source, rows of other units, a tiny imaginary
// part) would keep few or none of its bits, where FMAs keep them all.  Such
// results are told by their size and by their operands, and formed by FMAs
// (split_guard), so that every result is good to a few ulp of the sum of its
// own terms' magnitudes.
//
// Cutting is integer work and bounds these kernels (the integer pipe does 64
// lanes per clock per SM, measured): digits of a byte need no shifts, only a
// byte permute and a mask for two entries, which is why there are seven of
// them and not six of ten bits.
//
// Columns whose largest entry lies outside 2^-923 .. 2^477 (or is not finite)
// take FP64 FMAs instead, so overflow, infinities and NaN behave as there.
#pragma once
#include "cr_device.cuh"

namespace crs {

constexpr int kSplitDigits = 7;
// Range of the biased exponents (and, in joint scaling, of their sums) that the
// split takes.  The lower limits keep E - e above 58 for entries with exponent
// field 0, so that zeros are cut off; the upper ones keep results finite.
constexpr unsigned kSplitExpLo = 100, kSplitExpHi = 1500;
constexpr int kSplitSumHi = 2600;
// exponent sums below which a result may leave the normal range when it is scaled
constexpr int kSplitSumTiny = 1100;

// One FP16 digit plane of a 16 x 16 A operand and a 16 x 8 B operand.
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// |v| as an ordered integer (its high word without the sign).
__device__ __forceinline__ unsigned mag_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// Exponent field of a column from the largest mag_hi of its entries: a column
// of zeros takes that of 1.0 (its digits are zero).  Entries below 2^-1042
// have mag_hi = 0 and count as zero.
__device__ __forceinline__ int split_exp(unsigned mx) { return mx == 0u ? 1023 : (int)(mx >> 20); }
__device__ __forceinline__ bool split_unsafe(unsigned mx) {
    return mx != 0u && (mx < (kSplitExpLo << 20) || mx >= (kSplitExpHi << 20));
}

// n = trunc(|v| 2^(56 - E)) for exponent field e of the column, plus 128 in each
// lower digit so that the digits can be read as unsigned bytes.
__device__ __forceinline__ void split_fix(double v, int e, uint32_t &lo, uint32_t &hi) {
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const int d = e - (int)(mag_hi(v) >> 20);
    uint64_t n = ((uint64_t)((__funnelshift_l(l, h, 4) & 0x00ffffffu) | 0x01000000u) << 32) | (l << 4);
    asm("shr.u64 %0, %0, %1;" : "+l"(n) : "r"(d));   // clamps at 64: tiny entries and zeros give 0
    n += 0x0000808080808080ull;
    lo = (uint32_t)n;
    hi = (uint32_t)(n >> 32);
}

// The digits of a (low halves) and b (high halves) as FP16 pairs: bytes paired
// by one permute, read as the mantissa of 1024 + byte, and the offset taken
// off with the entry's sign (bit 31 of sa, sb) by one exact FMA.
__device__ __forceinline__ void split_digits(uint32_t la, uint32_t ha, uint32_t lb, uint32_t hb, uint32_t sa, uint32_t sb,
                                             uint32_t (&d)[kSplitDigits]) {
    const uint32_t sg = __byte_perm(sa, sb, 0x7430) & 0x80008000u;
    const uint32_t one = sg ^ 0x3c003c00u, off0 = sg ^ 0xe400e400u, off = sg ^ 0xe480e480u;   // +-1, -+1024, -+1152
    d[6] = __byte_perm(la, lb, 0x5410);
    d[5] = __byte_perm(la, lb, 0x6521);
    d[4] = __byte_perm(la, lb, 0x7632);
    d[3] = __byte_perm(la, lb, 0x4703);
    d[2] = __byte_perm(ha, hb, 0x5410);
    d[1] = __byte_perm(ha, hb, 0x6521);
    d[0] = __byte_perm(ha, hb, 0x7632);
#pragma unroll
    for (int i = 0; i < kSplitDigits; ++i) {
        const uint32_t u = (d[i] & (i == 0 ? 0x03ff03ffu : 0x00ff00ffu)) | 0x64006400u;
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d[i]) : "r"(u), "r"(one), "r"(i == 0 ? off0 : off));
    }
}

__device__ __forceinline__ void split_pair(double a, double b, int ea, int eb, uint32_t (&d)[kSplitDigits]) {
    uint32_t la, ha, lb, hb;
    split_fix(a, ea, la, ha);
    split_fix(b, eb, lb, hb);
    split_digits(la, ha, lb, hb, (uint32_t)__double2hiint(a), (uint32_t)__double2hiint(b), d);
}

// An entry on its grid, kept in the place of the double: n with its digit
// offsets and the sign in bit 63.  Operands that many tiles read are put on
// their grid once, which leaves the tiles the digits alone (a third of the
// integer work of a cut).
__device__ __forceinline__ double split_onto(double v, int e) {
    uint32_t lo, hi;
    split_fix(v, e, lo, hi);
    return __hiloint2double((int)(hi | ((uint32_t)__double2hiint(v) & 0x80000000u)), (int)lo);
}
__device__ __forceinline__ z2 split_onto(z2 z, int e) { return zmk(split_onto(z.x, e), split_onto(z.y, e)); }
// ... of zero: the digits' offsets.
__device__ __forceinline__ z2 split_zero_on() {
    const double z = __hiloint2double(0x00008080, (int)0x80808080u);
    return zmk(z, z);
}
__device__ __forceinline__ void split_pair_on(double a, double b, uint32_t (&d)[kSplitDigits]) {
    const uint32_t ha = (uint32_t)__double2hiint(a), hb = (uint32_t)__double2hiint(b);
    split_digits((uint32_t)__double2loint(a), ha, (uint32_t)__double2loint(b), hb, ha, hb, d);
}

// The three complex products of a tile, as the real A operand of row g (Re)
// and row g + 8 (Im) over K = [re of 8 terms | im of 8 terms].
enum SplitKind {
    kConjA,    // sum conj(a) b
    kPlain,    // sum a b
    kConjB     // sum a conj(b)
};

// The digits of the two terms k = 2t, 2t + 1 that a lane holds of its row or column.
struct SplitCut {
    uint32_t re[kSplitDigits], im[kSplitDigits];
};
__device__ __forceinline__ void split_cut(SplitCut &c, z2 z0, z2 z1, int e0, int e1) {
    split_pair(z0.x, z1.x, e0, e1, c.re);
    split_pair(z0.y, z1.y, e0, e1, c.im);
}

__device__ __forceinline__ void split_cut_on(SplitCut &c, z2 z0, z2 z1) {
    split_pair_on(z0.x, z1.x, c.re);
    split_pair_on(z0.y, z1.y, c.im);
}

using SplitAcc = float[kSplitDigits][4];
// Accumulators of one K-step start at 1.5 * 2^23, so that their bits are their
// integer values plus kSplitMagic (|sum| <= 2^22 over 16 terms).
constexpr float kSplitStart = 12582912.f;
constexpr int kSplitMagic = 0x4b400000;

__device__ __forceinline__ void split_start(SplitAcc &acc, float v) {
#pragma unroll
    for (int d = 0; d < kSplitDigits; ++d)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[d][j] = v;
}

// acc[i + j] += A_i B_j for i + j <= 6.
template <SplitKind KIND>
__device__ __forceinline__ void split_mma(const SplitCut &a, const SplitCut &b, SplitAcc &acc) {
#pragma unroll
    for (int i = 0; i < kSplitDigits; ++i) {
        constexpr uint32_t kNeg = 0x80008000u;
        const uint32_t a1 = KIND == kConjA ? a.im[i] ^ kNeg : a.im[i];
        const uint32_t a2 = KIND == kPlain ? a.im[i] ^ kNeg : a.im[i];
        const uint32_t a3 = KIND == kConjB ? a.re[i] ^ kNeg : a.re[i];
#pragma unroll
        for (int j = 0; i + j < kSplitDigits; ++j) mma_f16(acc[i + j], a.re[i], a1, a2, a3, b.re[j], b.im[j]);
    }
}

// The integer sum of a tile's digit products over KS K-steps (16 KS real terms) as
// a double, in units of 2^(Ea + Eb - 54), above 8 K-steps of 2^(Ea + Eb - 53), from
// the sums per digit (KS = 1: each offset by kSplitMagic).  It is below 2^63 for up
// to 128 real terms, in the larger unit up to 256.  A real term adds up to 196608 =
// 2 * 512 * 128 + 4 * 128^2 to s[5] and 212992 to s[6]: 256 s[5] + s[6] stays below
// 2^31 over the 32 terms of two K-steps, beyond it is formed in 64 bits.
template <int KS>
__host__ __device__ __forceinline__ double split_value(const int (&s)[kSplitDigits]) {
    constexpr int H = KS > 8 ? 1 : 0;
    constexpr uint64_t M = KS == 1 ? (uint64_t)kSplitMagic : 0;
    constexpr uint64_t off = (M << (38 - H)) + (M << (30 - H)) + (M << (22 - H)) + (M << (14 - H)) + (M << (6 - H));
    uint64_t v;
    if constexpr (KS <= 2) {
        const int low = (int)((uint32_t)s[5] * 256u + (uint32_t)s[6] + ((512u << H) - (uint32_t)(M * 257)));
        v = (uint64_t)(int64_t)(low >> (10 + H)) - off;
    } else {
        const int64_t low = (int64_t)s[5] * 256 + s[6] + (512 << H);
        v = (uint64_t)(low >> (10 + H));
    }
    v += (uint64_t)((int64_t)s[4] * (1 << (6 - H)));
    v += (uint64_t)((int64_t)s[3] * (1 << (14 - H)));
    v += (uint64_t)((int64_t)s[2] * (1 << (22 - H)));
    v += (uint64_t)((int64_t)s[1] * (1 << (30 - H)));
    v += (uint64_t)(uint32_t)(s[0] << (6 - H)) << 32;
    return (double)(int64_t)v;
}

// The lane's two entries of a tile of one K-step.
__device__ __forceinline__ void split_sums(const SplitAcc &acc, z2 (&v)[2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        int s0[kSplitDigits], s1[kSplitDigits];
#pragma unroll
        for (int d = 0; d < kSplitDigits; ++d) {
            s0[d] = __float_as_int(acc[d][j]);
            s1[d] = __float_as_int(acc[d][j + 2]);
        }
        v[j] = zmk(split_value<1>(s0), split_value<1>(s1));
    }
}

// v times 2^(k - 2100) for a value of split_value and a sum k of two biased
// exponents, by the exponent field (no FP64 instruction); and that factor.
__device__ __forceinline__ double split_scaled(double v, int k) {
    const int hi = __double2hiint(v);
    return (hi << 1) == 0 ? v : __hiloint2double(hi + ((k - 2100) << 20), __double2loint(v));
}
__device__ __forceinline__ double split_scale(int k) { return __hiloint2double((k - 1077) << 20, 0); }

// One 8 x 8 tile of a product of two 8-wide complex operands over 8 ks terms,
// by one warp: lane (g, t) = (lane / 4, lane % 4) gets the entries
// (row g, columns 2t + j), j = 0, 1, as v[j] times 2^(e[j] - 2100).
// la(i, k): entry k of row i of the first operand, lb(i, k): entry k of column
// i of the second; both return zero outside the block, and capture by value.
//
// Scaling.  kJoint = false: rows of the first and columns of the second
// operand each on their own binary grid.  kJoint = true, for products X b
// where the second operand holds the rows of X and the contraction runs over
// its columns: every term k has an exponent c_k, that of the tile's largest
// |X_ik|; X goes on the grid of c_k and b_k on that of max_k(|b_k| 2^c_k).  A
// scaling of the unknowns (X_ik -> X_ik / d_k, b_k -> d_k b_k) leaves such a
// product's digits as they are, as it leaves the rounding errors of FP64 FMAs.
//
// Entries whose row or column leaves the split's range, and those that
// split_guard tells, are formed by FP64 FMAs (e[j] = 2100).  use(i, c): which
// parts of entry (i, c) the caller uses (SplitUse).
//
// same: both operands are the same columns (cut once).
__device__ __forceinline__ unsigned split_mag(z2 z) { return max(mag_hi(z.x), mag_hi(z.y)); }

// c0, c1: exponents of the lane's two terms of the joint scaling (from the tile
// of X, whose terms b0, b1 the lane holds); m0, m1: the largest magnitudes.
__device__ __forceinline__ void split_joint_exp(z2 b0, z2 b1, unsigned &m0, unsigned &m1) {
    m0 = split_mag(b0);
    m1 = split_mag(b1);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
        m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
}

// Running state of the joint exponent of a row: ea (with bit 20 set when out of
// range) and the largest exponent of X's nonzero terms.
struct SplitJoint {
    int ea = 0, cmax = 0;
    __device__ __forceinline__ void term(unsigned n, unsigned mx) {
        // a term with a zero X column needs no room (its digits are zero or
        // cut off); one that is not finite is out of range in any case
        const int c = split_exp(mx);
        if (mx) cmax = max(cmax, c);
        if (n && mx) ea = max(ea, (int)(n >> 20) + c);
        if (split_unsafe(mx) || n >= 0x7ff00000u) ea |= 1 << 20;
    }
    // over the four lanes of a row: its exponent sum, and whether it is out of range
    __device__ __forceinline__ bool finish() {
        if (ea > kSplitSumHi) ea |= 1 << 20;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, o));
            cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
        }
        const bool bad = (ea >> 20) != 0 || (ea != 0 && ea < cmax + 64);
        ea &= 0xfffff;
        if (ea == 0) ea = 2046;
        return bad;
    }
};

// The largest magnitude over the four lanes of a row or column.
__device__ __forceinline__ unsigned split_max4(unsigned m) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    return max(m, __shfl_xor_sync(0xffffffffu, m, 2));
}

// ---- results much smaller than their grids' product g = 2^(Ea + Eb)
//
// The error of a result over K real terms is below K 2^-53.3 g (two operands off by
// less than 2^-56 of their grids, dropped digits below 2^-55.3 g, per term).  A
// result is kept where that is small against the sum S of its own terms' magnitudes:
// where its modulus is at least 2^-8 g and the part (real or imaginary) at least
// 2^-14 g, or where one of its real products is at least 2^-8 g.  Its error is then
// below K 2^-45.3 times the moduli's sum and K 2^-39.3 S, in the worst case that the
// largest errors of all terms add up (they have either sign).  Else, if any product is
// not zero, the entry is formed by FMAs.  On the random systems 1% of the
// tiles come here for a look at their operands, most of them (single-term rows of
// triangles) also for the FMAs; where entries decay inside a block, most tiles do.
constexpr int kSplitMod = 8, kSplitPart = 14, kSplitBig = 4;

__device__ __forceinline__ bool nonzero(double v) {
    return ((unsigned)__double2hiint(v) << 1 | (unsigned)__double2loint(v)) != 0u;
}
__device__ __forceinline__ bool nonzero(z2 z) { return nonzero(z.x) || nonzero(z.y); }

// Bits 0 and 1: the real and the imaginary part of a tile's result (in units of
// split_value<KS>) may have lost bits.
template <int KS>
__device__ __forceinline__ unsigned split_small(z2 v) {
    constexpr unsigned one = 1023 + (KS > 8 ? 53 : 54), mod = (one - kSplitMod) << 20, part = (one - kSplitPart) << 20;
    const unsigned x = mag_hi(v.x), y = mag_hi(v.y);
    return max(x, y) < mod ? 3u : (x < part ? 1u : 0u) | (y < part ? 2u : 0u);
}

// The parts of a tile's entries that a caller uses and that can be small (bits as
// of split_small): rows i < na and columns c < nb.  kHermitian: of a Hermitian tile
// the lower triangle, the diagonal real; kGram: without the diagonal, a sum of
// squares of at least g.
enum SplitShape { kFull, kHermitian, kGram };
struct SplitUse {
    int na, nb;
    SplitShape shape;
    __device__ __forceinline__ unsigned operator()(int i, int c) const {
        if (i >= na || c >= nb) return 0u;
        if (shape == kFull || c < i) return 3u;
        return shape == kHermitian && c == i ? 1u : 0u;
    }
};

// Which results of a lane have a product that is not zero (nz), or one of at
// least 2^-8 g (big): bits 2 j + (0: real, 1: imaginary part) of entry (g, 2t + j).
struct SplitSeen {
    unsigned nz = 0, big = 0;
    // one of the lane's terms: a of row g, b of column g, with their grids' exponents
    __device__ __forceinline__ void term(z2 a, int ea, z2 b, int eb) {
        constexpr unsigned kAll = 0xffffffffu;
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        auto near = [](double v, int e) { return (int)(mag_hi(v) >> 20) >= e - kSplitBig; };
        const unsigned n[4] = {__ballot_sync(kAll, nonzero(a.x)), __ballot_sync(kAll, nonzero(a.y)), __ballot_sync(kAll, nonzero(b.x)),
                               __ballot_sync(kAll, nonzero(b.y))};
        const unsigned l[4] = {__ballot_sync(kAll, near(a.x, ea)), __ballot_sync(kAll, near(a.y, ea)),
                               __ballot_sync(kAll, near(b.x, eb)), __ballot_sync(kAll, near(b.y, eb))};
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            // the four lanes of row g and those of column 2t + j
            const int r = 4 * g, c = 4 * (2 * t + j);
            auto parts = [&](const unsigned (&v)[4]) {
                const unsigned ar = v[0] >> r, ai = v[1] >> r, br = v[2] >> c, bi = v[3] >> c;
                return ((((ar & br) | (ai & bi)) & 15u) != 0u ? 1u : 0u) | ((((ar & bi) | (ai & br)) & 15u) != 0u ? 2u : 0u);
            };
            nz |= parts(n) << (2 * j);
            big |= parts(l) << (2 * j);
        }
    }
};

// A lane's entries (g, 2t + j) with fma[j] by FMAs over the K-steps in steps (bits).
// The warp goes through the terms together, without a branch on fma.  real: all
// operands are real, one FMA per term instead of four.
template <SplitKind KIND, class LA, class LB>
__device__ __forceinline__ void split_entries(int ks, unsigned steps, LA la, LB lb, bool real, const bool (&fma)[2], z2 (&v)[2],
                                              int (&ex)[2]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, c = 2 * (lane & 3);
    if (!__any_sync(0xffffffffu, fma[0] | fma[1])) return;
    z2 r[2] = {zmk(0.0, 0.0), zmk(0.0, 0.0)};
#pragma unroll 1
    for (int s = 0; s < ks; ++s) {
        if (!(steps >> s & 1u)) continue;
        if (real) {
#pragma unroll
            for (int k = 8 * s; k < 8 * s + 8; ++k) {
                const double x = la(g, k).x;
#pragma unroll
                for (int j = 0; j < 2; ++j) r[j].x = ::fma(x, lb(c + j, k).x, r[j].x);
            }
            continue;
        }
#pragma unroll 4
        for (int k = 8 * s; k < 8 * s + 8; ++k) {
            const z2 x = la(g, k);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const z2 y = lb(c + j, k);
                if constexpr (KIND == kConjA) zmac_ca(r[j], x, y);
                else if constexpr (KIND == kPlain) zmac(r[j], x, y);
                else zmac_cb(r[j], x, y);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        v[j].x = fma[j] ? r[j].x : v[j].x;
        v[j].y = fma[j] ? r[j].y : v[j].y;
        ex[j] = fma[j] ? 2100 : ex[j];
    }
}

// Grids of a product for split_guard: the exponents of a lane's two terms of K-step s.
struct SplitGrid {          // rows and columns on their own
    int ea, eb;
    __device__ __forceinline__ void operator()(int, z2, z2, int (&ga)[2], int (&gb)[2]) const {
        ga[0] = ga[1] = ea;
        gb[0] = gb[1] = eb;
    }
};
struct SplitGridJoint {     // rows of exponent sum ea on the terms' own
    int ea;
    __device__ __forceinline__ void operator()(int, z2 b0, z2 b1, int (&ga)[2], int (&gb)[2]) const {
        unsigned m0, m1;
        split_joint_exp(b0, b1, m0, m1);
        ga[0] = ea - (gb[0] = split_exp(m0));
        ga[1] = ea - (gb[1] = split_exp(m1));
    }
};

// Which of a lane's entries with small parts (bits of split_small) to form by FMAs.
// For all lanes of a warp.  Returns the K-steps (bits, the same in all lanes) that
// have a nonzero product for such an entry: blocks of triangular and banded operands
// have them in few.
template <class LA, class LB, class GRID>
__device__ __forceinline__ unsigned split_guard(int ks, LA la, LB lb, GRID grid, const unsigned (&small)[2], bool (&need)[2]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    SplitSeen seen;
    unsigned steps = 0;
    const unsigned mine = (small[0] ? 3u : 0u) | (small[1] ? 12u : 0u);     // (both parts of an entry are formed)
#pragma unroll 1
    for (int s = 0; s < ks; ++s) {
        SplitSeen now;
        z2 a[2], b[2];
        int ea[2], eb[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a[u] = la(g, 8 * s + 2 * t + u);
            b[u] = lb(g, 8 * s + 2 * t + u);
        }
        grid(s, b[0], b[1], ea, eb);
#pragma unroll
        for (int u = 0; u < 2; ++u) now.term(a[u], ea[u], b[u], eb[u]);
        seen.nz |= now.nz;
        seen.big |= now.big;
        if (__any_sync(0xffffffffu, (now.nz & mine) != 0u)) steps |= 1u << s;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) need[j] = (small[j] & ((seen.nz & ~seen.big) >> (2 * j))) != 0u;
    return steps;
}

// The imaginary part of an operand as bits, 0: none.
__device__ __forceinline__ unsigned im_bits(z2 z) { return (unsigned)__double2hiint(z.y) << 1; }

// Are the warp's operands, of whose bits im is the OR, all real?
__device__ __forceinline__ bool split_real(unsigned im) { return !__any_sync(0xffffffffu, im != 0u); }

// Has any lane a result that split_small tells of, among those that the caller uses?
template <int KS>
__device__ __forceinline__ bool split_any_small(SplitUse use, bool real, const z2 (&v)[2]) {
    constexpr unsigned one = 1023 + (KS > 8 ? 53 : 54), mod = (one - kSplitMod) << 20, part = (one - kSplitPart) << 20;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    bool any = false;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const unsigned x = mag_hi(v[j].x), y = mag_hi(v[j].y);
        const unsigned p = use(g, 2 * t + j);
        any |= (max(x, y) < mod || min(x, real || p == 1u ? x : y) < part) && p != 0u;
    }
    return any;
}

// small[j]: the parts of the lane's result v[j] that may have lost bits.
template <int KS>
__device__ __forceinline__ bool split_smalls(SplitUse use, bool real, const z2 (&v)[2], unsigned (&small)[2]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < 2; ++j) small[j] = split_small<KS>(v[j]) & use(g, 2 * t + j) & (real ? 1u : 3u);
    return __any_sync(0xffffffffu, (small[0] | small[1]) != 0u);
}

// The uncommon cases of a product, out of line so that they cost the kernels no
// registers: la, lb and grid are taken by value and capture no references.  They
// are called by whole warps and end converged, as the callers go on to warp-wide
// instructions.

// Has a product with small results one to form by FMAs in any lane?
template <int KS, class LA, class LB, class GRID>
__device__ __noinline__ bool split_look(int ks, LA la, LB lb, GRID grid, SplitUse use, bool real, z2 v0, z2 v1) {
    const z2 v[2] = {v0, v1};
    unsigned small[2];
    if (!split_smalls<KS>(use, real, v, small)) return false;
    bool need[2];
    split_guard(ks, la, lb, grid, small, need);
    return __any_sync(0xffffffffu, need[0] | need[1]);
}

// Results v, e of a tile after its entries with bad[j], small results that need it
// and exponents below the normal range.
struct SplitOut {
    z2 v[2];
    int e[2];
};
template <SplitKind KIND, int KS, class LA, class LB, class GRID>
__device__ __noinline__ SplitOut split_slow(int ks, LA la, LB lb, GRID grid, SplitUse use, bool real, bool bad0, bool bad1, SplitOut o) {
    const bool bad[2] = {bad0, bad1};
    bool need[2] = {false, false};
    unsigned small[2];
    unsigned steps = 0;
    if (split_smalls<KS>(use, real, o.v, small)) steps = split_guard(ks, la, lb, grid, small, need);
    const bool any_bad = __any_sync(0xffffffffu, bad0 | bad1);
    if (any_bad) steps = 0xffffffffu;       // (zeros times infinity or NaN count)
    // each entry decides for itself, so that it does not depend on which
    // columns share its tile
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        need[j] = need[j] || bad[j];
        if (!need[j] && o.e[j] < kSplitSumTiny) {
            // two exact factors down to the last, which rounds into the subnormal range
            const double s0 = split_scale(2100 - 950), s1 = split_scale(o.e[j] + 950);
            o.v[j].x = o.v[j].x * s0 * s1;
            o.v[j].y = o.v[j].y * s0 * s1;
            o.e[j] = 2100;
        }
    }
    split_entries<KIND>(ks, steps, la, lb, real && !any_bad, need, o.v, o.e);
    __syncwarp();
    return o;
}

// split_look for results v of operands in the split's range.
template <int KS, class LA, class LB, class GRID>
__device__ __forceinline__ bool split_needs(int ks, LA la, LB lb, SplitUse use, unsigned im, GRID grid, const z2 (&v)[2]) {
    const bool real = split_real(im);
    return __any_sync(0xffffffffu, split_any_small<KS>(use, real, v)) && split_look<KS>(ks, la, lb, grid, use, real, v[0], v[1]);
}
// ... with the FMAs.
template <SplitKind KIND, int KS, class LA, class LB, class GRID>
__device__ __forceinline__ void split_recheck(int ks, LA la, LB lb, SplitUse use, unsigned im, GRID grid, z2 (&v)[2], int (&ex)[2]) {
    const bool real = split_real(im);
    if (!__any_sync(0xffffffffu, split_any_small<KS>(use, real, v))) return;
    const SplitOut o = split_slow<KIND, KS>(ks, la, lb, grid, use, real, false, false, SplitOut{{v[0], v[1]}, {ex[0], ex[1]}});
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        v[j] = o.v[j];
        ex[j] = o.e[j];
    }
}

template <SplitKind KIND, bool kJoint, int KS, class LA, class LB>
__device__ __forceinline__ void split_tile(int ks, LA la, LB lb, SplitUse use, bool same, z2 (&v)[2], int (&e)[2]) {
    constexpr unsigned kAll = 0xffffffffu;
    // up to two K-steps the lane keeps its operands in registers between the
    // pass for the exponents and the products; beyond, it loads them again
    constexpr bool kKeep = KS <= 2;
    constexpr int NK = kKeep ? KS : 1;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if constexpr (KS == 1) ks = 1;
    z2 a[NK][2], b[NK][2];
    int ea = 0, eb = 0;
    unsigned m0[NK] = {}, m1[NK] = {};
    bool rbad = false, cbad = false;
    auto load = [&](int s, int i) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a[i][u] = la(g, 8 * s + 2 * t + u);
            b[i][u] = lb(g, 8 * s + 2 * t + u);
        }
    };
    if constexpr (kKeep) {
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            a[s][0] = a[s][1] = b[s][0] = b[s][1] = zmk(0.0, 0.0);
            if (s < ks) load(s, s);     // (the operands end with K-step ks - 1)
        }
    }
    SplitJoint jt;
    unsigned ma = 0, mb = 0, im = 0;
    auto exps = [&](int i) {
        im |= im_bits(a[i][0]) | im_bits(a[i][1]) | im_bits(b[i][0]) | im_bits(b[i][1]);
        if constexpr (kJoint) {
            split_joint_exp(b[i][0], b[i][1], m0[i], m1[i]);
            jt.term(split_mag(a[i][0]), m0[i]);
            jt.term(split_mag(a[i][1]), m1[i]);
        } else {
            ma = max(ma, max(split_mag(a[i][0]), split_mag(a[i][1])));
            mb = max(mb, max(split_mag(b[i][0]), split_mag(b[i][1])));
        }
    };
    if constexpr (kKeep) {
#pragma unroll
        for (int s = 0; s < KS; ++s)
            if (s < ks) exps(s);
    } else {
        for (int s = 0; s < ks; ++s) {
            load(s, 0);
            exps(0);
        }
    }
    if constexpr (kJoint) {
        rbad = jt.finish();
        ea = jt.ea;
    } else {
        ma = split_max4(ma);
        mb = split_max4(mb);
        rbad = split_unsafe(ma);
        cbad = split_unsafe(mb);
        ea = split_exp(ma);
        eb = split_exp(mb);
    }
    SplitCut ca, cb;
    SplitAcc acc;
    int sum[4][kSplitDigits];
    split_start(acc, KS == 1 ? kSplitStart : 0.f);
    if constexpr (KS > 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int d = 0; d < kSplitDigits; ++d) sum[j][d] = 0;
    }
    auto step = [&](int i) {
        if constexpr (kJoint) {
            // b is cut on the grid of c_k, a on that of 2^(ea - c_k)
            const int c0 = split_exp(m0[i]), c1 = split_exp(m1[i]);
            split_cut(ca, a[i][0], a[i][1], ea - c0, ea - c1);
            split_cut(cb, b[i][0], b[i][1], c0, c1);
        } else {
            split_cut(ca, a[i][0], a[i][1], ea, ea);
            if (same) cb = ca;
            else split_cut(cb, b[i][0], b[i][1], eb, eb);
        }
        split_mma<KIND>(ca, cb, acc);
    };
    if constexpr (kKeep) {
#pragma unroll
        for (int s = 0; s < KS; ++s)
            if (s < ks) step(s);
    } else {
#pragma unroll 1
        for (int s = 0; s < ks; ++s) {
            load(s, 0);
            if constexpr (kJoint) split_joint_exp(b[0][0], b[0][1], m0[0], m1[0]);
            step(0);
            if constexpr (KS > 4) {
                if ((s & 3) == 3) {     // 64 terms: what FP32 holds exactly
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int d = 0; d < kSplitDigits; ++d) sum[j][d] += __float2int_rn(acc[d][j]);
                    split_start(acc, 0.f);
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int d = 0; d < kSplitDigits; ++d) {
            if constexpr (KS == 1) sum[j][d] = __float_as_int(acc[d][j]);
            else if constexpr (KS <= 4) sum[j][d] = __float2int_rn(acc[d][j]);
            else sum[j][d] += __float2int_rn(acc[d][j]);
        }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        v[j] = zmk(split_value<KS>(sum[j]), split_value<KS>(sum[j + 2]));
        e[j] = ea + (kJoint ? 0 : __shfl_sync(kAll, eb, 8 * t + 4 * j)) + (KS > 8 ? 1 : 0);
    }
    const bool real = split_real(im);
    if (__any_sync(kAll, rbad || cbad || split_any_small<KS>(use, real, v) || min(e[0], e[1]) < kSplitSumTiny)) {
        bool bad[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int col_bad = __shfl_sync(kAll, (int)cbad, 8 * t + 4 * j);     // (for all lanes)
            bad[j] = rbad | (col_bad != 0);
        }
        SplitOut o = {{v[0], v[1]}, {e[0], e[1]}};
        if constexpr (kJoint) o = split_slow<KIND, KS>(ks, la, lb, SplitGridJoint{ea}, use, real, bad[0], bad[1], o);
        else o = split_slow<KIND, KS>(ks, la, lb, SplitGrid{ea, eb}, use, real, bad[0], bad[1], o);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            v[j] = o.v[j];
            e[j] = o.e[j];
        }
    }
}

// split_tile for operands that are on their grids already: v[j] in units of
// 2^(Ea + Eb - 54), without a look at small results.
template <SplitKind KIND, int KS, class LA, class LB>
__device__ __forceinline__ void split_tile_on(int ks, LA la, LB lb, bool same, z2 (&v)[2]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    SplitCut ca, cb;
    SplitAcc acc;
    int sum[4][kSplitDigits];
    split_start(acc, 0.f);
    if constexpr (KS > 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int d = 0; d < kSplitDigits; ++d) sum[j][d] = 0;
    }
#pragma unroll 1
    for (int s = 0; s < ks; ++s) {
        split_cut_on(ca, la(g, 8 * s + 2 * t), la(g, 8 * s + 2 * t + 1));
        if (same) cb = ca;
        else split_cut_on(cb, lb(g, 8 * s + 2 * t), lb(g, 8 * s + 2 * t + 1));
        split_mma<KIND>(ca, cb, acc);
        if constexpr (KS > 4) {
            if ((s & 3) == 3) {     // 64 terms: what FP32 holds exactly
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int d = 0; d < kSplitDigits; ++d) sum[j][d] += __float2int_rn(acc[d][j]);
                split_start(acc, 0.f);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int d = 0; d < kSplitDigits; ++d) {
            if constexpr (KS <= 4) sum[j][d] = __float2int_rn(acc[d][j]);
            else sum[j][d] += __float2int_rn(acc[d][j]);
        }
#pragma unroll
    for (int j = 0; j < 2; ++j) v[j] = zmk(split_value<(KS > 2 ? KS : 2)>(sum[j]), split_value<(KS > 2 ? KS : 2)>(sum[j + 2]));
}

}  // namespace crs
