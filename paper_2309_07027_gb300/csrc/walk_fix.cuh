// FP64-class walks in 64-bit fixed point on the integer pipes.
//
// Why: one FP64 instruction of a warp holds its scheduler's FP64 pipe for 64
// cycles on this part (2 lanes per SM and clock), a 32 x 32 -> 64 bit integer
// multiply-add (IMAD.WIDE) the FMA-heavy pipe for 4.  A complex product costs
// 4 FP64 instructions (256 cycles) or, on two-limb 62-bit mantissas, 12
// IMAD.WIDE (48 cycles) with the remaining integer work on the ALU beside
// them -- and the mantissas are 8 bits longer than a double's.
//
// Numbers.
//   * Column sums are exact.  Pack scales column j by 2^(63 - e_j), 2^e_j >
//     sum_rows M (|Re a| + |Im a|) (1 + 2^-20), and rounds every entry once
//     to an integer; c0 and the rows 2a are integers modulo 2^64, and the
//     sums |Re c| + |Im c| < 2^63 (1 - 2^-21), so the walk's 64-bit additions
//     give c0 - sum_j Delta_j 2a_j of the rounded matrix without any drift,
//     whatever the chunk length.
//   * A product operand is (h, l), value h 2^32 + l with l a signed 32-bit
//     limb.  A product keeps the high 64 of its 128 bits: hh + cross / 2^32,
//     the two cross terms summed in 64 bits and rounded, the low x low term
//     (below one unit of the result, zero mean) left out.  Operands are kept
//     normalised (larger component in [2^61, 2^62)) with an integer exponent
//     beside them: a normalised operand loses about 2^-57 per product, where
//     a double loses 2^-53.
//   * Bounds.  |h| <= 2^30 for normalised operands; for column sums
//     |h_re| + |h_im| <= 2^31 (1 - 2^-21) + 1; |l| <= 2^31.  Every cross sum
//     stays below 2^63 in magnitude (four terms of at most 2^61, or two of
//     2^61 and two that add up to less than 2^62), every high sum below 2^62.
//     Only high limbs are negated (a low limb of -2^31 has no negative).
//   * What this loses by itself, and what is done about it: a pair of column
//     sums is multiplied before it is normalised, so sums that cancel lose
//     their bits against the bounds (fix_product<1> and suffix_chains<1>
//     normalise the sums first, where it matters); both parts of a column
//     share one scale (columns whose parts' bounds differ by more than 8 get a
//     scale per part, and their jobs' addends are formed in double).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "bs_job.h"
#include "gray.h"
#include "walk.cuh"

namespace bs {

// A packed entry: a complex 64-bit integer.
struct __align__(16) zfix {
    long long re, im;
};

// Product operand: two signed limbs per component.
struct zlimb {
    int rl, rh, il, ih;
};

// Raw product: 64-bit components.
struct zraw {
    unsigned long long re, im;
};

// Limbs of a 64-bit value.
__device__ __forceinline__ zlimb limbs_of(const zraw& v) {
    zlimb o;
    o.rl = (int)(uint32_t)v.re;
    o.rh = (int)((uint32_t)(v.re >> 32) + ((uint32_t)v.re >> 31));
    o.il = (int)(uint32_t)v.im;
    o.ih = (int)((uint32_t)(v.im >> 32) + ((uint32_t)v.im >> 31));
    return o;
}

__device__ __forceinline__ zraw raw_of(const zlimb& v) {
    return zraw{((unsigned long long)(uint32_t)v.rh << 32) + (unsigned long long)(long long)v.rl,
                ((unsigned long long)(uint32_t)v.ih << 32) + (unsigned long long)(long long)v.il};
}

// high + cross / 2^32, rounded down.
__device__ __forceinline__ long long fix_combine(long long high, long long cross) { return high + (cross >> 32); }

__device__ __forceinline__ long long mul_wide(int a, int b) {
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}

// c + a b in one IMAD.WIDE (the compiler fuses this form; from mad.wide it
// makes a product and a 64-bit addition).
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return c + mul_wide(a, b); }

// z + a b / 2^64 (ADD = 1) or a b / 2^64.
template <int ROUND, int ADD>
__device__ __forceinline__ zraw fix_cmul_add(const zraw& z, const zlimb& a, const zlimb& b) {
    constexpr long long half = ROUND ? 0x80000000ll : 0ll;
    const long long x = mad_wide(a.rl, b.rh, mad_wide(a.rh, b.rl, half)) - mad_wide(a.il, b.ih, mul_wide(a.ih, b.il));
    long long y = mad_wide(a.rl, b.ih, mad_wide(a.rh, b.il, half));
    y = mad_wide(a.il, b.rh, mad_wide(a.ih, b.rl, y));
    const long long p = (ADD ? mad_wide(a.rh, b.rh, (long long)z.re) : mul_wide(a.rh, b.rh)) - mul_wide(a.ih, b.ih);
    const long long q = mad_wide(a.ih, b.rh, ADD ? mad_wide(a.rh, b.ih, (long long)z.im) : mul_wide(a.rh, b.ih));
    return zraw{(unsigned long long)fix_combine(p, x), (unsigned long long)fix_combine(q, y)};
}
template <int ROUND = 1>
__device__ __forceinline__ zraw fix_cmul(const zlimb& a, const zlimb& b) {
    return fix_cmul_add<ROUND, 0>(zraw{0ull, 0ull}, a, b);
}

// The real (part = 0) or imaginary (part = 1) component of fix_cmul(a, b).
__device__ __forceinline__ long long fix_cmul_part(const zlimb& a, const zlimb& b, int part) {
    const int uh = part ? b.ih : b.rh, ul = part ? b.il : b.rl;   // times a's real part
    const int vh = part ? b.rh : b.ih, vl = part ? b.rl : b.il;   // times +-a's imaginary part
    const int sah = part ? a.ih : -a.ih, svh = part ? vh : -vh;
    const long long x = mad_wide(a.rl, uh, mad_wide(a.rh, ul, 0x80000000ll)) + mad_wide(a.il, svh, mul_wide(sah, vl));
    const long long p = mad_wide(sah, vh, mul_wide(a.rh, uh));
    return fix_combine(p, x);
}

// Shift that brings the larger component of v (|v| < 2^62) into
// [2^61, 2^62); at most 30 (a value below 2^32 comes out shifted by 30).
__device__ __forceinline__ int fix_norm_shift(const zraw& v) {
    const int rh = (int)(v.re >> 32), ih = (int)(v.im >> 32);
    return __clz(abs(rh) | abs(ih)) - 2;
}

// Limbs of v 2^s.
__device__ __forceinline__ zlimb fix_shift(const zraw& v, int s) {
    const uint32_t rl = (uint32_t)v.re, rh = (uint32_t)(v.re >> 32);
    const uint32_t il = (uint32_t)v.im, ih = (uint32_t)(v.im >> 32);
    zlimb o;
    const uint32_t a = rl << s, b = il << s;
    o.rl = (int)a;
    o.rh = (int)(__funnelshift_l(rl, rh, s) + (a >> 31));
    o.il = (int)b;
    o.ih = (int)(__funnelshift_l(il, ih, s) + (b >> 31));
    return o;
}

__device__ __forceinline__ zlimb fix_normalise(const zraw& v, int& e) {
    const int s = fix_norm_shift(v);
    e -= s;
    return fix_shift(v, s);
}

// 2^(e + BS_FIX_BIAS) w for w a nonzero double of magnitude 1 to 2^64, by the
// exponent field; zero where that is below 2^-1000 (an addend 2^-1450 below the
// column bounds, or the exponent of a product that is zero).
__device__ __forceinline__ double scale_pow2(double w, int e) {
    return e < -1000 - BS_FIX_BIAS ? 0.0 : __hiloint2double(__double2hiint(w) + ((e + BS_FIX_BIAS) << 20), __double2loint(w));
}

// v 2^e as a double (e: a constant that keeps the result normal).
__device__ __forceinline__ double scale_int(long long v, int e) {
    const double x = (double)v;
    return v == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// Column sums of the decoded state, c0 - sum_j Delta_j 2a_j, for N columns
// from column cbase on.
template <int N, int KP>
__device__ __forceinline__ void fix_seed(zraw (&c)[N], const bs_gray& g, const zfix* __restrict__ c0, int nbin,
                                         int nrows) {
    const zfix* a2 = c0 + KP;
#pragma unroll
    for (int t = 0; t < N; ++t) {
        const zfix v = c0[t];
        c[t].re = (unsigned long long)v.re;
        c[t].im = (unsigned long long)v.im;
    }
    uint64_t bits = g.dbin;
    while (bits) {
        const int j = bs_ctz64(bits);
        bits &= bits - 1;
        const zfix* row = a2 + (size_t)j * KP;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const zfix v = row[t];
            c[t].re -= (unsigned long long)v.re;
            c[t].im -= (unsigned long long)v.im;
        }
    }
    for (int j = nbin; j < nrows; ++j) {
        const int d = g.del[j];
        if (d == 0) continue;
        const zfix* row = a2 + (size_t)j * KP;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const zfix v = row[t];
            c[t].re -= (unsigned long long)v.re * (unsigned long long)d;
            c[t].im -= (unsigned long long)v.im * (unsigned long long)d;
        }
    }
}

// One digit move of N column sums: c -= row (neg = 1) or c += row.  The
// whole warp calls it; nearly always its lanes move the same way (they walk
// aligned chunks), and the two uniform branches spend no instruction on the
// sign.
template <int N>
__device__ __forceinline__ void fix_update(zraw (&c)[N], const zfix* __restrict__ row, uint32_t neg) {
    const longlong2* p = reinterpret_cast<const longlong2*>(row);
    const unsigned down = __ballot_sync(0xffffffffu, neg != 0u);
    if (down == 0u) {
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const longlong2 v = __ldg(p + t);
            c[t].re += (unsigned long long)v.x;
            c[t].im += (unsigned long long)v.y;
        }
    } else if (down == 0xffffffffu) {
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const longlong2 v = __ldg(p + t);
            c[t].re -= (unsigned long long)v.x;
            c[t].im -= (unsigned long long)v.y;
        }
    } else {
        const long long m = -(long long)neg;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const longlong2 v = __ldg(p + t);
            c[t].re += (unsigned long long)((v.x ^ m) - m);
            c[t].im += (unsigned long long)((v.y ^ m) - m);
        }
    }
}

// A leaf of a lane's product, as a raw value below 2^62 with exponent
// kLeafExp against the column bounds: the product of a pair of column sums,
// or half an odd last one (a column sum may reach 2^63).
constexpr int kLeafExp = -62;
template <int N>
__device__ __forceinline__ zraw fix_leaf(const zraw (&c)[N], int j) {
    if (2 * j + 1 < N) return fix_cmul<0>(limbs_of(c[2 * j]), limbs_of(c[2 * j + 1]));
    return zraw{(unsigned long long)((long long)c[2 * j].re >> 1), (unsigned long long)((long long)c[2 * j].im >> 1)};
}

// A column sum (below 2^63) normalised, and its shift (-1..60).
__device__ __forceinline__ zlimb norm_column(const zraw& v, int& k) {
    zraw n = v;
    k = fix_norm_shift(v);
    if (k < 0) n = zraw{(unsigned long long)((long long)v.re >> 1), (unsigned long long)((long long)v.im >> 1)};
    if (k > 0) n = zraw{v.re << k, v.im << k};
    if (k < 29) return limbs_of(n);
    const int k2 = fix_norm_shift(n);
    k += k2;
    return fix_shift(n, k2);
}

// Product of a lane's N column sums as a normalised operand, and its exponent
// against the column bounds: leaves (independent of one another), then their
// running product, normalised after every leaf.  A typical column sum is
// 2^59.5 (its bound 2^63 is a sum of moduli, it is a root of squares), a pair
// 2^55, and a pair times a normalised operand 2^52.5, so a pair costs about
// 2^-54 in relative rounding, where two products of doubles cost 2^-53.  Sums
// that cancel lose more: smax is the largest of the normalising shifts, so the
// relative error is a few 2^(smax - 61).  NORM: leaves of normalised column
// sums, 2^-56 at most for any sums.  A product that is zero (or lost: smax
// shows it) has a last shift of 29 or 30 and gets no weight.
template <int NORM, int N>
__device__ __forceinline__ zlimb fix_product(const zraw (&c)[N], int& e, int& smax) {
    zlimb p;
    int s = 0;
    smax = 0;
    e = -64;
#pragma unroll
    for (int j = 0; 2 * j < N; ++j) {
        zraw leaf;
        e += 64 + kLeafExp;
        if (NORM) {
            int ka, kb = 1;
            const zlimb a = norm_column(c[2 * j], ka);
            leaf = 2 * j + 1 < N ? fix_cmul<0>(a, norm_column(c[2 * j + 1], kb)) : raw_of(a);
            e -= ka + kb;
        } else {
            leaf = fix_leaf(c, j);
        }
        const zraw r = j ? fix_cmul(p, limbs_of(leaf)) : leaf;
        s = fix_norm_shift(r);
        smax = max(smax, s);
        e -= s;
        p = fix_shift(r, s);
    }
    if (s >= 29) e -= 1 << 14;
    return p;
}

// Exact column sums in double, in units of kDblUnit bits below each column's
// bound: 48 columns at their bounds stay in range, as do products 2^-1800 below
// them.
constexpr int kDblUnit = 18;
// A column sum in those units, with parts of their own scales; x: the column's
// colexp.
__device__ __forceinline__ cx<double> split_column(const zraw& c, int x) {
    const int d = BS_COLEXP_D(x);
    return cx<double>{scale_int((long long)c.re, kDblUnit - 63 + min(d, 0)),
                      scale_int((long long)c.im, kDblUnit - 63 - max(d, 0))};
}
// colexp of column t of a lane's columns, which begin with column `first` (a
// pad column: parts of one scale).
__device__ __forceinline__ int lane_colexp(const bs_job& jb, const int* __restrict__ radix, int first, int t) {
    return first + t < jb.K ? radix[BS_META_COLEXP(jb) - jb.meta_off + first + t] : BS_COLEXP(0, 0);
}

__device__ __forceinline__ zlimb shfl_xor_zlimb(const zlimb& v, int mask) {
    zlimb o;
    o.rh = __shfl_xor_sync(0xffffffffu, v.rh, mask);
    o.rl = __shfl_xor_sync(0xffffffffu, v.rl, mask);
    o.ih = __shfl_xor_sync(0xffffffffu, v.ih, mask);
    o.il = __shfl_xor_sync(0xffffffffu, v.il, mask);
    return o;
}

// ---------------------------------------------------------------- one task: permanent
// Two lanes share one chunk: lane 2p + h owns the columns [h HX, h HX + HX),
// HX = ceil(K / 2) (an odd K leaves lane h = 1 a pad column that is exactly
// 1), so the column sums take 4 HX registers and 4 warps per scheduler fit
// up to K = 32.  Per addend each lane forms the product of its columns, the
// lanes swap them (5 shuffles), and lane h = 0 forms the real, h = 1 the
// imaginary part of the product of the two: half a complex product each.
// That part is converted to double and added with the weight 2^e W (one
// conversion and one FMA per lane on the FP64 pipe, which nothing else here
// uses), in runs of FOLD folded into a double-double.  A task's 32 chunks
// are walked by two warps, 16 each (`half_task`); a warp's sum ends in its
// lane 0.  Every lane walks the warp's longest chunk, with weight 0 after its
// own end, so that the warp stays converged.
//
// Cancelling column sums.  An addend is formed again from normalised sums
// (fix_product<1>) when a normalising shift exceeds s0 = 12 + log2 K (its
// relative error is then above 2^(s0 - 61)) and that error is more than
// 2^(s0 - 65) of the lane's largest addend so far, or when a product that is
// not zero is lost altogether.  So the error of an addend stays below K 2^-49 of
// itself or K 2^-53 of the largest one, per pair of columns, for any matrix (two
// blocks [[B, B], [B + 1, -B]], B = 3^25: 2.8e-7, or all of it with the blocks'
// columns in different pairs, without this).  Haar matrices need it for one
// addend of a warp in 300 at 30 columns: 28.6 -> 29.1 ms, 23 columns 214 -> 221
// us (at s0 - 1 29.4 ms and 223 us; formed in double instead, 6 FP64
// instructions per column, the same for Haar matrices, but 1.9 ms instead of
// 0.9 for 24 columns of roots of unity, whose sums cancel more often).
//
// 30 x 30 permanent (2^29 addends): 165 ms in double (FP64 pipe 94 % busy),
// 36.2 ms with one lane per chunk (255 registers, 2 warps per scheduler), 29.1
// ms here; 72 cycles per warp, column and addend, of which the 12 integer
// products hold the FMA-heavy pipe 52 (78 % busy with what else runs there) and
// 26 other integer instructions take the rest.  Relative error (23 x 23, Haar): 6.8e-15, in
// double 2.7e-14.
template <int KB, int HX>
__device__ void walk_task_perm_fix(const bs_job& jb, const zfix* __restrict__ data, const int* __restrict__ radix,
                                   uint32_t local, int half_task, int lane, ddv& sum, ddv& im) {
    constexpr uint32_t FOLD = 64;
    constexpr int KP = KB;  // = BS_ROW_STRIDE(K) for every K of the bucket
    const int half = lane & 1;
    const zfix* c0 = data + jb.data_off + half * HX;
    const zfix* a2 = c0 + KP;
    // exponent of a product of both lanes' operands: the last product's 64,
    // and 1 for the pad column (2^62 stands for 1, bound 2)
    const int e_pair = 64 + (jb.K & 1);
    sum = im = ddv{0.0, 0.0};
    const uint64_t i0_own = ((uint64_t)local * 32u + (uint64_t)(16 * half_task + (lane >> 1))) << jb.log2L;
    const bool has = i0_own < jb.C;
    const uint64_t i0 = has ? i0_own : 0ull;
    uint32_t len = 0;
    if (has) {
        const uint64_t rem = jb.C - i0;
        len = (uint32_t)(rem < (1ull << jb.log2L) ? rem : (1ull << jb.log2L));
    }
    const uint32_t steps = __reduce_max_sync(0xffffffffu, len);
    if (steps == 0u) return;
    bs_gray g;
    ChunkStepper st;
    st.init(g, i0, jb.nbin, jb.nrows, radix, reinterpret_cast<const uint64_t*>(radix + (BS_META_BINOM(jb) - jb.meta_off)));
    zraw c[HX];
    fix_seed<HX, KP>(c, g, c0, jb.nbin, jb.nrows);
    double ws = signed_weight<double>(g.w, g.parity);
    double acc = 0.0;
    int emax = -(1 << 28);  // largest exponent of an addend so far
    const int s0 = 12 + (31 - __clz(jb.K));
    for (uint32_t s = 0; s < steps; ++s) {
        int e, smax;
        zlimb p = fix_product<0, HX>(c, e, smax);
        long long v = fix_cmul_part(p, shfl_xor_zlimb(p, 1), half);
        e += __shfl_xor_sync(0xffffffffu, e, 1) + e_pair;
        double f = s < len ? scale_pow2(ws, e) : 0.0;
        e += __double2hiint(ws) >> 20 & 0x7ff;  // (for comparison, with the weight's exponent)
        emax = max(emax, e);
        if (__any_sync(0xffffffffu, smax > s0)) {
            bool redo = s < len && smax > s0 && (smax >= 28 || e - emax + smax > s0 - 4);
            if (__any_sync(0xffffffffu, redo)) {
#pragma unroll
                for (int t = 0; t < HX; ++t) redo = redo && (c[t].re | c[t].im) != 0ull;
                if (__any_sync(0xffffffffu, redo)) {
                    p = fix_product<1, HX>(c, e, smax);
                    v = fix_cmul_part(p, shfl_xor_zlimb(p, 1), half);
                    e += __shfl_xor_sync(0xffffffffu, e, 1) + e_pair;
                    f = s < len ? scale_pow2(ws, e) : 0.0;
                    emax = max(emax, e + (__double2hiint(ws) >> 20 & 0x7ff));
                }
            }
        }
        acc = bfma(f, (double)v, acc);
        if (((s + 1u) & (FOLD - 1u)) == 0u) {
            sum = dd_add_d(sum, acc);
            acc = 0.0;
        }
        if (s + 1 == steps) break;
        uint32_t neg = 0;
        int row = 0;  // a lane past its chunk moves on with weight 0
        if (s + 1 < len) {
            int wch;
            row = st.step(g, s, radix, &neg, &wch);
            ws = wch ? signed_weight<double>(g.w, g.parity) : flip_sign(ws);
        }
        fix_update<HX>(c, a2 + (size_t)row * KP, neg);
    }
    sum = dd_add_d(sum, acc);
    // over the 16 lanes of each part, then the imaginary part to lane 0
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) sum = dd_add_sum2(sum, shfl_down_dd(sum, off));
    im = shfl_down_dd(sum, 1);
}

// The same task with every addend in double from the exact sums: jobs with
// columns of very unequal parts, whose smaller parts the products above would
// round at the larger ones' scale (a 5 x 5 matrix with imaginary parts of 1e-9:
// 1.6e-10 of Im, here 1e-15).  Up to 6 FP64 instructions per column and addend,
// the pipe's time for a product of doubles.
template <int KB, int HX>
__device__ __noinline__ void walk_task_perm_dbl(const bs_job& jb, const zfix* __restrict__ data,
                                                const int* __restrict__ radix, uint32_t local, int half_task, int lane,
                                                ddv& sum, ddv& im) {
    const int half = lane & 1;
    const zfix* c0 = data + jb.data_off + half * HX;
    sum = im = ddv{0.0, 0.0};
    const uint64_t i0_own = ((uint64_t)local * 32u + (uint64_t)(16 * half_task + (lane >> 1))) << jb.log2L;
    const uint64_t i0 = i0_own < jb.C ? i0_own : 0ull;
    const uint64_t rem = i0_own < jb.C ? jb.C - i0_own : 0ull;
    const uint32_t len = (uint32_t)(rem < (1ull << jb.log2L) ? rem : (1ull << jb.log2L));
    const uint32_t steps = __reduce_max_sync(0xffffffffu, len);
    if (steps == 0u) return;
    bs_gray g;
    ChunkStepper st;
    st.init(g, i0, jb.nbin, jb.nrows, radix, reinterpret_cast<const uint64_t*>(radix + (BS_META_BINOM(jb) - jb.meta_off)));
    zraw c[HX];
    fix_seed<HX, KB>(c, g, c0, jb.nbin, jb.nrows);
    double ws = signed_weight<double>(g.w, g.parity), acc = 0.0;
    for (uint32_t s = 0; s < steps; ++s) {
        cx<double> x;
#pragma unroll
        for (int t = 0; t < HX; ++t) {
            const cx<double> v = split_column(c[t], lane_colexp(jb, radix, half * HX, t));
            x = t ? cmul(x, v) : v;
        }
        cx<double> y;
        y.re = __shfl_xor_sync(0xffffffffu, x.re, 1);
        y.im = __shfl_xor_sync(0xffffffffu, x.im, 1);
        const double w = s < len ? scale_pow2(ws, (jb.K & 1) - 2 * HX * kDblUnit) : 0.0;
        acc = bfma(w, half ? bfma(x.re, y.im, x.im * y.re) : bfma(x.re, y.re, -(x.im * y.im)), acc);
        if (((s + 1u) & 63u) == 0u) {
            sum = dd_add_d(sum, acc);
            acc = 0.0;
        }
        if (s + 1 == steps) break;
        uint32_t neg = 0;
        int row = 0;
        if (s + 1 < len) {
            int wch;
            row = st.step(g, s, radix, &neg, &wch);
            ws = wch ? signed_weight<double>(g.w, g.parity) : flip_sign(ws);
        }
        fix_update<HX>(c, c0 + (size_t)(1 + row) * KB, neg);
    }
    sum = dd_add_d(sum, acc);
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) sum = dd_add_sum2(sum, shfl_down_dd(sum, off));
    im = shfl_down_dd(sum, 1);
}

// ---------------------------------------------------------------- one task: minors
// v >> d, 0 <= d <= 63 (rounded down).
__device__ __forceinline__ zraw fix_shr(const zraw& v, int d) {
    return zraw{(unsigned long long)((long long)v.re >> d), (unsigned long long)((long long)v.im >> d)};
}

// Longest integer run of the minors, in addends (a power of two).
constexpr uint32_t kFixRun = 8;

// Shared memory of one warp of the minors kernel, HX columns per lane, NP =
// ceil(HX / 2) leaves: the integer sums [col][lane] (rows of 33, so that
// neighbouring columns of one lane fall into different banks when a run is
// flushed), the suffix products and the leaves [leaf][lane] (at the
// end of a run the units' exponents), the K
// double-double totals, plain-double sums, and a factor per chunk.
template <int G, int HX>
struct MinorsSmem {
    longlong2 acc[HX * 33];
    longlong2 leaf[((HX + 1) / 2) * 32];
    int4 pair[((HX + 1) / 2) * 32];
    double4 tot[G * HX];
    double2 run[G * HX];
    float2 est[G * HX];  // see minors_look (y: an integer)
    double fac[32 / G];
};

// Runs whose plain-double sum goes to the double-double totals at once.
constexpr uint32_t kFixFold = 16;

// How far a column's run sums v lie above the rounding of their unit: adds w
// (|Re v| + |Im v| - 2^kSumBits), w the unit's weight, to est.x, a float with
// exponent est.y (that of the largest w so far).  Sums that are zero do not count.  fac, ex: as in the flush.
constexpr int kSumBits = 45;
template <int N>
__device__ __forceinline__ float2 minors_look(float2 est, const longlong2* __restrict__ v, const int* __restrict__ ex,
                                              const double* __restrict__ fac, int G) {
    int ref = __float_as_int(est.y);
    auto pow2 = [](int e) { return __int_as_float((max(e, -126) + 127) << 23); };  // e <= 0
#pragma unroll 4
    for (int p = 0; p < N; ++p) {
        const int e = (__double2hiint(fac[p]) >> 20 & 0x7ff) + ex[4 * G * p], up = max(ref, e);
        if ((v[G * p].x | v[G * p].y) == 0ll) continue;
        const int hi = abs((int)(v[G * p].x >> 32)) + abs((int)(v[G * p].y >> 32)) - (1 << (kSumBits - 32));
        est.x = bfma(est.x, pow2(ref - up), pow2(e - up) * __int2float_rn(hi));
        ref = up;
    }
    est.y = __int_as_float(ref);
    return est;
}

// End of a run: lane t takes column t (and t + 32) and adds the integer sums
// of the lanes that own it, times their chunks' factors and their units
// 2^exp, to the column's plain-double sum, and clears the sums; with fold, the
// plain-double sum goes to the column's double-double total.
template <int G, int HX>
__device__ __forceinline__ void minors_flush_fix(MinorsSmem<G, HX>& sm, double f, int e_unit, const int (&em)[(HX + 1) / 2],
                                                 int lane, int K, bool fold, bool look) {
    if ((lane & (G - 1)) == 0) sm.fac[lane / G] = f;
#pragma unroll
    for (int j = 0; j < (HX + 1) / 2; ++j) sm.pair[j * 32 + lane].x = em[j] + e_unit;
    __syncwarp();
#pragma unroll 1
    for (int t = lane; t < K; t += 32) {
        const int q = t / HX, u = t - q * HX;
        longlong2* a = sm.acc + u * 33 + q;
        const int4* ex = sm.pair + (u >> 1) * 32 + q;
        if (look) sm.est[t] = minors_look<32 / G>(sm.est[t], a, &ex->x, sm.fac, G);
        double2 r = sm.run[t];
#pragma unroll 4
        for (int p = 0; p < 32 / G; ++p) {
            const longlong2 v = a[G * p];
            a[G * p] = make_longlong2(0, 0);
            const double w = scale_pow2(sm.fac[p], ex[G * p].x);
            r.x = bfma(w, (double)v.x, r.x);
            r.y = bfma(w, (double)v.y, r.y);
        }
        if (fold) {
            const double4 v = sm.tot[t];
            const ddv sr = dd_add_d(ddv{v.x, v.y}, r.x), si = dd_add_d(ddv{v.z, v.w}, r.y);
            sm.tot[t] = make_double4(sr.hi, sr.lo, si.hi, si.lo);
            r = make_double2(0.0, 0.0);
        }
        sm.run[t] = r;
    }
    __syncwarp();
}

// fix_normalise that also notes the largest shift.
__device__ __forceinline__ zlimb fix_normalise(const zraw& v, int& e, int& smax) {
    const int s = fix_norm_shift(v);
    smax = max(smax, s);
    e -= s;
    return fix_shift(v, s);
}

// Leaf j of the minors.  NORM: of normalised column sums, and their shifts in
// byte j of ls (plus kLeafBias); else fix_leaf.  Its exponent is leaf_exp.
constexpr int kLeafBias = 2;
template <int NORM, int HX>
__device__ __forceinline__ zraw minors_leaf(const zraw (&c)[HX], int j, uint32_t (&ls)[((HX + 1) / 2 + 3) / 4]) {
    if (!NORM) return fix_leaf(c, j);
    int ka, kb = 1;
    const zlimb a = norm_column(c[2 * j], ka);
    zraw r = raw_of(a);
    if (2 * j + 1 < HX) r = fix_cmul<0>(a, norm_column(c[2 * j + 1], kb));
    ls[j / 4] = (ls[j / 4] & ~(255u << (8 * (j % 4)))) | (uint32_t)(ka + kb + kLeafBias) << (8 * (j % 4));
    return r;
}
template <int HX>
__device__ __forceinline__ int leaf_exp(const uint32_t (&ls)[((HX + 1) / 2 + 3) / 4], int j) {
    return kLeafExp + kLeafBias - (int)(ls[j / 4] >> (8 * (j % 4)) & 255u);
}

// One step of a suffix chain: r (exponent e) is the product of the chain's
// leaves after leaf j; keeps it, normalised, as leaf j's suffix, and takes
// leaf j in.
template <int NORM, int HX>
__device__ __forceinline__ void suffix_step(const zraw (&c)[HX], uint32_t (&ls)[((HX + 1) / 2 + 3) / 4], int j, zraw& r, int& e, int& smax,
                                            int (&es)[(HX + 1) / 2], longlong2* __restrict__ sm_leaf,
                                            int4* __restrict__ sm_pair) {
    const zlimb sf = fix_normalise(r, e, smax);
    sm_leaf[j * 32] = *reinterpret_cast<const longlong2*>(&sf);
    es[j] = e;
    const zlimb d = limbs_of(minors_leaf<NORM>(c, j, ls));
    sm_pair[j * 32] = make_int4(d.rl, d.rh, d.il, d.ih);
    r = fix_cmul(sf, d);
    e += 64 + (NORM ? leaf_exp<HX>(ls, j) : kLeafExp);
}

// Both suffix chains of a lane's leaves, of NA = ceil(NP / 2) and the rest:
// the suffixes and leaves in shared memory, their exponents es, the chains'
// products qa, qb (exponents ea, eb).  smax: the largest normalising shift.
template <int NORM, int HX>
__device__ __forceinline__ void suffix_chains(const zraw (&c)[HX], uint32_t (&ls)[((HX + 1) / 2 + 3) / 4], zlimb& qa,
                                              zlimb& qb, int& ea, int& eb, int& smax, int (&es)[(HX + 1) / 2],
                                              longlong2* __restrict__ sm_leaf, int4* __restrict__ sm_pair) {
    constexpr int NP = (HX + 1) / 2, NA = (NP + 1) / 2, NB = NP - NA;
    zraw ra = minors_leaf<NORM>(c, NA - 1, ls), rb = {0ull, 0ull};
    ea = NORM ? leaf_exp<HX>(ls, NA - 1) : kLeafExp;
    if constexpr (NB > 0) rb = minors_leaf<NORM>(c, NP - 1, ls);
    eb = NORM ? leaf_exp<HX>(ls, NP - 1) : kLeafExp;
    smax = 0;
#pragma unroll
    for (int i = 1; i < NA; ++i) {
        suffix_step<NORM, HX>(c, ls, NA - 1 - i, ra, ea, smax, es, sm_leaf, sm_pair);
        if (i < NB) suffix_step<NORM, HX>(c, ls, NP - 1 - i, rb, eb, smax, es, sm_leaf, sm_pair);
    }
    qa = fix_normalise(ra, ea, smax);
    if constexpr (NB > 0) qb = fix_normalise(rb, eb, smax);
}

// One step of a prefix chain.  m_j = p S_j (p itself for the chain's last
// leaf), below 2^61; times the one column of the pair it is added to the
// other column's sum, whose unit 2^em follows the run's largest addend (that
// one comes to [2^60, 2^61): m_j is carried 4 times over, so that its shift
// is to the right); then p takes leaf j in.
template <int HX>
__device__ __forceinline__ void prefix_step(const zraw (&c)[HX], const uint32_t (&ls)[((HX + 1) / 2 + 3) / 4], int j, bool last, zlimb& p, int& e, int es, int& em,
                                            longlong2* __restrict__ sm_acc, const longlong2* __restrict__ sm_leaf,
                                            const int4* __restrict__ sm_pair) {
    zraw m;
    if (last) {
        m = fix_shr(raw_of(p), 1);
        es = e + 1;
    } else {
        const longlong2 v = sm_leaf[j * 32];
        m = fix_cmul<0>(p, *reinterpret_cast<const zlimb*>(&v));
        es += e + 64;
        const int4 d = sm_pair[j * 32];
        e += 64 + leaf_exp<HX>(ls, j);
        p = fix_normalise(fix_cmul(p, zlimb{d.x, d.y, d.z, d.w}), e);
    }
    const int sm = fix_norm_shift(m);
    const int up = max(em, sm < 29 ? es - min(sm - 1, 2) : -(1 << 20));  // (zero has no exponent)
    const int dl = min(up - em, 63);
    em = up;
    m = fix_shr(zraw{m.re << 2, m.im << 2}, (int)min((uint32_t)(up - es + 2), 63u));
    const longlong2 a = sm_acc[2 * j * 33];
    zraw z = fix_shr(zraw{(unsigned long long)a.x, (unsigned long long)a.y}, dl);
    if (2 * j + 1 < HX) {
        const zlimb ml = limbs_of(m);
        z = fix_cmul_add<0, 1>(z, ml, limbs_of(c[2 * j + 1]));
        sm_acc[2 * j * 33] = make_longlong2((long long)z.re, (long long)z.im);
        const longlong2 b = sm_acc[(2 * j + 1) * 33];
        z = fix_cmul_add<0, 1>(fix_shr(zraw{(unsigned long long)b.x, (unsigned long long)b.y}, dl), ml,
                               limbs_of(c[2 * j]));
        sm_acc[(2 * j + 1) * 33] = make_longlong2((long long)z.re, (long long)z.im);
    } else {  // no partner: m_j itself, in the same unit (m / 2)
        const zraw h = fix_shr(m, 1);
        sm_acc[2 * j * 33] = make_longlong2((long long)(z.re + h.re), (long long)(z.im + h.im));
    }
}

// The minors' addend of one chunk in double, from the exact column sums: for
// each of its columns a lane leaves w times the product of all other columns
// of its chunk in a slot (in units of kDblUnit bits below each column's
// bound).  All lanes of the warp call it.
template <int HX>
__device__ __forceinline__ double2* dbl_slot(longlong2* sm_leaf, int4* sm_pair, int t) {
    constexpr int NP = (HX + 1) / 2;
    return t < NP ? reinterpret_cast<double2*>(sm_leaf + t * 32) : reinterpret_cast<double2*>(sm_pair + (t - NP) * 32);
}
template <int G, int HX>
__device__ __forceinline__ void minors_addend_dbl(const zraw (&c)[HX], const bs_job& jb, const int* __restrict__ radix,
                                                  int first, double w, longlong2* sm_leaf, int4* sm_pair) {
    cx<double> x[HX];
#pragma unroll
    for (int t = 0; t < HX; ++t) x[t] = split_column(c[t], lane_colexp(jb, radix, first, t));
    auto swap = [](const cx<double>& v, int mask) {
        return cx<double>{__shfl_xor_sync(0xffffffffu, v.re, mask), __shfl_xor_sync(0xffffffffu, v.im, mask)};
    };
    cx<double> r = x[HX - 1];
#pragma unroll
    for (int t = HX - 2; t >= 0; --t) {
        *dbl_slot<HX>(sm_leaf, sm_pair, t) = make_double2(r.re, r.im);
        r = cmul(r, x[t]);
    }
    cx<double> p = swap(r, 1);
    if constexpr (G == 4) p = cmul(p, swap(cmul(r, p), 2));
    p.re *= w;
    p.im *= w;
#pragma unroll
    for (int t = 0; t < HX; ++t) {
        double2* slot = dbl_slot<HX>(sm_leaf, sm_pair, t);
        const cx<double> v = t + 1 < HX ? cmul(p, cx<double>{slot->x, slot->y}) : p;
        *slot = make_double2(v.re, v.im);
        if (t + 1 < HX) p = cmul(p, x[t]);
    }
}

// Lane t adds the lanes' double sums of column t (and t + 32) to its
// double-double total and clears them.
template <int G, int HX>
__device__ __forceinline__ void minors_flush_dbl(MinorsSmem<G, HX>& sm, int lane, int K) {
    __syncwarp();
#pragma unroll 1
    for (int t = lane; t < K; t += 32) {
        const int q = t / HX, u = t - q * HX;
        double2* a = reinterpret_cast<double2*>(sm.acc + u * 33 + q);
        const double4 v = sm.tot[t];
        ddv re = {v.x, v.y}, im = {v.z, v.w};
#pragma unroll 1
        for (int p = 0; p < 32 / G; ++p) {
            re = dd_add_d(re, a[G * p].x);
            im = dd_add_d(im, a[G * p].y);
            a[G * p] = make_double2(0.0, 0.0);
        }
        sm.tot[t] = make_double4(re.hi, re.lo, im.hi, im.lo);
    }
    __syncwarp();
}

// The whole task with the addends of minors_addend_dbl, summed per lane in
// double in runs of 64: tasks whose integer sums came too close to their
// units, and jobs with columns of very unequal parts.
template <int G, int KB, int HX>
__device__ __noinline__ void walk_task_minors_dbl(const bs_job& jb, const zfix* __restrict__ data,
                                                  const int* __restrict__ radix, uint32_t local, int lane,
                                                  MinorsSmem<G, HX>& sm) {
    const int q = lane & (G - 1), K = jb.K;
    const zfix* c0 = data + jb.data_off + q * HX;
    double2* acc = reinterpret_cast<double2*>(sm.acc + lane);
#pragma unroll
    for (int t = 0; t < HX; ++t) acc[t * 33] = make_double2(0.0, 0.0);
    for (int t = lane; t < K; t += 32) sm.tot[t] = make_double4(0.0, 0.0, 0.0, 0.0);
    for (int round = 0; round < G / 2; ++round) {
        const uint64_t i0_own = ((uint64_t)local * 16u + (uint64_t)(round * (32 / G) + lane / G)) << jb.log2L;
        const uint64_t i0 = i0_own < jb.C ? i0_own : 0ull;
        const uint64_t rem = i0_own < jb.C ? jb.C - i0_own : 0ull;
        const uint32_t len = (uint32_t)(rem < (1ull << jb.log2L) ? rem : (1ull << jb.log2L));
        const uint32_t steps = __reduce_max_sync(0xffffffffu, len);
        if (steps == 0u) break;
        bs_gray g;
        ChunkStepper st;
        st.init(g, i0, jb.nbin, jb.nrows, radix, reinterpret_cast<const uint64_t*>(radix + (BS_META_BINOM(jb) - jb.meta_off)));
        zraw c[HX];
        fix_seed<HX, KB>(c, g, c0, jb.nbin, jb.nrows);
        double ws = signed_weight<double>(g.w, g.parity);
        for (uint32_t s = 0; s < steps; ++s) {
            const double w = s < len ? scale_pow2(ws, (G * HX - K) - (G * HX - 1) * kDblUnit) : 0.0;
            minors_addend_dbl<G, HX>(c, jb, radix, q * HX, w, sm.leaf + lane, sm.pair + lane);
#pragma unroll
            for (int t = 0; t < HX; ++t) {
                const double2 v = *dbl_slot<HX>(sm.leaf + lane, sm.pair + lane, t);
                acc[t * 33].x += v.x;
                acc[t * 33].y += v.y;
            }
            if (((s + 1u) & 63u) == 0u || s + 1 == steps) minors_flush_dbl<G, HX>(sm, lane, K);
            if (s + 1 == steps) break;
            uint32_t neg = 0;
            int row = 0;
            if (s + 1 < len) {
                int wch;
                row = st.step(g, s, radix, &neg, &wch);
                ws = wch ? signed_weight<double>(g.w, g.parity) : flip_sign(ws);
            }
            fix_update<HX>(c, c0 + (size_t)(1 + row) * KB, neg);
        }
    }
}

// G lanes share one chunk: lane G p + q owns the HX columns [q HX, q HX + HX)
// (HX = ceil(K / G); the last lane's missing columns are pads, exactly 1).
// Per addend each lane
//   1. forms its leaves d_j (column pairs), in two chains their exclusive
//      suffix products S_j, and the product Q of its columns;
//   2. takes X, the product of the other lanes' Q, by shuffles;
//   3. runs the prefix products from X over the chains; m_j = prefix_j S_j
//      is all columns but those of pair j, and m_j times the one column of
//      the pair is added to the other column's sum, in 64-bit integers whose
//      unit, one per pair and lane, follows the largest addend of the run
//      (the sums move down when it grows).
// 3 K - 3 complex products per addend, as any prefix / suffix scheme needs.
// A task covers 16 chunks, with four lanes per chunk in two rounds.
//
// The sums.  A conversion to double and an FMA hold the FP64 pipe for 128
// cycles; done for every addend that would cost more than the products do
// (minors at K = 28: 453 cycles per column and addend), so integer sums run
// over at most 8 addends (|m_j c| < 2^60 (1 - 2^-21), so 8 stay below 2^63;
// never across a change of the binomial weight) and go to plain-double column
// sums beside the products, sign, weight and unit in one factor; 16 of those
// runs to the double-double totals.  The unit is what the accuracy hangs on:
// m_j is brought to [2^60, 2^61) at the run's largest addend (one unit for the
// whole warp: 3.5e-12 at 27 columns).  Shifts and the products summed round
// down; with every run of the same sign their half units add up over the
// walk, so every other run and chunk is summed with the opposite sign.  Errors
// against exact minors (root mean square relative; kernels in double / runs of
// 4 of one sign / here): 20 columns 1.0e-14 / 2.9e-15 / 1.3e-15, 24 columns
// 2.2e-14 / 1.3e-14 / 4.8e-15, 27 columns with collisions 1.0e-13 / 5e-14 /
// 1.6e-14.  Rounding the products summed as well: 1.1e-15, 4.0e-15, 1.4e-14,
// 1.4 % slower; truncating the exchanged products too: 1.2e-14 at 24 columns.
//
// Cancelling column sums.  A chain whose normalising shifts exceed s0 = 13 +
// log2 K (its products then err by more than 2^(s0 - 61)) is formed again from
// normalised column sums (suffix_chains<1>), which costs the addend half as
// much again; 5 % of a warp's addends at 30 columns, 1 % at 24.  A run's sum may
// still lie far below the unit that the run's largest m_j gave it, where
// columns are small whenever the products of the others are large: every
// eighth run (by a hash of its number) is looked at, and a task whose run
// sums add up to less than 2^45 units is walked again in double
// (walk_task_minors_dbl).  Without these, four blocks [[B, B], [B + 1, -B]] with B
// = 8e8 gave minors wrong by 30 times their value.  Normalising every column
// sum before its products, with a unit per column, needs neither, but takes 16
// % more instructions and spills above 20 columns (30 columns 65 ms).  The
// addends in double instead of suffix_chains<1>: 52.4 ms, and 10 us of latency
// for one in a small call; the look at every run in double: 2.6 ms more.
//
// Time.  29 x 30 minors (2^28 addends): 190 ms in double, 49.0 ms here (1.42e9 ->
// 5.48e9 addends/s; 45.2 without the provisions for cancelling sums, and 47.8
// with runs of 4, 49.7 with the m_j of an addend kept before any is added);
// 24 columns 0.640 ms (0.603 without, 0.670 with runs of 4).  The
// FMA-heavy pipe is about 70 % busy with integer products (4.35 cycles per
// warp and product) and every other integer instruction costs about 1.3
// cycles beside them, so what bounds it is the instruction count.
template <int G, int KB, int HX>
__device__ void walk_task_minors_fix(const bs_job& jb, const zfix* __restrict__ data, const int* __restrict__ radix,
                                     bs_zdd* __restrict__ slot, bool more, uint32_t local, int lane,
                                     MinorsSmem<G, HX>& sm) {
    constexpr int KP = KB;            // = BS_ROW_STRIDE(K) for every K of the bucket
    constexpr int NP = (HX + 1) / 2;  // leaves, in two chains of NA and NB
    constexpr int NA = (NP + 1) / 2, NB = NP - NA;
    const int K = jb.K;
    const int q = lane & (G - 1);
    const zfix* c0 = data + jb.data_off + q * HX;
    const zfix* a2 = c0 + KP;
    longlong2* sm_acc = sm.acc + lane;
    longlong2* sm_leaf = sm.leaf + lane;
    int4* sm_pair = sm.pair + lane;
#pragma unroll
    for (int t = 0; t < HX; ++t) sm_acc[t * 33] = make_longlong2(0, 0);
    for (int t = lane; t < K; t += 32) {
        sm.tot[t] = make_double4(0.0, 0.0, 0.0, 0.0);
        sm.run[t] = make_double2(0.0, 0.0);
        sm.est[t] = make_float2(0.f, __int_as_float(-(1 << 24)));
    }
    const int s0 = 13 + (31 - __clz(K));
    bool dbl = radix[BS_META_SPLIT(jb) - jb.meta_off] != 0;  // (columns of very unequal parts)
    for (int round = 0; round < G / 2 && !dbl; ++round) {
        const uint64_t i0_own = ((uint64_t)local * 16u + (uint64_t)(round * (32 / G) + lane / G)) << jb.log2L;
        const bool has = i0_own < jb.C;
        const uint64_t i0 = has ? i0_own : 0ull;
        uint32_t len = 0;
        if (has) {
            const uint64_t rem = jb.C - i0;
            len = (uint32_t)(rem < (1ull << jb.log2L) ? rem : (1ull << jb.log2L));
        }
        const uint32_t steps = __reduce_max_sync(0xffffffffu, len);
        if (steps == 0u) break;
        // runs end where a repeated-row digit moves (the weight changes there:
        // after every 2^nbin addends)
        const uint32_t run_mask = jb.nbin >= 3 ? kFixRun - 1u : (1u << jb.nbin) - 1u;
        static_assert(kFixRun == 8, "2^3 addends per run");
        bs_gray g;
        ChunkStepper st;
        st.init(g, i0, jb.nbin, jb.nrows, radix, reinterpret_cast<const uint64_t*>(radix + (BS_META_BINOM(jb) - jb.meta_off)));
        zraw c[HX];
        fix_seed<HX, KP>(c, g, c0, jb.nbin, jb.nrows);
        double ws = signed_weight<double>(g.w, g.parity);
        double wrun = ws;          // of the run's first addend
        // exponent of a sum's unit against m's: the last product's 64, its
        // column's -63, and 1 for every pad column (2^62 stands for 1, bound 2)
        const int e_unit = 64 - 63 + (G * HX - K);
        int em[NP];
        uint32_t runs = 0;
        const uint32_t flip = (uint32_t)(lane / G);  // parity of the chunk
        for (uint32_t s = 0; s < steps; ++s) {
            // 1. leaves, suffix products, Q
            int es[NP];
            zlimb qa, qb, pr;
            int ea, eb, e, smax;
            uint32_t ls[(NP + 3) / 4];
#pragma unroll
            for (int j = 0; j < (NP + 3) / 4; ++j) ls[j] = 0x01010101u * kLeafBias;
            suffix_chains<0, HX>(c, ls, qa, qb, ea, eb, smax, es, sm_leaf, sm_pair);
            if (__any_sync(0xffffffffu, smax > s0)) {
                // (a sum that is zero is exact, and with the others above 2^55
                // every other pair is accurate)
                bool zero = false, small = false;
#pragma unroll
                for (int t = 0; t < HX; ++t) {
                    const bool z = (c[t].re | c[t].im) == 0ull;
                    zero |= z;
                    small |= !z && (abs((int)(c[t].re >> 32)) | abs((int)(c[t].im >> 32))) < 1 << 23;
                }
                if (__any_sync(0xffffffffu, smax > s0 && (small || !zero)))
                    suffix_chains<1, HX>(c, ls, qa, qb, ea, eb, smax, es, sm_leaf, sm_pair);
            }
            {
                zraw ra;
                e = ea;
                if constexpr (NB > 0) {
                    ra = fix_cmul(qa, qb);
                    e += eb + 64;
                } else {
                    ra = raw_of(qa);
                }
                // the addend's sign against the run's first one goes here, and a
                // lane past its chunk adds zeros from here on.  Every other run
                // (and chunk) is summed with the opposite sign: shifts round down, and the
                // half unit each of them loses would add up over the runs.
                const unsigned long long m = 0ull - (unsigned long long)(((s & run_mask) ^ runs ^ flip) & 1u);
                ra.re = s < len ? (ra.re ^ m) - m : 0ull;
                ra.im = s < len ? (ra.im ^ m) - m : 0ull;
                pr = limbs_of(ra);
            }
            // 2. X
            if constexpr (G == 4) {
                const zlimb o1 = shfl_xor_zlimb(pr, 1);
                const int e1 = __shfl_xor_sync(0xffffffffu, e, 1);
                int e2 = e + e1 + 64;
                const zlimb o2 = shfl_xor_zlimb(fix_normalise(fix_cmul(pr, o1), e2), 2);
                e = e1 + __shfl_xor_sync(0xffffffffu, e2, 2) + 64;
                pr = fix_normalise(fix_cmul(o1, o2), e);
            } else {
                pr = shfl_xor_zlimb(pr, 1);
                e = __shfl_xor_sync(0xffffffffu, e, 1);
            }
            // 3. the prefix chains and the sums
            if ((s & run_mask) == 0u) {
#pragma unroll
                for (int j = 0; j < NP; ++j) em[j] = -(1 << 20);
            }
            {
                zlimb pa, pb;
                int fa = e, fb = e;
                pa = pr;
                if constexpr (NB > 0) {
                    fa += eb + 64;
                    fb += ea + 64;
                    pa = fix_normalise(fix_cmul(pr, qb), fa);
                    pb = fix_normalise(fix_cmul(pr, qa), fb);
                }
#pragma unroll
                for (int i = 0; i < NA; ++i) {
                    prefix_step<HX>(c, ls, i, i + 1 == NA, pa, fa, es[i], em[i], sm_acc, sm_leaf, sm_pair);
                    if (i < NB)
                        prefix_step<HX>(c, ls, NA + i, i + 1 == NB, pb, fb, es[NA + i], em[NA + i], sm_acc, sm_leaf, sm_pair);
                }
            }
            // the end of a run
            if (((s + 1u) & run_mask) == 0u || s + 1 == steps) {
                const double f = ((runs ^ flip) & 1u) ? -wrun : wrun;
                const bool look = runs * 0x9e3779b9u < 1u << 29;
                ++runs;
                minors_flush_fix<G, HX>(sm, f, e_unit, em, lane, K, (runs & (kFixFold - 1u)) == 0u || s + 1 == steps, look);
            }
            if (s + 1 == steps) break;
            uint32_t neg = 0;
            int row = 0;  // a lane past its chunk moves on, adding zeros
            if (s + 1 < len) {
                int wch;
                row = st.step(g, s, radix, &neg, &wch);
                ws = wch ? signed_weight<double>(g.w, g.parity) : flip_sign(ws);
            }
            if (((s + 1u) & run_mask) == 0u) wrun = ws;
            fix_update<HX>(c, a2 + (size_t)row * KP, neg);
        }
    }
    for (int t = lane; t < K; t += 32) dbl |= sm.est[t].x < 0.f;
    if (__any_sync(0xffffffffu, dbl)) walk_task_minors_dbl<G, KB, HX>(jb, data, radix, local, lane, sm);
    for (int t = lane; t < K; t += 32) {
        const double4 v = sm.tot[t];
        store_partial(slot + t, ddv{v.x, v.y}, ddv{v.z, v.w}, more);
    }
    __syncwarp();  // the next task's initialisation overwrites the totals
}

}  // namespace bs
