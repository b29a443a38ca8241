// Packing of one job (shared by the batch pack kernel and the sampler's
// device planner): the start sums c0[col] = sum over rows of M_row * a_row,col
// (every delta = +1) and 2a[j][col] for every digit row, rows of stride KP.
// Every column is scaled by a power of two whose exponent goes to colexp[col]
// and is undone exactly by the reduce kernel.
// FP64 jobs and double-float permanents: 64-bit fixed point (pack_job below,
// walk_fix.cuh).
// FP32 jobs: c0 exact, rounded once to double, then to float; column pairs {re(2p), re(2p+1),
// im(2p), im(2p+1)} (the packed layout of walk_fp32.cuh), column col scaled
// by 2^-e (e: smallest integer with sum_rows M_row (|Re a| + |Im a|) <= 2^e);
// pad columns have zero rows and c0 = 1 (a neutral factor).
// Double-float (DF) minors: rows of stride BS_ROW_STRIDE_DF(K) (a multiple of
// 8), column col scaled by 2^(2 - e) (colexp = e - 2) so that every column
// sum has |Re|, |Im| <= 4, and every entry quantised to a high part on the
// grid 2^-20 and a low part on the grid 2^-44, both exact floats
// (walk_df.cuh); pair p of a row is {re h, re h, im h, im h} of columns
// (2p, 2p+1), then the same for the low parts; pad columns have c0 = 1.
#pragma once
#include <cuda_runtime.h>
#include "bs_job.h"
#include "gray.h"
#include "walk.cuh"
#include "walk_fix.cuh"

namespace bs {

constexpr int kPackLanes = 8;    // lanes per column
constexpr int kPackBlock = 256;  // threads per job: 32 columns in one round

__device__ __forceinline__ double2 src_elem(const double2* __restrict__ src, const bs_job& jb, int r, int c) {
    return jb.src_trans ? src[jb.src_off + (int64_t)c * jb.src_ld + r] : src[jb.src_off + (int64_t)r * jb.src_ld + c];
}

// Element (row r, column col) of an FP32 job's packed rows.
__device__ __forceinline__ void put_f32(void* data, const bs_job& jb, int KP, int r, int col, float re, float im) {
    float* q = static_cast<float*>(data) + 2 * (jb.data_off + (int64_t)r * KP) + 4 * (col >> 1) + (col & 1);
    q[0] = re;
    q[2] = im;
}

// x 2^e: one multiplication where 2^e is a normal double (the same rounding
// as ldexp, whose general form takes several times as long).
__device__ __forceinline__ double scale2(double x, int e) {
    return abs(e) <= 1000 ? x * __hiloint2double((1023 + e) << 20, 0) : ldexp(x, e);
}

// FP32 and DF start sums are formed in 128-bit integers of unit
// 2^(e - kWideBits) for a column scaled by 2^-e: exact for entries down to
// 2^-68 of the column's bound (smaller ones lose what lies below 2^-120 of
// it), in any order of the rows, and without the double-double additions
// that an FP64 pipe of one instruction in 64 cycles makes the longest part
// of the packing.
constexpr int kWideBits = 120;

// x 2^(kWideBits - e), truncated; x finite, |x| <= 2^(e + 2).
__device__ __forceinline__ __int128 wide_of(double x, int e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    int ex = (int)(b >> 52) & 0x7ff;
    unsigned long long m = b & 0xfffffffffffffull;
    if (ex)
        m |= 1ull << 52;
    else
        ex = 1;
    const int s = ex - 1075 - e + kWideBits;
    const unsigned __int128 v = s >= 0 ? (unsigned __int128)m << min(s, 127) : (unsigned __int128)(s > -64 ? m >> -s : 0ull);
    return (long long)b < 0 ? -(__int128)v : (__int128)v;
}

// The wide integer v as a double, rounded to nearest.
__device__ __forceinline__ double wide_double(__int128 v) {
    const unsigned __int128 u = v < 0 ? -(unsigned __int128)v : (unsigned __int128)v;
    if (u == 0) return 0.0;
    const unsigned long long hi = (unsigned long long)(u >> 64);
    const int lz = hi ? __clzll((long long)hi) : 64 + __clzll((long long)(unsigned long long)u);
    const unsigned __int128 n = u << lz;
    // 64 leading bits and a sticky bit below them: one rounding
    const unsigned long long top = (unsigned long long)(n >> 64) | ((unsigned long long)n != 0ull ? 1ull : 0ull);
    const double d = scale2(__ull2double_rn(top), 64 - lz - kWideBits);
    return v < 0 ? -d : d;
}

// v / 2^S rounded to the nearest integer, halves to even.
template <int S>
__device__ __forceinline__ int wide_round(__int128 v) {
    const unsigned __int128 r = (unsigned __int128)v & (((unsigned __int128)1 << S) - 1), half = (unsigned __int128)1 << (S - 1);
    const int q = (int)(v >> S);
    return q + (int)(r > half || (r == half && (q & 1)));
}

// The DF split of v 2^-kWideBits (magnitude < 16): hi = v rounded to the grid
// 2^-20, lo = the rest rounded to the grid 2^-44, both exact floats.
__device__ __forceinline__ float2 df_split(__int128 v) {
    const int h = wide_round<kWideBits - 20>(v);
    const int l = wide_round<kWideBits - 44>(v - ((__int128)h << (kWideBits - 20)));
    return make_float2(__int2float_rn(h) * 0x1p-20f, __int2float_rn(l) * 0x1p-44f);
}

__device__ __forceinline__ __int128 wide_add_lanes(__int128 v) {  // over the lanes of a column
#pragma unroll
    for (int m = 1; m < kPackLanes; m <<= 1) {
        const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, m);
        const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), m);
        v += (__int128)(((unsigned __int128)hi << 64) | lo);
    }
    return v;
}

// Element (row r, column col) of a DF job's packed rows.
__device__ __forceinline__ void put_df(void* data, const bs_job& jb, int KP, int r, int col, float2 re, float2 im) {
    float* q = static_cast<float*>(data) + 4 * (jb.data_off + (int64_t)r * KP) + 8 * (col >> 1) + (col & 1);
    q[0] = re.x;
    q[2] = im.x;
    q[4] = re.y;
    q[6] = im.y;
}

// One job.  A column's entries are read once, by kPackLanes lanes with every
// eighth digit row each, all loads in flight together: a small job's packing
// is a chain of dependent loads (metadata, then the source, which may be in
// host memory) and of FP64 instructions, and both are as short as the lanes
// make them.  Sums over a column's rows are combined in a fixed order, the
// integer ones exactly, so the result does not depend on the block size.
// One FP32 job of 25 rows and 26 columns: 68 us with a thread per column and
// double-double sums, 11 us so; a sampler step's planning and packing at 26
// columns 87 -> 17 us; an FP64 job of 20 columns 15 -> 8 us.
//
// FP64 jobs and double-float permanents (walk_fix.cuh): column col scaled by
// 2^(63 - e), e (stored in colexp) the smallest integer with 2^e > b (1 +
// 2^-20), b = sum over rows of M_row (|Re a| + |Im a|); every entry rounded
// once to an integer, c0 and 2a formed from those integers modulo 2^64.  Where
// one part's bound is less than 1/8 of the other's, each part is scaled by its
// own (colexp holds the larger and how far the other lies below it) and the
// job is marked: its addends are formed in double (walk_fix.cuh), which keeps
// the accuracy of the smaller part.
// Ryser and Nijenhuis-Wilf jobs: product column col is matrix row sc; digit j
// is matrix column dsrc[j], added with +1 when it enters the subset, so the
// packed row is -a (the walk subtracts rows of digits whose Delta is 1);
// start sums 0 (Ryser) or x = a_(sc, n-1) - (sum_j a_(sc, j)) / 2
// (Nijenhuis-Wilf, whose entries are rounded to even integers so that the
// half is exact).
// A column with an entry that is not finite gets zeros in that part and
// BS_COLEXP_NAN_*: the reduce kernel writes NaN wherever such a column enters
// a product.
__device__ __forceinline__ void pack_job(const bs_job& jb, const double2* __restrict__ src, int* __restrict__ meta,
                                         void* __restrict__ data, int prec, int tid, int nthreads) {
    const bool df = BS_DF_MINORS(prec, jb.kind), f32 = prec == BS_PREC_FP32;
    const int* radix = meta + BS_META_RADIX(jb);
    const int* dsrc = meta + BS_META_DIGIT_SRC(jb);
    const int* csrc = meta + BS_META_COL_SRC(jb);
    int* colexp = meta + BS_META_COLEXP(jb);
    const int prow = meta[BS_META_PINNED(jb)];
    // binomial table C(M_j, d), digit after digit: a thread per digit
    for (int j = tid; j < jb.nrows; j += nthreads) {
        uint64_t* binom = reinterpret_cast<uint64_t*>(meta + BS_META_BINOM(jb)) + 2 * min(j, jb.nbin);
        for (int i = jb.nbin; i < j; ++i) binom += radix[i];
        const int M = radix[j] - 1;
        uint64_t v = 1;
        binom[0] = v;
        for (int d = 1; d <= M; ++d) {
            if (M > 1) v = v * (uint64_t)(M - d + 1) / (uint64_t)d;  // exact
            binom[d] = v;
        }
    }
    const int KP = df ? BS_ROW_STRIDE_DF(jb.K) : BS_ROW_STRIDE(jb.K);
    const bool bbfg = jb.formula == BS_JOB_BBFG, nw = jb.formula == BS_JOB_NW;
    constexpr int kRows = (BS_MAX_DIGITS + kPackLanes - 1) / kPackLanes;  // digit rows of a lane
    const int part = tid % kPackLanes;
    int split = 0;
    for (int base = 0; base < KP; base += nthreads / kPackLanes) {  // (every lane runs every round)
        const int col = base + tid / kPackLanes;
        const bool live = col < jb.K;
        const int sc = csrc[live ? col : 0];
        const bool first = part == 0 && (bbfg || nw);  // this lane also takes the start row
        double2 a0 = make_double2(0.0, 0.0), a[kRows];
        int m[kRows];
        if (first) a0 = src_elem(src, jb, bbfg ? prow : jb.n - 1, sc);
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int j = part + kPackLanes * i;
            a[i] = make_double2(0.0, 0.0);
            m[i] = 0;
            if (j < jb.nrows) {
                a[i] = src_elem(src, jb, dsrc[j], sc);
                m[i] = bbfg ? radix[j] - 1 : 1;
            }
        }
        double bre = fabs(a0.x), bim = fabs(a0.y);
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            if (kPackLanes * i >= jb.nrows) break;
            bre += (double)m[i] * fabs(a[i].x);
            bim += (double)m[i] * fabs(a[i].y);
        }
#pragma unroll
        for (int s = 1; s < kPackLanes; s <<= 1) {
            bre += __shfl_xor_sync(0xffffffffu, bre, s);
            bim += __shfl_xor_sync(0xffffffffu, bim, s);
        }
        // columns near the ends of the exponent range: the bounds once more, of
        // entries scaled by 2^up (finite entries may overflow in their sum, and
        // bounds of subnormal ones lose their bits below)
        int up = 0;
        const bool end = !(bre + bim < 0x1p1000) || (bre + bim < 0x1p-900 && bre + bim > 0.0);
        if (__any_sync(0xffffffffu, end)) {
            if (end) up = bre + bim < 1.0 ? 200 : -12;
            bre = fabs(scale2(a0.x, up));
            bim = fabs(scale2(a0.y, up));
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                bre += (double)m[i] * fabs(scale2(a[i].x, up));
                bim += (double)m[i] * fabs(scale2(a[i].y, up));
            }
#pragma unroll
            for (int s = 1; s < kPackLanes; s <<= 1) {
                bre += __shfl_xor_sync(0xffffffffu, bre, s);
                bim += __shfl_xor_sync(0xffffffffu, bim, s);
            }
        }
        int flags = 0;
        if (!isfinite(bre)) flags |= BS_COLEXP_NAN_RE;
        if (!isfinite(bim)) flags |= BS_COLEXP_NAN_IM;
        if ((flags & BS_COLEXP_NAN_RE) || !live) {
            bre = a0.x = 0.0;
#pragma unroll
            for (int i = 0; i < kRows; ++i) a[i].x = 0.0;
        }
        if ((flags & BS_COLEXP_NAN_IM) || !live) {
            bim = a0.y = 0.0;
#pragma unroll
            for (int i = 0; i < kRows; ++i) a[i].y = 0.0;
        }
        int e = 0;
        const double b = bre + bim;
        if (b > 0.0) {
            (void)frexp(f32 || df ? b : b * (1.0 + 0x1p-20), &e);
            e -= up;
        }
        if (df) e -= 2;  // column sums up to 4 (walk_df.cuh)
        int ere = e, eim = e;
        if (!f32 && !df && !flags && bre > 0.0 && bim > 0.0 && (bre < 0.125 * bim || bim < 0.125 * bre)) {
            (void)frexp(bre * (1.0 + 0x1p-20), &ere);
            (void)frexp(bim * (1.0 + 0x1p-20), &eim);
            ere = max(ere, eim - 900) - up;
            eim = max(eim - up, ere - 900);
            e = max(ere, eim);
            split |= live;
        }
        if (live && part == 0) colexp[col] = flags | BS_COLEXP(e, ere - eim);
        if (f32 || df) {
            __int128 sre = wide_of(a0.x, e), sim = wide_of(a0.y, e);
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                if (kPackLanes * i >= jb.nrows) break;
                const int j = part + kPackLanes * i;
                const __int128 qre = wide_of(a[i].x, e), qim = wide_of(a[i].y, e);
                sre += qre * m[i];
                sim += qim * m[i];
                if (j >= jb.nrows || col >= KP) continue;
                if (df)
                    put_df(data, jb, KP, 1 + j, col, df_split(2 * qre), df_split(2 * qim));
                else
                    put_f32(data, jb, KP, 1 + j, col, (float)scale2(a[i].x, 1 - e), (float)scale2(a[i].y, 1 - e));
            }
            sre = wide_add_lanes(sre);
            sim = wide_add_lanes(sim);
            if (part == 0 && col < KP) {
                if (df)
                    put_df(data, jb, KP, 0, col, live ? df_split(sre) : make_float2(1.f, 0.f), df_split(sim));
                else
                    put_f32(data, jb, KP, 0, col, live ? (float)wide_double(sre) : 1.f, (float)wide_double(sim));
            }
            continue;
        }
        zfix* out = static_cast<zfix*>(data) + jb.data_off;
        const int shre = (nw ? 62 : 63) - ere, shim = (nw ? 62 : 63) - eim;
        unsigned long long sre = (unsigned long long)__double2ll_rn(scale2(a0.x, shre));  // the start sums
        unsigned long long sim = (unsigned long long)__double2ll_rn(scale2(a0.y, shim));
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            if (kPackLanes * i >= jb.nrows) break;
            const int j = part + kPackLanes * i;
            const unsigned long long qre = (unsigned long long)__double2ll_rn(scale2(a[i].x, shre));
            const unsigned long long qim = (unsigned long long)__double2ll_rn(scale2(a[i].y, shim));
            zfix row;
            if (bbfg) {
                sre += (unsigned long long)m[i] * qre;
                sim += (unsigned long long)m[i] * qim;
                row.re = (long long)(2ull * qre);
                row.im = (long long)(2ull * qim);
            } else {
                // Nijenhuis-Wilf start: 2 x = 2 a_last - sum over all
                // columns = a_last - sum over the digits, in even units
                sre -= nw ? qre : 0ull;
                sim -= nw ? qim : 0ull;
                row.re = -(long long)(qre << (nw ? 1 : 0));
                row.im = -(long long)(qim << (nw ? 1 : 0));
            }
            if (j < jb.nrows && col < KP) out[(size_t)(1 + j) * KP + col] = row;
        }
#pragma unroll
        for (int s = 1; s < kPackLanes; s <<= 1) {
            sre += __shfl_xor_sync(0xffffffffu, sre, s);
            sim += __shfl_xor_sync(0xffffffffu, sim, s);
        }
        // a pad column's sum is exactly 1 = 2^62 / 2^63 2^1
        if (part == 0 && col < KP) out[col] = live ? zfix{(long long)sre, (long long)sim} : zfix{1ll << 62, 0};
    }
    if (f32 || df) return;
    split = __syncthreads_or(split);
    if (tid == 0) meta[BS_META_SPLIT(jb)] = split ? 1 : 0;
}

}  // namespace bs
