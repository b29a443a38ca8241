// Packing of one job (shared by the batch pack kernel and the sampler's
// device planner): the start sums c0[col] = sum over rows of M_row * a_row,col
// (every delta = +1) and 2a[j][col] for every digit row, rows of stride KP.
// Every column is scaled by a power of two whose exponent goes to colexp[col]
// and is undone exactly by the reduce kernel.
// FP64 jobs and double-float permanents: 64-bit fixed point (pack_fix below,
// walk_fix.cuh).
// FP32 jobs: c0 in double-double, rounded; column pairs {re(2p), re(2p+1),
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

__device__ __forceinline__ double2 src_elem(const double2* __restrict__ src, const bs_job& jb, int r, int c) {
    return jb.src_trans ? src[jb.src_off + (int64_t)c * jb.src_ld + r] : src[jb.src_off + (int64_t)r * jb.src_ld + c];
}

// Element (row r, column col) of an FP32 job's packed rows.
__device__ __forceinline__ void put_f32(void* data, const bs_job& jb, int KP, int r, int col, float re, float im) {
    float* q = static_cast<float*>(data) + 2 * (jb.data_off + (int64_t)r * KP) + 4 * (col >> 1) + (col & 1);
    q[0] = re;
    q[2] = im;
}

// The DF split of v (|v| < 16): hi = v rounded to the grid 2^-20, lo = the
// rest rounded to the grid 2^-44; vlo: a low-order double added to v
// (double-double input), 0 otherwise.
__device__ __forceinline__ float2 df_quantise(double v, double vlo) {
    const double hi = rint(v * 0x1p20) * 0x1p-20;
    const double rest = (v - hi) + vlo;  // v - hi is exact
    const double lo = rint(rest * 0x1p44) * 0x1p-44;
    return make_float2((float)hi, (float)lo);
}

// Element (row r, column col) of a DF job's packed rows.
__device__ __forceinline__ void put_df(void* data, const bs_job& jb, int KP, int r, int col, float2 re, float2 im) {
    float* q = static_cast<float*>(data) + 4 * (jb.data_off + (int64_t)r * KP) + 8 * (col >> 1) + (col & 1);
    q[0] = re.x;
    q[2] = im.x;
    q[4] = re.y;
    q[6] = im.y;
}

// Fixed-point rows of an FP64 job (walk_fix.cuh): column col scaled by
// 2^(63 - e), e (stored in colexp) the smallest integer with 2^e > b (1 +
// 2^-20), b = sum over rows of M_row (|Re a| + |Im a|); every entry rounded
// once to an integer, c0 and 2a formed from those integers modulo 2^64.  Ryser and Nijenhuis-Wilf jobs:
// product column col is matrix row sc; digit j is matrix column dsrc[j],
// added with +1 when it enters the subset, so the packed row is -a (the walk
// subtracts rows of digits whose Delta is 1); start sums 0 (Ryser) or
// x = a_(sc, n-1) - (sum_j a_(sc, j)) / 2 (Nijenhuis-Wilf, whose entries are
// rounded to even integers so that the half is exact).  A column with an
// entry that is not finite gets zeros and BS_COLEXP_NAN_*: the reduce kernel
// writes NaN wherever such a column enters the product.
__device__ __forceinline__ void pack_fix(const bs_job& jb, const double2* __restrict__ src, int* __restrict__ meta,
                                         zfix* __restrict__ out, int tid, int nthreads) {
    const int* radix = meta + BS_META_RADIX(jb);
    const int* dsrc = meta + BS_META_DIGIT_SRC(jb);
    const int* csrc = meta + BS_META_COL_SRC(jb);
    int* colexp = meta + BS_META_COLEXP(jb);
    const int prow = meta[BS_META_PINNED(jb)];
    const int KP = BS_ROW_STRIDE(jb.K);
    const bool bbfg = jb.formula == BS_JOB_BBFG, nw = jb.formula == BS_JOB_NW;
    // four lanes per column, each with every fourth digit row: the packing of
    // a small job is a chain of dependent loads, and this one is a quarter as
    // long (12 photons: 12.1 -> 7.1 us); the sums are combined in a fixed
    // order, the integer ones exactly.
    const int part = tid & 3;
    for (int base = 0; base < KP; base += nthreads >> 2) {  // (every lane runs every round)
        const int col = base + (tid >> 2);
        const bool live = col < jb.K;
        const int sc = csrc[live ? col : 0];
        const bool first = part == 0 && (bbfg || nw);  // this lane also takes the start row
        const int frow = bbfg ? prow : jb.n - 1;
        double bre = 0.0, bim = 0.0;
        if (first) {
            const double2 a = src_elem(src, jb, frow, sc);
            bre = fabs(a.x);
            bim = fabs(a.y);
        }
#pragma unroll 2
        for (int j = part; j < jb.nrows; j += 4) {
            const double2 d = src_elem(src, jb, dsrc[j], sc);
            const double m = bbfg ? (double)(radix[j] - 1) : 1.0;
            bre += m * fabs(d.x);
            bim += m * fabs(d.y);
        }
        bre += __shfl_xor_sync(0xffffffffu, bre, 1);
        bim += __shfl_xor_sync(0xffffffffu, bim, 1);
        bre += __shfl_xor_sync(0xffffffffu, bre, 2);
        bim += __shfl_xor_sync(0xffffffffu, bim, 2);
        int flags = 0;
        if (!isfinite(bre)) flags |= BS_COLEXP_NAN_RE;
        if (!isfinite(bim)) flags |= BS_COLEXP_NAN_IM;
        int e = 0;
        const double b = 0.25 * bre + 0.25 * bim;  // a quarter: b must not overflow
        if (!flags && b > 0.0) {
            (void)frexp(b * (1.0 + 0x1p-20), &e);
            e += 2;
        }
        const bool use = live && !flags;
        const int sh = nw ? 62 - e : 63 - e;
        unsigned long long sre = 0, sim = 0;  // the start sums
        if (use && first) {
            const double2 a = src_elem(src, jb, frow, sc);
            sre = (unsigned long long)__double2ll_rn(ldexp(a.x, sh));
            sim = (unsigned long long)__double2ll_rn(ldexp(a.y, sh));
        }
#pragma unroll 2
        for (int j = part; j < jb.nrows; j += 4) {
            zfix row = {0, 0};
            if (use) {
                const double2 d = src_elem(src, jb, dsrc[j], sc);
                const unsigned long long qre = (unsigned long long)__double2ll_rn(ldexp(d.x, sh));
                const unsigned long long qim = (unsigned long long)__double2ll_rn(ldexp(d.y, sh));
                if (bbfg) {
                    const unsigned long long m = (unsigned long long)(radix[j] - 1);
                    sre += m * qre;
                    sim += m * qim;
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
            }
            if (col < KP) out[(size_t)(1 + j) * KP + col] = row;
        }
        sre += __shfl_xor_sync(0xffffffffu, sre, 1);
        sim += __shfl_xor_sync(0xffffffffu, sim, 1);
        sre += __shfl_xor_sync(0xffffffffu, sre, 2);
        sim += __shfl_xor_sync(0xffffffffu, sim, 2);
        if (part == 0 && col < KP) {
            // a pad column's sum is exactly 1 = 2^62 / 2^63 2^1
            out[col] = live ? zfix{(long long)sre, (long long)sim} : zfix{1ll << 62, 0};
            if (live) colexp[col] = flags ? flags : e;
        }
    }
}

__device__ __forceinline__ void pack_job(const bs_job& jb, const double2* __restrict__ src, int* __restrict__ meta,
                         void* __restrict__ data, int prec, int tid, int nthreads) {
    const int df = BS_DF_MINORS(prec, jb.kind);
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
    if (prec != BS_PREC_FP32 && !df) {
        pack_fix(jb, src, meta, static_cast<zfix*>(data) + jb.data_off, tid, nthreads);
        return;
    }
    const int KP = df ? BS_ROW_STRIDE_DF(jb.K) : BS_ROW_STRIDE(jb.K);
    for (int col = tid; col < KP; col += nthreads) {
        if (col >= jb.K) {  // pad column
            if (df) {
                put_df(data, jb, KP, 0, col, make_float2(1.f, 0.f), make_float2(0.f, 0.f));
                for (int j = 1; j <= jb.nrows; ++j) put_df(data, jb, KP, j, col, make_float2(0.f, 0.f), make_float2(0.f, 0.f));
            } else {
                put_f32(data, jb, KP, 0, col, 1.f, 0.f);
                for (int j = 1; j <= jb.nrows; ++j) put_f32(data, jb, KP, j, col, 0.f, 0.f);
            }
            continue;
        }
        const int sc = csrc[col];
        int e = 0;
        double2 a = src_elem(src, jb, prow, sc);
        double b = fabs(a.x) + fabs(a.y);
        for (int j = 0; j < jb.nrows; ++j) {
            double2 d = src_elem(src, jb, dsrc[j], sc);
            b += (double)(radix[j] - 1) * (fabs(d.x) + fabs(d.y));
        }
        if (b > 0.0) (void)frexp(b, &e);  // b = f 2^e, f in [0.5, 1)
        if (df) e -= 2;                   // DF: column sums up to 4 (walk_df.cuh)
        colexp[col] = e;
        // c0 in double-double (each product split exactly with an FMA), rounded
        ddv sre = {ldexp(a.x, -e), 0.0}, sim = {ldexp(a.y, -e), 0.0};
        for (int j = 0; j < jb.nrows; ++j) {
            double2 d = src_elem(src, jb, dsrc[j], sc);
            double m = (double)(radix[j] - 1);
            double dre = ldexp(d.x, -e), dim = ldexp(d.y, -e);
            double pre = m * dre, pim = m * dim;
            double ere = __fma_rn(m, dre, -pre), eim = __fma_rn(m, dim, -pim);
            sre = dd_add_d(dd_add_d(sre, pre), ere);
            sim = dd_add_d(dd_add_d(sim, pim), eim);
        }
        if (df) {
            put_df(data, jb, KP, 0, col, df_quantise(sre.hi, sre.lo), df_quantise(sim.hi, sim.lo));
            for (int j = 0; j < jb.nrows; ++j) {
                double2 d = src_elem(src, jb, dsrc[j], sc);
                put_df(data, jb, KP, 1 + j, col, df_quantise(ldexp(d.x, 1 - e), 0.0),
                       df_quantise(ldexp(d.y, 1 - e), 0.0));
            }
        } else {
            put_f32(data, jb, KP, 0, col, (float)sre.hi, (float)sim.hi);
            for (int j = 0; j < jb.nrows; ++j) {
                double2 d = src_elem(src, jb, dsrc[j], sc);
                put_f32(data, jb, KP, 1 + j, col, (float)ldexp(d.x, 1 - e), (float)ldexp(d.y, 1 - e));
            }
        }
    }
}

}  // namespace bs
