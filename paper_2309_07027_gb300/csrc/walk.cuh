// What the Gray-walk kernels for the generalized BB/FG sum (Eq. bbfgrepeated)
// and its fused Laplace-minor variant share.
//
// Work decomposition (Sec. 2.1: contiguous index ranges walked
// independently, each seeded by decoding its first index):
//   * a job's index range [0, C) is cut into chunks of L = 2^log2L addends;
//   * a warp task is a run of consecutive chunks; a chunk is walked by one
//     lane or by a small group of lanes that split the columns;
//   * persistent warps pull tasks from a global counter (largest jobs are
//     planned first), so uneven jobs share one launch;
//   * every lane decodes its chunk start (seeding its column sums from the
//     matrix) and then steps through the chunk one digit move at a time.
// Because chunk starts are multiples of L, all lanes of a warp flip the same
// binary digit at each step except at the rare carries past bit log2L, so the
// row they read is a broadcast load.
//
// Per addend:
//   update   c_col += +-2 a_row,col
//   product  P = prod_col c_col
//   weight   acc += (+-W) * P                      (Eq. bbfgrepeated weight)
// Minors additionally form, for every column l, prod_{col != l} c_col from
// suffix and prefix products (about 3 products per column instead of K).
//
// The arithmetic: walk_fix.cuh (FP64 jobs), walk_fp32.cuh (FP32 jobs),
// walk_df.cuh (double-float jobs).  In each, a lane sums its addends for a
// short run and folds the run into a compensated sum, and the lanes of a task
// are combined in a fixed order.  Tasks write one partial per output; the
// reduce kernel sums them in a fixed order.  The cut into tasks and that order
// are functions of the job (bs_cut in sample.h), so results do not depend on
// which warp ran which task, on what else was in the launch or on the memory
// at hand.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "bs_job.h"
#include "gray.h"
#include "kernels.h"

namespace bs {

template <typename T>
struct cx {
    T re, im;
};

__device__ __forceinline__ float bfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double bfma(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename T>
__device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) {
    cx<T> r;
    r.re = bfma(a.re, b.re, -(a.im * b.im));
    r.im = bfma(a.re, b.im, a.im * b.re);
    return r;
}

// ---------------------------------------------------------------- compensated sums
struct ddv {
    double hi, lo;
};

// TwoSum (Knuth) then renormalisation; adds a double into a double-double.
__device__ __forceinline__ ddv dd_add_d(ddv a, double b) {
    double s = __dadd_rn(a.hi, b);
    double bb = __dsub_rn(s, a.hi);
    double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, bb)), __dsub_rn(b, bb));
    e = __dadd_rn(e, a.lo);
    double h = __dadd_rn(s, e);
    ddv r;
    r.hi = h;
    r.lo = __dsub_rn(e, __dsub_rn(h, s));
    return r;
}

// Double-double addition in Sum2 form (Ogita, Rump and Oishi 2005): TwoSum
// of the high parts, its error and both low parts added in double, one
// renormalisation; 11 FP64 operations instead of 20.  Sums of many terms
// formed this way are as accurate as summation in twice double precision,
// which is what the task and cross-lane combinations need (the FP64 pipe is
// 1/64 of the FP32 pipe here, and a small job's latency is its warps' FP64
// instruction count).
__device__ __forceinline__ ddv dd_add_sum2(ddv a, ddv b) {
    const double s = __dadd_rn(a.hi, b.hi);
    const double bb = __dsub_rn(s, a.hi);
    double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, bb)), __dsub_rn(b.hi, bb));
    e = __dadd_rn(e, __dadd_rn(a.lo, b.lo));
    ddv r;
    r.hi = __dadd_rn(s, e);
    r.lo = __dsub_rn(e, __dsub_rn(r.hi, s));
    return r;
}

struct ffv {
    float hi, lo;
};

// TwoSum in single precision: adds a float into a float-float.
__device__ __forceinline__ ffv ff_add_f(ffv a, float b) {
    float s = __fadd_rn(a.hi, b);
    float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    e = __fadd_rn(e, a.lo);
    ffv r;
    r.hi = __fadd_rn(s, e);
    r.lo = __fsub_rn(e, __fsub_rn(r.hi, s));
    return r;
}

__device__ __forceinline__ ddv dd_from_ff(ffv a) {
    ddv r;
    r.hi = (double)a.hi;
    r.lo = 0.0;
    return dd_add_d(r, (double)a.lo);
}

// Float-float addition (TwoSum of the high parts, low parts added, one
// renormalisation); used for cross-lane sums in the FP32 kernels so that no
// FP64 instruction runs in their loops.
__device__ __forceinline__ ffv ff_add(ffv a, ffv b) {
    float s = __fadd_rn(a.hi, b.hi);
    float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    ffv r;
    r.hi = __fadd_rn(s, e);
    r.lo = __fsub_rn(e, __fsub_rn(r.hi, s));
    return r;
}

__device__ __forceinline__ ffv shfl_down_ff(ffv v, int off) {
    ffv r;
    r.hi = __shfl_down_sync(0xffffffffu, v.hi, off);
    r.lo = __shfl_down_sync(0xffffffffu, v.lo, off);
    return r;
}

__device__ __forceinline__ ddv shfl_down_dd(ddv v, int off) {
    ddv r;
    r.hi = __shfl_down_sync(0xffffffffu, v.hi, off);
    r.lo = __shfl_down_sync(0xffffffffu, v.lo, off);
    return r;
}

__device__ __forceinline__ double flip_sign(double x) {
    return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}
__device__ __forceinline__ float flip_sign(float x) {
    return __int_as_float(__float_as_int(x) ^ (int)0x80000000u);
}

// +1 or -1 (neg = 1) built from bits, so no int-to-float conversion runs in
// the loop.
__device__ __forceinline__ float unit_sign_f(uint32_t neg) { return __int_as_float(0x3f800000u | (neg << 31)); }
// In-chunk stepper.  A chunk starts at a multiple i0 of L = 2^log2L and
// takes fewer than L steps, so the index i0 + s has exactly the trailing
// ones of s: the digit that moves at step s -> s + 1 is t = ctz(s + 1) < 12
// when t < nbin (a binary flip, 32-bit arithmetic only), and otherwise every
// binary digit is saturated and a repeated-row digit moves (general step).
// The stepper itself holds only scalars (kept in registers); the full Gray
// state g, whose repeated-row digit arrays are indexed at run time and so
// live in local memory, is a separate object that only the general step
// touches.
struct ChunkStepper {
    uint64_t i0;
    const uint64_t* binom;
    uint32_t dlo;   // Delta bits of binary digits 0..31
    int parity0;    // parity at the chunk start
    int nbin;

    __device__ __forceinline__ void init(bs_gray& g, uint64_t start, int nb, int nrows, const int* radix,
                                         const uint64_t* tab) {
        binom = tab;
        bs_gray_decode(g, start, nb, nrows, radix, tab);
        i0 = start;
        dlo = (uint32_t)g.dbin;
        parity0 = g.parity;
        nbin = nb;
    }
    // The step to index i0 + u when it moves a binary digit (ctz(u) < nbin,
    // which the caller guarantees): returns the row, *neg as in step().
    __device__ __forceinline__ int step_bin(uint32_t u, uint32_t* neg) {
        const int t = __ffs((int)u) - 1;
        const uint32_t was = (dlo >> t) & 1u;
        dlo ^= 1u << t;
        *neg = was ^ 1u;
        return t;
    }
    // Move from index i0 + s to i0 + s + 1.  Returns the digit row; *neg is 1
    // when the column sums move by -2a_row (Delta rises), 0 for +2a_row;
    // *wch is 1 when the binomial weight changed (then g.w, g.parity are
    // current).
    __device__ __forceinline__ int step(bs_gray& g, uint32_t s, const int* radix, uint32_t* neg, int* wch) {
        const int t = __ffs((int)(s + 1u)) - 1;
        if (t < nbin) {
            const uint32_t was = (dlo >> t) & 1u;
            dlo ^= 1u << t;
            *neg = was ^ 1u;
            *wch = 0;
            return t;
        }
        g.i = i0 + s;
        g.parity = parity0 ^ (int)(s & 1u);
        g.dbin = (g.dbin & ~0xffffffffull) | (uint64_t)dlo;
        int coef;
        const int row = bs_gray_step(g, radix, &coef, wch, binom);
        *neg = coef < 0 ? 1u : 0u;
        return row;
    }
};

// The packed rows of a job with K columns have stride BS_ROW_STRIDE(K), the
// width KB of the bucket kernel that walks it: inside a kernel the stride is
// the compile-time KB.
static_assert(BS_ROW_STRIDE(29) == 32 && BS_ROW_STRIDE(32) == 32 && BS_ROW_STRIDE(1) == 4,
              "row stride must equal the 4-column bucket width");

template <typename T>
__device__ __forceinline__ T signed_weight(uint64_t w, int parity) {
    T x = (T)w;
    return parity ? -x : x;
}

// One Sum2 step: (s, c) + (hi, lo) -> (s', c + e + lo) with s' + e = s + hi
// exactly (TwoSum, Knuth).
__device__ __forceinline__ ddv sum2_add(ddv a, double hi, double lo) {
    const double s = __dadd_rn(a.hi, hi);
    const double bb = __dsub_rn(s, a.hi);
    const double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, bb)), __dsub_rn(hi, bb));
    return ddv{s, __dadd_rn(a.lo, __dadd_rn(e, lo))};
}

__device__ __forceinline__ bs_zdd sum2_add(const bs_zdd& a, const bs_zdd& b) {
    const ddv re = sum2_add(ddv{a.re_hi, a.re_lo}, b.re_hi, b.re_lo), im = sum2_add(ddv{a.im_hi, a.im_lo}, b.im_hi, b.im_lo);
    return bs_zdd{re.hi, re.lo, im.hi, im.lo};
}

// A task's partial into its slot; `more`: it joins those of its group before it.
__device__ __forceinline__ void store_partial(bs_zdd* p, ddv re, ddv im, bool more) {
    const bs_zdd v = {re.hi, re.lo, im.hi, im.lo};
    *p = more ? sum2_add(*p, v) : v;
}

__device__ __forceinline__ void store_partial(bs_zdd* p, ddv re, ddv im) {
    bs_zdd o;
    o.re_hi = re.hi;
    o.re_lo = re.lo;
    o.im_hi = im.hi;
    o.im_lo = im.lo;
    *p = o;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Job owning global task t: the last job (in list order) whose task_begin
// <= t.  Jobs are jobs[i], or jobs[list[i]] when a device-built list is
// given.
__device__ __forceinline__ int find_job(const bs_job* __restrict__ jobs, const int* __restrict__ list, int njobs,
                                        unsigned long long t) {
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        const int jm = list ? list[mid] : mid;
        if (jobs[jm].task_begin <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return list ? list[lo] : lo;
}

// Pull the next warp task (lane 0 takes it, all lanes learn it).  A task
// index >= total means stop: either the work is done or the deadline passed
// (then the status word says so and the host reports a timeout).
// deadline_ns is absolute (%globaltimer), 0 = none.
__device__ __forceinline__ unsigned long long next_task(unsigned long long* counter, unsigned long long total,
                                                        int* status, unsigned long long deadline_ns, int lane) {
    unsigned long long t = 0;
    if (lane == 0) {
        if (deadline_ns != 0ull && global_ns() > deadline_ns) {
            atomicExch(status, BS_STATUS_TIMEOUT);
            t = total;
        } else {
            t = atomicAdd(counter, 1ull);
        }
    }
    return __shfl_sync(0xffffffffu, t, 0);
}

// Whether the cut's task `local` of chunks_per_task chunks has any addends.
__device__ __forceinline__ bool task_exists(const bs_job& jb, uint32_t local, uint32_t chunks_per_task) {
    return (uint64_t)local * chunks_per_task << jb.log2L < jb.C;
}

// Per-warp absolute deadline from a relative one (0 = none).
__device__ __forceinline__ unsigned long long warp_deadline(unsigned long long rel_ns) {
    return rel_ns == 0ull ? 0ull : global_ns() + rel_ns;
}

// Task total and job count: from device memory when planned on the device.
__device__ __forceinline__ unsigned long long task_total(const WalkArgsBase& a) {
    return a.total_dev ? *a.total_dev : a.total_tasks;
}
__device__ __forceinline__ int job_count(const WalkArgsBase& a) { return a.njobs_dev ? *a.njobs_dev : a.njobs; }

}  // namespace bs
