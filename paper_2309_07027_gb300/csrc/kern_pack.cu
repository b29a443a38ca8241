// Pack and reduce kernels.
//
// pack:   for every job, reads its source matrix (device) and writes
//           c0[col]   = sum over all rows of M_row * a_row,col  (all delta = +1)
//           2a[j][col] = 2 * a_digit_j,col
//         in the job's working precision, every column scaled by a power of
//         two (pack.cuh); the exponents go to colexp[] and are undone exactly
//         by the reduce kernel (Appendix A.5 normalises columns for the same
//         reason; here the factors are powers of two, so the rescaling is
//         exact).
// reduce: sums each job's task partials (Sum2, twice double precision) in a fixed order and
//         applies 2^(1-n) (Eq. bbfgrepeated prefactor) and the column scales.
#include <cuda_runtime.h>
#include "kernels.h"
#include "pack.cuh"
#include "walk.cuh"

namespace bs {

// The first CTA also clears `nclear` control words at `clear` (a memset of
// its own is one more stream operation in a call's chain).
__global__ void __launch_bounds__(kPackBlock) pack_kernel(const bs_job* __restrict__ jobs, const double2* __restrict__ src, int* __restrict__ meta,
                            void* __restrict__ data, int prec, unsigned long long* __restrict__ clear, int nclear) {
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < nclear; i += blockDim.x) clear[i] = 0ull;
    const bs_job jb = jobs[blockIdx.x];
    pack_job(jb, src, meta, data, prec, threadIdx.x, blockDim.x);
}

cudaError_t launch_pack(const bs_job* jobs, int njobs, const double2* src, int* meta, void* data, int prec,
                        cudaStream_t s, unsigned long long* clear, int nclear) {
    if (njobs <= 0) return cudaSuccess;
    pack_kernel<<<njobs, kPackBlock, 0, s>>>(jobs, src, meta, data, prec, clear, clear ? nclear : 0);
    return cudaGetLastError();
}

constexpr int kReduceBlock = 256;

// (s, c) -> normalised double-double (TwoSum of s and c: c may exceed s when
// the sum cancels).
__device__ __forceinline__ ddv sum2_final(ddv a) {
    const double h = __dadd_rn(a.hi, a.lo);
    const double bb = __dsub_rn(h, a.hi);
    return ddv{h, __dadd_rn(__dsub_rn(a.hi, __dsub_rn(h, bb)), __dsub_rn(a.lo, bb))};
}

// One CTA per (job, output column).  A CTA's time is its chain of dependent
// FP64 operations and loads, so the tree starts at the level the task count
// needs (in one warp, by shuffles, up to 32 tasks: no barrier), the column
// exponents are read by a warp at once, and the four results are scaled by
// four lanes.  9 tasks, 12 columns: 10.5 -> 7.6 us.
__global__ void __launch_bounds__(kReduceBlock) reduce_kernel(const bs_job* __restrict__ jobs,
                                                              const bs_zdd* __restrict__ partials,
                                                              const int* __restrict__ meta, double2* __restrict__ out,
                                                              double2* __restrict__ out_lo,
                                                              const int* __restrict__ status,
                                                              int* __restrict__ status_out) {
    // Sum2 (Ogita, Rump and Oishi 2005): the high parts are added with TwoSum,
    // the TwoSum errors and the low parts go to one plain double c; result
    // (s, c) as accurate as a sum in twice the working precision, at 8 FP64
    // operations per addition instead of about 20 for a double-double add.
    __shared__ ddv sre[kReduceBlock];
    __shared__ ddv sim[kReduceBlock];
    if (status_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *status_out = *status;
    const bs_job& jb = jobs[blockIdx.x];
    const int K = jb.K;
    const bool minors = jb.kind != BS_KIND_PERM;
    const int ncols = minors ? K : 1;
    const int col = blockIdx.y;
    if (col >= ncols) return;
    const uint32_t ntasks = jb.ntasks, ngroups = (ntasks + (1u << jb.fold_log2) - 1u) >> jb.fold_log2;
    const int lane = threadIdx.x & 31;
    if (ngroups <= 32u && threadIdx.x >= 32) return;
    const bs_zdd* p = partials + jb.partial_off + col;
    ddv re = {0.0, 0.0}, im = {0.0, 0.0};  // (s, c)
    for (uint32_t t = threadIdx.x; t < ngroups; t += kReduceBlock) {
        bs_zdd v = p[(int64_t)(t << jb.fold_log2) * ncols];
        // a group's slots first, as a warp that walks a whole group sums them
        const uint32_t end = min((t + 1) << jb.fold_log2, ntasks);
        for (uint32_t i = (t << jb.fold_log2) + 1; i < end; ++i) v = sum2_add(v, p[(int64_t)i * ncols]);
        re = sum2_add(re, v.re_hi, v.re_lo);
        im = sum2_add(im, v.im_hi, v.im_lo);
    }
    int e = 0, bad = 0;
    if (threadIdx.x < 32) {  // the exponents of the columns that enter the product
        const int* colexp = meta + BS_META_COLEXP(jb);
        for (int c = lane; c < K; c += 32) {
            if (minors && c == col) continue;
            const int x = colexp[c];
            bad |= x & (BS_COLEXP_NAN_RE | BS_COLEXP_NAN_IM);
            e += BS_COLEXP_E(x);
        }
        e = __reduce_add_sync(0xffffffffu, e);
        bad = (int)__reduce_or_sync(0xffffffffu, (unsigned)bad);
    }
    if (ngroups > 32u) {
        sre[threadIdx.x] = re;
        sim[threadIdx.x] = im;
        __syncthreads();
        int w = kReduceBlock / 2;
        while (w >= (int)ngroups) w >>= 1;  // the upper half holds zeros
        for (; w >= 32; w >>= 1) {
            if ((int)threadIdx.x < w) {
                const ddv r2 = sre[threadIdx.x + w], i2 = sim[threadIdx.x + w];
                sre[threadIdx.x] = re = sum2_add(re, r2.hi, r2.lo);
                sim[threadIdx.x] = im = sum2_add(im, i2.hi, i2.lo);
            }
            __syncthreads();
        }
        if (threadIdx.x >= 32) return;
    }
    for (int off = 16; off > 0; off >>= 1) {
        if (off >= (int)ngroups) continue;
        const ddv r2 = shfl_down_dd(re, off), i2 = shfl_down_dd(im, off);
        re = sum2_add(re, r2.hi, r2.lo);
        im = sum2_add(im, i2.hi, i2.lo);
    }
    // prefactor: 2^(1-n) times the column scales (Eq. bbfgrepeated), or
    // (-1)^n (Eq. ryser), or (-1)^(n-1) 2 (Nijenhuis-Wilf)
    double sgn = 1.0;
    if (jb.formula == BS_JOB_BBFG) {
        e += 1 - jb.n;
    } else if (jb.formula == BS_JOB_RYSER) {
        sgn = (jb.n & 1) ? -1.0 : 1.0;
    } else {
        e += 1;
        sgn = ((jb.n - 1) & 1) ? -1.0 : 1.0;
    }
    if (BS_FIXED(jb.prec, jb.kind)) e -= BS_FIX_BIAS;
    re = sum2_final(re);
    im = sum2_final(im);
    const double rh = __shfl_sync(0xffffffffu, re.hi, 0), rl = __shfl_sync(0xffffffffu, re.lo, 0);
    const double ih = __shfl_sync(0xffffffffu, im.hi, 0), il = __shfl_sync(0xffffffffu, im.lo, 0);
    if (lane >= 4) return;
    double x = lane == 0 ? rh : lane == 1 ? ih : lane == 2 ? rl : il;
    x = sgn * scale2(x, e);
    // an input that is not finite (a product of two or more columns mixes
    // both components)
    if (bad && (K - (minors ? 1 : 0) > 1 || (bad & ((lane & 1) ? BS_COLEXP_NAN_IM : BS_COLEXP_NAN_RE))))
        x = __longlong_as_double(0x7ff8000000000000ll);
    double2* o = lane < 2 ? out : out_lo;
    if (o) reinterpret_cast<double*>(o + jb.out_index + col)[lane & 1] = x;
}

cudaError_t launch_reduce(const bs_job* jobs, int njobs, const bs_zdd* partials, const int* meta, double2* out,
                          double2* out_lo, int max_cols, cudaStream_t s, const int* status, int* status_out) {
    if (njobs <= 0) return cudaSuccess;
    dim3 grid(njobs, max_cols < 1 ? 1 : max_cols);
    reduce_kernel<<<grid, kReduceBlock, 0, s>>>(jobs, partials, meta, out, out_lo, status, status_out);
    return cudaGetLastError();
}

}  // namespace bs
