// FP64 walk kernels: permanents and fused Laplace minors in 64-bit fixed
// point (walk_fix.cuh), weights and sums in double and double-double.
// One kernel per column bucket KB (K in (KB-4, KB]); the host groups jobs by
// bucket, so each kernel keeps its own register allocation.  Inside, each
// task runs the walk instance for its lanes' exact column count.
#include "kernels.h"
#include "sample.h"
#include "walk.cuh"
#include "walk_fix.cuh"

namespace bs {

constexpr int kPermBlock = 64;  // one task per CTA: two warps, half of its chunks each
constexpr int kMinorsBlock = 64;

// 128 registers (16 warps per SM) up to width 32, 168 above; 12 warps ran 2 %
// slower at widths 26 to 30.  Two warps per task instead of one with twice
// the chunks: a task's latency halves, which is the time of a job with fewer
// tasks than resident warps (20 x 20: 109 -> 58 us).
// GROUPS: tasks may be groups (walk_log2); instances of their own, as the loop
// over a group costs 2 to 4 % in registers.
template <int KB, bool GROUPS>
__global__ void __launch_bounds__(kPermBlock, KB <= 32 ? 8 : 6) walk_fp64_perm_kernel(WalkArgs a) {
    __shared__ unsigned long long s_task;
    __shared__ ddv s_half[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bs_job* __restrict__ jobs = a.jobs;
    const zfix* __restrict__ data = static_cast<const zfix*>(a.data);
    const unsigned long long total = task_total(a);
    const int njobs = job_count(a);
    const unsigned long long deadline = warp_deadline(a.deadline_rel_ns);
    for (;;) {
        if (warp == 0) {
            const unsigned long long next = next_task(a.counter, total, a.status, deadline, lane);
            if (lane == 0) s_task = next;
        }
        __syncthreads();
        const unsigned long long t = s_task;
        if (t >= total) break;
        const bs_job jb = jobs[find_job(jobs, a.job_list, njobs, t)];
        const bool ok = ((jb.K + 3) >> 2) == KB / 4 && jb.kind == BS_KIND_PERM;
        const uint32_t local = (uint32_t)(t - jb.task_begin) + jb.task_offset;
        const int* radix = a.meta + BS_META_RADIX(jb);
        if (!ok && threadIdx.x == 0) atomicExch(a.status, BS_STATUS_BADJOB);
        for (uint32_t i = 0; GROUPS ? i >> jb.walk_log2 == 0 : i < 1; ++i) {
            const uint32_t task = GROUPS ? (local << jb.walk_log2) + i : local;
            if (!ok || (GROUPS && !task_exists(jb, task, 32))) break;
            ddv re = {0.0, 0.0}, im = {0.0, 0.0};
            if (radix[BS_META_SPLIT(jb) - jb.meta_off] != 0) {
                if (((jb.K + 1) >> 1) == KB / 2)
                    walk_task_perm_dbl<KB, KB / 2>(jb, data, radix, task, warp, lane, re, im);
                else
                    walk_task_perm_dbl<KB, KB / 2 - 1>(jb, data, radix, task, warp, lane, re, im);
            } else if (((jb.K + 1) >> 1) == KB / 2) {  // the instance whose lanes own exactly ceil(K / 2) columns
                walk_task_perm_fix<KB, KB / 2>(jb, data, radix, task, warp, lane, re, im);
            } else {
                walk_task_perm_fix<KB, KB / 2 - 1>(jb, data, radix, task, warp, lane, re, im);
            }
            if (threadIdx.x == 32) {
                s_half[0] = re;
                s_half[1] = im;
            }
            __syncthreads();
            if (threadIdx.x == 0)
                store_partial(a.partials + jb.partial_off + local, dd_add_sum2(re, s_half[0]), dd_add_sum2(im, s_half[1]), i > 0);
            if (GROUPS) __syncthreads();  // (s_half is written again)
        }
        if (GROUPS || !ok) __syncthreads();  // (s_task as well)
    }
}

// Resident CTAs per SM that the fused-minor kernels are compiled for (64
// threads each): 168 registers, 3 warps per scheduler from width 16 on.  Two
// warps at 254 registers ran 9 % slower (width 28), four at 128 spill.
template <int KB>
struct MinorsMinBlocks {
    static constexpr int value = KB <= 4 ? 14 : KB <= 8 ? 10 : KB <= 12 ? 8 : 6;
};

template <int KB, bool GROUPS>
__global__ void __launch_bounds__(kMinorsBlock, MinorsMinBlocks<KB>::value) walk_fp64_minors_kernel(WalkArgs a) {
    constexpr int G = BS_MINORS_FP64_GROUP_KB(KB);
    constexpr int HM = KB / G;  // most columns a lane owns
    extern __shared__ double4 smem_fp64[];
    const int lane = threadIdx.x & 31;
    char* smem = reinterpret_cast<char*>(smem_fp64) + (threadIdx.x >> 5) * sizeof(MinorsSmem<G, HM>);
    const bs_job* __restrict__ jobs = a.jobs;
    const zfix* __restrict__ data = static_cast<const zfix*>(a.data);
    const unsigned long long total = task_total(a);
    const int njobs = job_count(a);
    const unsigned long long deadline = warp_deadline(a.deadline_rel_ns);
    for (;;) {
        unsigned long long t = next_task(a.counter, total, a.status, deadline, lane);
        if (t >= total) break;
        const bs_job jb = jobs[find_job(jobs, a.job_list, njobs, t)];
        if (((jb.K + 3) >> 2) != KB / 4 || jb.kind != BS_KIND_MINORS) {
            if (lane == 0) atomicExch(a.status, BS_STATUS_BADJOB);
            continue;
        }
        const uint32_t local = (uint32_t)(t - jb.task_begin) + jb.task_offset;
        const int* radix = a.meta + BS_META_RADIX(jb);
        bs_zdd* slot = a.partials + jb.partial_off + (int64_t)local * jb.K;
        for (uint32_t i = 0; GROUPS ? i >> jb.walk_log2 == 0 : i < 1; ++i) {
            const uint32_t task = GROUPS ? (local << jb.walk_log2) + i : local;
            if (GROUPS && !task_exists(jb, task, 16)) break;
            // the instance whose lanes own exactly ceil(K / G) columns
            if (G == 4 || ((jb.K + 1) >> 1) == HM)
                walk_task_minors_fix<G, KB, HM>(jb, data, radix, slot, i > 0, task, lane,
                                                *reinterpret_cast<MinorsSmem<G, HM>*>(smem));
            else
                walk_task_minors_fix<G, KB, HM - 1>(jb, data, radix, slot, i > 0, task, lane,
                                                    *reinterpret_cast<MinorsSmem<G, HM - 1>*>(smem));
        }
    }
}

template <typename Kern>
static int persistent_grid(Kern k, int block, size_t smem, int threads_per_task, const WalkArgs& a) {
    int dev = 0;
    cudaGetDevice(&dev);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem);
    if (per_sm < 1) per_sm = 1;
    long long grid = (long long)per_sm * sm_count(dev);
    if (!a.total_dev) {
        long long need = ((long long)a.total_tasks * threads_per_task + block - 1) / block;
        if (need < grid) grid = need;
    }
    if (a.grid_cap > 0 && grid > a.grid_cap) grid = a.grid_cap;
    if (grid < 1) grid = 1;
    return (int)grid;
}

template <int KB>
static cudaError_t run_perm(const WalkArgs& a, cudaStream_t s) {
    const auto kernel = a.groups ? walk_fp64_perm_kernel<KB, true> : walk_fp64_perm_kernel<KB, false>;
    int grid = persistent_grid(kernel, kPermBlock, 0, kPermBlock, a);
    kernel<<<grid, kPermBlock, 0, s>>>(a);
    return cudaGetLastError();
}

template <int KB>
static cudaError_t run_minors(const WalkArgs& a, cudaStream_t s) {
    constexpr int G = BS_MINORS_FP64_GROUP_KB(KB);
    const size_t smem = (kMinorsBlock / 32) * sizeof(MinorsSmem<G, KB / G>);
    const auto kernel = a.groups ? walk_fp64_minors_kernel<KB, true> : walk_fp64_minors_kernel<KB, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int grid = persistent_grid(kernel, kMinorsBlock, smem, 32, a);
    kernel<<<grid, kMinorsBlock, smem, s>>>(a);
    return cudaGetLastError();
}

#define BS_B48(X) X(1, 4) X(2, 8) X(3, 12) X(4, 16) X(5, 20) X(6, 24) X(7, 28) X(8, 32) X(9, 36) X(10, 40) X(11, 44) X(12, 48)

// a.max_K selects the bucket: every job of the launch must share it.
cudaError_t launch_walk_fp64_perm(const WalkArgs& a, cudaStream_t s) {
    if (a.total_tasks == 0 && !a.total_dev) return cudaSuccess;
    switch ((a.max_K + 3) >> 2) {
#define BS_CASE(b, kb) \
    case b: return run_perm<kb>(a, s);
        BS_B48(BS_CASE)
#undef BS_CASE
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_walk_fp64_minors(const WalkArgs& a, cudaStream_t s) {
    if (a.total_tasks == 0 && !a.total_dev) return cudaSuccess;
    switch ((a.max_K + 3) >> 2) {
#define BS_CASE(b, kb) \
    case b: return run_minors<kb>(a, s);
        BS_B48(BS_CASE)
#undef BS_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace bs
