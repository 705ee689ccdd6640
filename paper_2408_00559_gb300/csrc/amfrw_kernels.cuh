// The solver kernels and their host launchers, instantiated once per N.
#pragma once
#include "amfrw_bundle.cuh"
#include "amfrw_f64.cuh"

namespace amfrw {

// The solver kernel.  CTA groups: one grid per block at a time from the
// launch's work counter.  Warp groups: a persistent multi-class launch -- every
// warp walks the launch's class list (ordered largest grids first) and takes
// chunks of 32 >> glog grids from each class's counter until it is exhausted,
// then moves on, so classes of uneven instances share one launch and no warp
// waits for another.
template <int N, bool MIXED, int KIND>
__global__ void __launch_bounds__(KIND == kWarpGroup ? 128 : kCtaMaxThreads, KIND == kWarpGroup ? (MIXED ? kWarpBlocksMixed : 3) : ((KIND == kMemGroup || MIXED) ? 2 : 1)) solve_kernel(SolveArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if constexpr (KIND == kWarpGroup) {
        const int warp = threadIdx.x >> 5;
        const int lane = threadIdx.x & 31;
        unsigned char* wbase = smem + (size_t)warp * (size_t)a.smem_warp;
        int c = 0;
        while (c < a.n_classes) {
            const ClassDesc cd = a.classes[c];
            int chunk = 0;
            if (lane == 0) chunk = atomicAdd(a.queue + cd.qidx, 32 >> cd.glog);
            chunk = __shfl_sync(0xffffffffu, chunk, 0);
            if (chunk >= cd.item_count) {
                ++c;
                continue;
            }
            const int item = chunk + (lane >> cd.glog);
            bool take = item < cd.item_count;
            Item it{};
            if (take) {
                it = a.items[cd.item_begin + item];
                take = !a.inst_mask || a.inst_mask[it.inst] != 0;
            }
            if (take) {
                const int gsize = 1 << cd.glog;
                unsigned char* base = wbase + (size_t)(lane >> cd.glog) * (size_t)cd.smem_group;
                if constexpr (MIXED)
                    solve_item_mixed<N, kWarpGroup>(a, it, base, base, lane & (gsize - 1), gsize);
                else
                    solve_item<N, false, kWarpGroup>(a, it, base, lane & (gsize - 1), gsize);
            }
        }
    } else {
        // CTA groups: the grid in shared memory; global-memory groups: in the
        // block's slice of the scratch array
        __shared__ int s_item;
        if constexpr (!MIXED) {
            // FP64: a grid per cluster of csize blocks (whole-block groups
            // where csize is 1), the slice shared by the cluster
            namespace cg = cooperative_groups;
            const int csize = a.csize, crank = csize > 1 ? (int)cg::this_cluster().block_rank() : 0;
            unsigned char* slice = a.lu_scratch + (size_t)(blockIdx.x / csize) * (size_t)a.lu_stride;
            auto csync = [&]() {
                if (csize > 1) cg::this_cluster().sync();
                else __syncthreads();
            };
            // another block's shared memory may be written only once that
            // block has started (the barriers below order the later passes)
            if (csize > 1) csync();
            for (;;) {
                if (crank == 0 && threadIdx.x == 0) {
                    const int v = atomicAdd(a.queue, 1);
                    s_item = v;
                    for (int r = 1; r < csize; ++r) *cg::cluster_group::map_shared_rank(&s_item, r) = v;
                }
                csync();
                const int item = s_item;
                csync();
                if (item >= a.n_items) break;
                const Item it = a.items[item];
                if (a.inst_mask && a.inst_mask[it.inst] == 0) continue;  // uniform across the cluster
                solve_item_f64<N, KIND>(a, it, smem, slice, crank, csize);
            }
        } else {
            unsigned char* base = KIND == kMemGroup ? a.lu_scratch + (size_t)blockIdx.x * (size_t)a.lu_stride : smem;
            for (;;) {
                if (threadIdx.x == 0) s_item = atomicAdd(a.queue, 1);
                __syncthreads();
                const int item = s_item;
                __syncthreads();
                if (item >= a.n_items) break;
                const Item it = a.items[item];
                if (a.inst_mask && a.inst_mask[it.inst] == 0) continue;  // uniform across the block
                // mixed-precision whole-block groups keep the unrolled stencil
                // of solve_item: with up to 256 threads on one grid the
                // per-node work dominates, and the unrolled form, each axis's
                // offsets in registers, measured 30 % faster on the d=6
                // modified level-6 workload than the table-driven form of the
                // warp groups
                solve_item<N, MIXED, KIND>(a, it, base, (int)threadIdx.x, (int)blockDim.x);
            }
        }
    }
}

// Host launch / occupancy helpers, instantiated once per N.
template <int N>
const void* kernel_for(bool mixed, int kind)
{
    if (kind == kBundle) return mixed ? (const void*)bundle_kernel<N, true> : (const void*)bundle_kernel<N, false>;
    if (kind == kWarpGroup)
        return mixed ? (const void*)solve_kernel<N, true, kWarpGroup> : (const void*)solve_kernel<N, false, kWarpGroup>;
    if (kind == kCtaGroup)
        return mixed ? (const void*)solve_kernel<N, true, kCtaGroup> : (const void*)solve_kernel<N, false, kCtaGroup>;
    return mixed ? (const void*)solve_kernel<N, true, kMemGroup> : (const void*)solve_kernel<N, false, kMemGroup>;
}

template <int N>
int launch_impl(const SolveArgs& a, bool mixed, int kind, int block, int grid, size_t smem, void* stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (kind == kWarpGroup) {
        if (mixed) solve_kernel<N, true, kWarpGroup><<<grid, block, smem, st>>>(a);
        else solve_kernel<N, false, kWarpGroup><<<grid, block, smem, st>>>(a);
    } else if (mixed) {
        if (kind == kCtaGroup) solve_kernel<N, true, kCtaGroup><<<grid, block, smem, st>>>(a);
        else solve_kernel<N, true, kMemGroup><<<grid, block, smem, st>>>(a);
    } else {  // FP64: `grid` clusters of csize blocks
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(grid * a.csize));
        cfg.blockDim = dim3((unsigned)block);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)a.csize;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = a.csize > 1 ? 1 : 0;
        return (int)(kind == kCtaGroup ? cudaLaunchKernelEx(&cfg, solve_kernel<N, false, kCtaGroup>, a)
                                       : cudaLaunchKernelEx(&cfg, solve_kernel<N, false, kMemGroup>, a));
    }
    return (int)cudaGetLastError();
}

template <int N>
int launch_bundle_impl(const BundleArgs& a, bool mixed, int grid, size_t smem, void* stream)
{
    if (mixed) bundle_kernel<N, true><<<grid, kBundleThreads, smem, (cudaStream_t)stream>>>(a);
    else bundle_kernel<N, false><<<grid, kBundleThreads, smem, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

template <int N>
int occupancy_impl(bool mixed, int kind, int block, size_t smem)
{
    int nb = 0;
    const void* f = kernel_for<N>(mixed, kind);
    // The limit is an attribute of the kernel, shared by all its launches, and
    // launches of one kernel request different amounts: past the default
    // 48 KB, allow the device's opt-in maximum (less the kernel's static
    // shared memory), so that no launch depends on which query came last.
    if (smem > 48 * 1024) {
        int dev = 0, optin = 0;
        cudaFuncAttributes fa{};
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, f) != cudaSuccess)
            return 0;
        const int lim = optin - (int)fa.sharedSizeBytes;
        if ((size_t)lim < smem ||
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess)
            return 0;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, block, smem) != cudaSuccess) return 0;
    return nb;
}

}  // namespace amfrw

#define AMFRW_INSTANTIATE(NN)                                                               \
    namespace amfrw {                                                                       \
    int launch_n##NN(const SolveArgs& a, bool m, int k, int b, int g, size_t s, void* st)   \
    {                                                                                       \
        return launch_impl<NN>(a, m, k, b, g, s, st);                                       \
    }                                                                                       \
    int launch_bundle_n##NN(const BundleArgs& a, bool m, int g, size_t s, void* st)         \
    {                                                                                       \
        return launch_bundle_impl<NN>(a, m, g, s, st);                                      \
    }                                                                                       \
    int occupancy_n##NN(bool m, int k, int b, size_t s) { return occupancy_impl<NN>(m, k, b, s); } \
    }
