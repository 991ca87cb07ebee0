/*
 * Device helpers shared by the unpack kernels (cfa_unpack.cu) and the TMA kernel (cfa_bulk.cu):
 * the per-vector checksum term and the warp reduction of checksums.  A checksum is the sum,
 * modulo 2^64, of a tensor's destination elements read as unsigned integers of the element size.
 */
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "cfa_internal.h"

namespace cfa_dev {

/* Sum of the elements of one 16-byte vector of ES-byte unsigned elements. */
template <int ES> __device__ __forceinline__ uint64_t vsum(uint4 v);
template <> __device__ __forceinline__ uint64_t vsum<1>(uint4 v)
{
    return (uint64_t)(__vsadu4(v.x, 0u) + __vsadu4(v.y, 0u) + __vsadu4(v.z, 0u) +
                      __vsadu4(v.w, 0u));
}
template <> __device__ __forceinline__ uint64_t vsum<2>(uint4 v)
{
    const uint32_t lo = (v.x & 0xFFFFu) + (v.y & 0xFFFFu) + (v.z & 0xFFFFu) + (v.w & 0xFFFFu);
    const uint32_t hi = (v.x >> 16) + (v.y >> 16) + (v.z >> 16) + (v.w >> 16);
    return (uint64_t)lo + hi;
}
template <> __device__ __forceinline__ uint64_t vsum<4>(uint4 v)
{
    return (uint64_t)v.x + v.y + v.z + v.w;
}
template <> __device__ __forceinline__ uint64_t vsum<8>(uint4 v)
{
    return (((uint64_t)v.y << 32) | v.x) + (((uint64_t)v.w << 32) | v.z);
}

/* Before a load that does not wait for the kernel before: nothing that an older kernel left in this
 * SM's L1 is to be read, whether or not an early start clears it.  (Staging slots and descriptor
 * memory are written again between launches.) */
__device__ __forceinline__ void launch_early(const cfa_launch_ctl &c)
{
    if (c.flags & CFA_LAUNCH_EARLY) __threadfence();
}

/* Before a kernel's first load of its source, every thread: the launch's place in its stream
 * (cfa_launch_ctl).  The fence comes after the wait, so that it also covers what came into L1
 * before the wait was over.
 * Dependents are released only after the wait, so that a later kernel of the group, which does
 * not wait for the source itself, cannot start before the source is there. */
__device__ __forceinline__ void launch_begin(const cfa_launch_ctl &c)
{
    if (c.flags & CFA_LAUNCH_WAIT_FIRST) asm volatile("griddepcontrol.wait;" ::: "memory");
    launch_early(c);
    if (c.flags & CFA_LAUNCH_RELEASE)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (c.clear) {
        const uint64_t n = (uint64_t)gridDim.x * blockDim.x;
        uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i < c.clear_words; i += n) c.clear[i] = 0;
    }
}

/* Last thing of a kernel: one CTA that waits for the kernel before keeps the whole grid from
 * ending first. */
__device__ __forceinline__ void launch_end(const cfa_launch_ctl &c)
{
    if ((c.flags & CFA_LAUNCH_WAIT_LAST) && blockIdx.x == 0)
        asm volatile("griddepcontrol.wait;" ::: "memory");
}

/* Host side: launches kernel fn as ctl says; args are the addresses of its parameters. */
inline cudaError_t launch_ctl(const void *fn, unsigned grid, unsigned threads, size_t smem,
                              cudaStream_t stream, const cfa_launch_ctl &ctl, void **args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr = {};
    if (ctl.flags & CFA_LAUNCH_EARLY) {
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelExC(&cfg, fn, args);
}

/* The same for a kernel whose one parameter holds its ctl. */
template <typename Args>
inline cudaError_t launch_ctl(void (*fn)(const Args), unsigned grid, unsigned threads, size_t smem,
                              cudaStream_t stream, const Args &args)
{
    void *p[] = {const_cast<Args *>(&args)};
    return launch_ctl(reinterpret_cast<const void *>(fn), grid, threads, smem, stream, args.ctl,
                      p);
}

/* Sum over the 32 lanes of a warp; lane 0 holds the total. */
__device__ __forceinline__ uint64_t warp_sum(uint64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    return v;
}

} // namespace cfa_dev
