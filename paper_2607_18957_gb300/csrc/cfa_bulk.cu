/*
 * TMA bulk-copy unpack: the "InGPU -> Loaded" copy of InstantInfer section 4.2 for large
 * contiguous runs that need no cast and whose source, destination and length are multiples of
 * 16 bytes.  Instead of every thread moving 16-byte vectors through registers, the Tensor
 * Memory Accelerator moves the bytes with non-tensor bulk copies:
 *
 *     global (staging) --cp.async.bulk--> shared stage --cp.async.bulk--> global (destination)
 *
 * Each CTA is two warps over a ring of two 32 KiB stages, three CTAs per SM:
 *   - warp 0 (one lane) loads: it waits until a stage is empty, then issues the bulk load of the
 *     next sub-block into it, completing on the stage's `full` mbarrier (complete_tx);
 *   - warp 1 consumes: it waits on `full`, sums the stage for the per-tensor checksum (all 32
 *     lanes), and one lane issues the bulk store; once the store of the previous sub-block has
 *     finished reading its stage (bulk_group read wait), that stage is released on its `empty`
 *     mbarrier.
 * An item is a contiguous run, or a block of rows of a column slice: then one bulk load per row
 * gathers the rows back to back in the stage and one bulk store writes them.
 * One launch takes the items of every element size (the consumer sums each stage by its item's
 * size), cut into parts (cfa_parts_log2).  With a launch per
 * element size, forked and joined with events, and whole 256 KiB slabs, an 8-bit checkpoint with
 * block scales unpacked in 64 MiB chunks (1.4 to 3 launches a chunk, 256 items for 456 CTAs) took
 * 1630 us for 3.4 GB; one launch of parts 1370.
 * No block-wide barrier runs inside the loop.  Plain cp.async.bulk only: no tensor maps, no
 * multicast, one CTA's own shared memory.
 *
 * Every wait is bounded: a wait that runs out ends both loops; the CTA then waits (again
 * bounded) for the loads it issued but did not consume, and for its stores, and returns with
 * status word 2, or 3 if that drain ran out as well (a load may then still be in flight into
 * shared memory the CTA no longer owns).
 */
#include <cuda_runtime.h>
#include <stdint.h>

#include "cfa_device.cuh"
#include "cfa_internal.h"

namespace {

using cfa_dev::launch_begin;
using cfa_dev::launch_ctl;
using cfa_dev::launch_early;
using cfa_dev::launch_end;
using cfa_dev::vsum;
using cfa_dev::warp_sum;

constexpr int kThreads = 64; /* warp 0 loads, warp 1 checksums and stores */
constexpr int kStages = 2;
constexpr uint32_t kStageBytes = 32 * 1024;
constexpr uint32_t kSmemBytes = kStages * kStageBytes; /* 64 KiB: three CTAs per SM */
constexpr uint32_t kSpinLimit = 1u << 20;              /* try_wait polls before giving up */
constexpr uint32_t kLoseLoads = 1u << 31;              /* self-test: the loader issues nothing */

struct BulkArgs {
    cfa_bulk_range range[CFA_BULK_RANGES]; /* item lists that are not empty */
    uint32_t n_items;    /* parts over all ranges */
    uint32_t parts_log2; /* every item is copied in 2^parts_log2 parts */
    uint32_t spin_limit; /* try_wait polls before a wait gives up; the self-test sets a short one
                            and tells the loader to issue nothing (spin_limit | kLoseLoads) */
    uint64_t src_base;
    uint64_t src_period; /* 0, or P: blob byte o sits at src_base + (o mod P) */
    uint64_t src_lo, src_hi;
    unsigned long long *ck;
    int *status;
    cfa_launch_ctl ctl;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(smem_addr(bar)), "r"(parity)
                 : "memory");
    return done != 0;
}

/* Waits for phase `parity` of the barrier to complete; false if the spin limit ran out. */
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit)
{
    for (uint32_t k = 0; k < limit; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void bulk_load(void *smem, const void *gsrc, uint32_t bytes,
                                          uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
                 "[%0], [%1], %2, [%3];" ::"r"(smem_addr(smem)),
                 "l"(gsrc), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void bulk_store(void *gdst, const void *smem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst),
                 "r"(smem_addr(smem)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

__device__ __forceinline__ void bulk_wait_read_all_but_one()
{
    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}

__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

/* Adds the consumer warp's checksum to slot ck; all 32 lanes call it. */
__device__ __forceinline__ void warp_flush(uint64_t &acc, uint32_t ck, unsigned long long *out)
{
    const uint64_t v = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) atomicAdd(out + ck, v);
    acc = 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

/* An item of either kind: `rows` rows of `cols` elements, `stride` apart in the source and back to
 * back in the destination; a contiguous run is one row. */
struct BulkItem {
    uint64_t src, dst;
    uint32_t rows, cols, stride, ck, mode;
};

/* A bulk item is sound if it is a plain copy, its source lies inside the launch's readable range
 * and source, destination, rows and row distance are multiples of 16 bytes. */
__device__ __forceinline__ bool bulk_item_ok(const BulkItem &w, const BulkArgs &a)
{
    const uint32_t l = w.mode & 3u;
    const uint64_t row = (uint64_t)w.cols << l, pitch = (uint64_t)w.stride << l;
    const uint64_t total = row * w.rows; /* may wrap only when row alone is refused below */
    if (w.mode != CFA_MODE(l, l, 0) || w.rows == 0 || w.cols == 0 || pitch < row ||
        row >= (1ull << 31) || total >= (1ull << 31) ||
        ((w.src | w.dst | row | (w.rows > 1 ? pitch : 0) | a.src_base | a.src_period) & 15u) != 0)
        return false;
    /* row is 16 at least here, so there are fewer than 2^27 rows of a pitch below 2^35 */
    const uint64_t extent = (w.rows - 1) * pitch + row;
    return w.src >= a.src_lo && w.src <= a.src_hi && extent <= a.src_hi - w.src;
}

/* Bytes [*at, *at + *len) of a checked item of `total` bytes at destination `dst` that are part k
 * of its 2^parts_log2 equal parts (cut as in the vector kernel); false if the part is empty. */
__device__ __forceinline__ bool bulk_part(uint64_t dst, uint32_t total, uint32_t k,
                                          uint32_t parts_log2, uint32_t *at, uint32_t *len)
{
    *at = 0;
    *len = total;
    if (parts_log2 == 0) return true;
    uint32_t step = (total + (1u << parts_log2) - 1u) >> parts_log2;
    if (step < CFA_MIN_PART_BYTES) step = CFA_MIN_PART_BYTES;
    step = (step + CFA_PART_ALIGN - 1u) & ~(CFA_PART_ALIGN - 1u);
    const uint32_t lead = (uint32_t)(dst & (CFA_PART_ALIGN - 1u));
    const uint64_t a = k ? (uint64_t)k * step - lead : 0;
    const uint64_t b = (k + 1u) >> parts_log2 ? total : (uint64_t)(k + 1u) * step - lead;
    if (a >= total) return false;
    *at = (uint32_t)a;
    *len = (uint32_t)((b < total ? b : total) - a);
    return true;
}

/* A descriptor as it lies in memory (cfa_work, or cfa_swork with its fifth word).  It is fetched
 * one part ahead and decoded only when its part comes up: any arithmetic at the fetch, even a copy of
 * one of its words, would wait for the load there and then (8-bit checkpoint in 64 MiB chunks: 1244
 * us, now 1233). */
struct RawItem {
    uint64_t q[5];
    uint32_t rows;
};

template <bool ROWS>
__device__ __forceinline__ RawItem bulk_fetch(const BulkArgs &a, uint32_t v)
{
    uint32_t i = v >> a.parts_log2;
    int r = 0;
    while (i >= a.range[r].n) i -= a.range[r++].n;
    RawItem b;
    b.rows = ROWS ? a.range[r].rows : 0;
    const size_t bytes = b.rows ? sizeof(cfa_swork) : sizeof(cfa_work);
    const uint64_t *p = reinterpret_cast<const uint64_t *>(
        static_cast<const uint8_t *>(a.range[r].items) + i * bytes);
#pragma unroll
    for (int k = 0; k < 4; ++k) b.q[k] = __ldg(reinterpret_cast<const unsigned long long *>(p) + k);
    if (b.rows) b.q[4] = __ldg(reinterpret_cast<const unsigned long long *>(p) + 4);
    return b;
}

static_assert(sizeof(cfa_work) == 32 && sizeof(cfa_swork) == 40, "descriptor layouts");

template <bool ROWS> __device__ __forceinline__ BulkItem bulk_decode(const RawItem &b)
{
    BulkItem w;
    w.src = b.q[0];
    w.dst = b.q[1];
    if (ROWS && b.rows) {
        w.rows = (uint32_t)b.q[2];
        w.cols = (uint32_t)(b.q[2] >> 32);
        w.stride = (uint32_t)b.q[3];
        w.ck = (uint32_t)(b.q[3] >> 32);
        w.mode = (uint32_t)b.q[4];
    } else {
        w.rows = 1;
        w.cols = w.stride = (uint32_t)b.q[2];
        w.ck = (uint32_t)(b.q[2] >> 32);
        w.mode = (uint32_t)b.q[3];
    }
    return w;
}

/* Asks for the first stage of part v, a contiguous run, in L2.  An early launch does so for each
 * CTA's first part before it may read it: consecutive 64 MiB chunks, 3.4 GB, 1245 us without, 1228
 * so, 1264 with two parts, 1285 with three; 16 MiB chunks, 1.4 GB, 802, 790, 797, 789. */
template <bool ROWS>
__device__ __forceinline__ void bulk_ask(const BulkArgs &a, uint32_t v, const RawItem &raw)
{
    const BulkItem w = bulk_decode<ROWS>(raw);
    uint32_t at, len;
    if (!bulk_item_ok(w, a) || w.rows != 1 ||
        !bulk_part(w.dst, w.cols << (w.mode & 3u), v & ((1u << a.parts_log2) - 1u),
                   a.parts_log2, &at, &len))
        return;
    const uint64_t so = a.src_period ? w.src % a.src_period : w.src;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.src_base + so + at),
                 "r"(min(len, kStageBytes))
                 : "memory");
}

/* Sum of a staged sub-block's elements over this lane's vectors: eight independent shared loads
 * in flight, then the ragged rest. */
template <int ES>
__device__ __forceinline__ uint64_t stage_sum(const uint4 *v, uint32_t nv, uint32_t lane)
{
    uint64_t acc = 0;
    uint32_t i = lane;
    for (; i + 7 * 32 < nv; i += 8 * 32) {
        uint4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = v[i + u * 32];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += vsum<ES>(x[u]);
    }
    for (; i < nv; i += 32) acc += vsum<ES>(v[i]);
    return acc;
}

/* What the consumer needs of a staged sub-block; written by the producer before the load is
 * issued, published to the consumer by the stage's `full` barrier.  len == 0 ends the stream. */
struct StageMeta {
    uint64_t dst;
    uint32_t len;
    uint32_t ck;
    uint32_t log2es;
};

/* ROWS: some items are row blocks.  Launches without any (all but tensor-parallel ranks) have none
 * of that arithmetic on the loader's path (44 registers against 52). */
template <bool ROWS>
__global__ void __launch_bounds__(kThreads) cfa_bulk_kernel(const BulkArgs a)
{
    extern __shared__ __align__(128) uint8_t stage[];
    __shared__ __align__(8) uint64_t full[kStages];
    __shared__ __align__(8) uint64_t empty[kStages];
    __shared__ StageMeta meta[kStages];
    __shared__ volatile int aborted;
    __shared__ uint32_t n_issued, n_consumed;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        aborted = 0;
        n_issued = 0;
        n_consumed = 0;
    }
    launch_early(a.ctl);
    /* the loader's first two descriptors (the plan's own memory, written before any launch) are
     * on their way while the launch waits for what is before it on the stream */
    RawItem cur{}, nxt{};
    if (threadIdx.x == 0) {
        if (blockIdx.x < a.n_items) cur = bulk_fetch<ROWS>(a, blockIdx.x);
        /* The source is not to be read yet (the kernel before may still be writing it), but asking
         * for it in L2, where every write arrives, is harmless, and fills the time in which the
         * kernel before ends; first of all, so that it gets the most of that time (3.4 GB in 64 MiB
         * chunks 1231 us, 1242 behind the second descriptor's fetch). */
        if ((a.ctl.flags & CFA_LAUNCH_WAIT_FIRST) && blockIdx.x < a.n_items)
            bulk_ask<ROWS>(a, blockIdx.x, cur);
        if (blockIdx.x + gridDim.x < a.n_items) nxt = bulk_fetch<ROWS>(a, blockIdx.x + gridDim.x);
    }
    launch_begin(a.ctl);
    /* what the kernel before wrote is read by bulk copies (the async proxy) from here on */
    if (threadIdx.x == 0 && (a.ctl.flags & CFA_LAUNCH_EARLY))
        asm volatile("fence.proxy.async.global;" ::: "memory");
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t limit = a.spin_limit & ~kLoseLoads;

    if (threadIdx.x < 32) {
        /* producer: sub-block p goes to stage p mod kStages once sub-block p - kStages, the
         * stage's previous tenant, has been released.  The next item's descriptor is fetched
         * while the current item's sub-blocks are issued. */
        if (lane == 0) {
            /* part `it` is being issued from w, bytes [off, end) left; the descriptor of part
             * it + gridDim.x is in flight into nxt */
            BulkItem w = bulk_decode<ROWS>(cur);
            uint32_t it = blockIdx.x, p = 0, off = 0, end = 0;
            bool have = it < a.n_items;
            uint32_t it_n = it + gridDim.x;
            auto step = [&]() { /* move to the next part of this CTA */
                it = it_n;
                have = it < a.n_items;
                if (have) {
                    w = bulk_decode<ROWS>(nxt);
                    it_n = it + gridDim.x;
                    if (it_n < a.n_items) nxt = bulk_fetch<ROWS>(a, it_n);
                }
            };
            auto settle = [&]() { /* skip items that fail the checks, and empty parts */
                for (; have; step()) {
                    if (!bulk_item_ok(w, a)) {
                        atomicCAS(a.status, 0, 1);
                        continue;
                    }
                    uint32_t len;
                    if (bulk_part(w.dst, (w.rows * w.cols) << (w.mode & 3u),
                                  it & ((1u << a.parts_log2) - 1u), a.parts_log2, &off, &len)) {
                        end = off + len;
                        break;
                    }
                }
            };
            settle();
            for (;;) {
                const int s = p % kStages;
                if (a.spin_limit & kLoseLoads) break; /* self-test: nothing arrives on full */
                if (p >= kStages && !mbar_wait(&empty[s], ((p / kStages) - 1u) & 1u, limit)) {
                    aborted = 1;
                    break;
                }
                if (!have || aborted) { /* end marker: a plain arrive completes the phase */
                    meta[s].len = 0;
                    mbar_arrive(&full[s]);
                    break;
                }
                /* of short rows, whole ones: a stage then holds no part of a row */
                const uint32_t row = w.cols << (w.mode & 3u);
                uint32_t len = kStageBytes;
                if (w.rows > 1 && row <= kStageBytes) {
                    const uint32_t in = off % row;
                    len = (kStageBytes + in) / row * row - in;
                }
                len = min(len, end - off);
                meta[s].dst = w.dst + off;
                meta[s].len = len;
                meta[s].ck = w.ck;
                meta[s].log2es = w.mode & 3u;
                mbar_expect_tx(&full[s], len);
                const uint64_t so = a.src_period ? w.src % a.src_period : w.src;
                const uint8_t *src = reinterpret_cast<const uint8_t *>(a.src_base + so);
                if (w.rows == 1) {
                    bulk_load(stage + s * kStageBytes, src + off, len, &full[s]);
                } else {
                    /* the rows, and parts of rows, under [off, off + len), back to back */
                    uint32_t r = off / row, c = off - r * row;
                    for (uint32_t at = 0; at < len; ++r, c = 0) {
                        const uint32_t k = min(row - c, len - at);
                        bulk_load(stage + s * kStageBytes + at,
                                  src + ((uint64_t)r * w.stride << (w.mode & 3u)) + c, k,
                                  &full[s]);
                        at += k;
                    }
                }
                ++p;
                n_issued = p;
                off += len;
                if (off >= end) {
                    step();
                    settle();
                }
            }
        }
    } else {
        /* consumer: checksum and store sub-block c, then release the stage of c - 1 */
        uint64_t acc = 0;
        uint32_t acc_ck = CFA_NO_CK;
        uint32_t c = 0;
        for (;; ++c) {
            const int s = c % kStages;
            const bool ok = mbar_wait(&full[s], (c / kStages) & 1u, limit);
            if (__any_sync(0xFFFFFFFFu, !ok)) {
                if (lane == 0) aborted = 1;
                break;
            }
            const StageMeta m = meta[s];
            if (m.len == 0) break;
            if (m.ck != acc_ck) {
                if (acc_ck != CFA_NO_CK) warp_flush(acc, acc_ck, a.ck);
                acc_ck = m.ck;
            }
            if (m.ck != CFA_NO_CK) {
                const uint4 *v = reinterpret_cast<const uint4 *>(stage + s * kStageBytes);
                const uint32_t nv = m.len >> 4;
                switch (m.log2es) {
                case 0: acc += stage_sum<1>(v, nv, lane); break;
                case 1: acc += stage_sum<2>(v, nv, lane); break;
                case 2: acc += stage_sum<4>(v, nv, lane); break;
                default: acc += stage_sum<8>(v, nv, lane); break;
                }
            }
            if (lane == 0) {
                bulk_store(reinterpret_cast<uint8_t *>(m.dst), stage + s * kStageBytes, m.len);
                bulk_commit();
                /* the store of c - 1 has read its stage, and every lane finished summing it
                 * before the __syncwarp that ended iteration c - 1 */
                bulk_wait_read_all_but_one();
                if (c >= 1) mbar_arrive(&empty[(c - 1) % kStages]);
            }
            __syncwarp();
        }
        if (acc_ck != CFA_NO_CK) warp_flush(acc, acc_ck, a.ck);
        if (lane == 0) {
            bulk_wait_all();
            n_consumed = c;
        }
    }
    __syncthreads();
    if (aborted && threadIdx.x == 0) {
        /* loads issued but not consumed: wait for them (bounded) before shared memory goes.  If
         * one of these waits runs out too, the CTA leaves with a bulk load that may still write
         * into shared memory it no longer owns: status 3 (over 1 and 2) tells the host that the
         * context is suspect, not merely that a wait timed out */
        bool drained = true;
        for (uint32_t k = n_consumed; k < n_issued && drained; ++k)
            drained = mbar_wait(&full[k % kStages], (k / kStages) & 1u, limit);
        if (drained) atomicCAS(a.status, 0, 2);
        else atomicMax(a.status, 3);
    }
    launch_end(a.ctl);
}

} // namespace

/* Resident CTAs per SM of the bulk kernel (0 if it cannot run). */
extern "C" int cfa_bulk_blocks_per_sm(void)
{
    int least = 0;
    for (int rows = 0; rows < 2; ++rows) {
        void (*fn)(const BulkArgs) = rows ? cfa_bulk_kernel<true> : cfa_bulk_kernel<false>;
        int n = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemBytes) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kThreads, kSmemBytes) !=
                cudaSuccess)
            return 0;
        least = rows && least < n ? least : n;
    }
    return least;
}

/* Launches the bulk unpack over up to CFA_BULK_RANGES lists of items whose source, destination and
 * byte length are multiples of 16, cut into parts as `cut` says; grid_cap bounds the persistent
 * grid. */
extern "C" cudaError_t cfa_launch_bulk(const cfa_bulk_range *ranges, uint32_t n_ranges,
                                       uint64_t src_base, uint64_t src_period,
                                       uint64_t src_lo, uint64_t src_hi,
                                       unsigned long long *ck, int *status, int grid_cap,
                                       const cfa_cut *cut, const cfa_launch_ctl *ctl,
                                       cudaStream_t stream)
{
    if (n_ranges > CFA_BULK_RANGES || grid_cap <= 0) return cudaErrorInvalidValue;
    BulkArgs a{};
    uint64_t n_items = 0;
    bool rows = false;
    for (uint32_t r = 0, k = 0; r < n_ranges; ++r) {
        if (!ranges[r].n) continue;
        a.range[k++] = ranges[r];
        rows |= ranges[r].rows != 0;
        n_items += ranges[r].n;
    }
    if (n_items == 0) return cudaSuccess;
    if (n_items >= CFA_MOST_VISITS) return cudaErrorInvalidValue;
    a.parts_log2 = cfa_parts_log2(cut, n_items, (uint32_t)grid_cap);
    a.n_items = (uint32_t)n_items << a.parts_log2;
    a.spin_limit = kSpinLimit;
    a.src_base = src_base;
    a.src_period = src_period;
    a.src_lo = src_lo;
    a.src_hi = src_hi;
    a.ck = ck;
    a.status = status;
    const uint32_t grid = a.n_items < (uint32_t)grid_cap ? a.n_items : (uint32_t)grid_cap;
    a.ctl = ctl ? *ctl : cfa_launch_ctl{};
    return launch_ctl(rows ? cfa_bulk_kernel<true> : cfa_bulk_kernel<false>, grid, kThreads,
                      kSmemBytes, stream, a);
}

/* Self-test of the bounded waits: one CTA of the TMA kernel over one valid 16-byte item, with a
 * short wait limit and its loader told to issue nothing, so the consumer's first wait on `full`
 * runs out.  The kernel must flag the status word (2) and return; the context stays usable. */
extern "C" cudaError_t cfa_bulk_selftest_timeout(int *status_host)
{
    cfa_work *d_item = nullptr;
    uint8_t *d_buf = nullptr;
    unsigned long long *d_ck = nullptr;
    int *d_status = nullptr;
    cudaError_t e = cudaSuccess;
    if (!status_host) return cudaErrorInvalidValue;
    *status_host = -1;
    if ((e = cudaFuncSetAttribute(cfa_bulk_kernel<false>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)kSmemBytes)) != cudaSuccess)
        return e;
    if ((e = cudaMalloc(&d_item, sizeof(cfa_work))) != cudaSuccess) goto out;
    if ((e = cudaMalloc(&d_buf, 512)) != cudaSuccess) goto out;
    if ((e = cudaMalloc(&d_ck, sizeof(unsigned long long))) != cudaSuccess) goto out;
    if ((e = cudaMalloc(&d_status, sizeof(int))) != cudaSuccess) goto out;
    {
        cfa_work w{};
        w.src = 0;
        w.dst = (uint64_t)(uintptr_t)(d_buf + 256);
        w.n = 8; /* 16 bytes of 16-bit elements */
        w.ck = 0;
        w.mode = CFA_MODE(1, 1, 0);
        if ((e = cudaMemcpy(d_item, &w, sizeof w, cudaMemcpyHostToDevice)) != cudaSuccess) goto out;
        if ((e = cudaMemset(d_status, 0, sizeof(int))) != cudaSuccess) goto out;
        if ((e = cudaMemset(d_ck, 0, sizeof(unsigned long long))) != cudaSuccess) goto out;
        BulkArgs a{};
        a.range[0] = cfa_bulk_range{d_item, 1, 0};
        a.n_items = 1;
        a.spin_limit = 256u | kLoseLoads;
        a.src_base = (uint64_t)(uintptr_t)d_buf;
        a.src_period = 0;
        a.src_lo = 0;
        a.src_hi = 256;
        a.ck = d_ck;
        a.status = d_status;
        cfa_bulk_kernel<false><<<1, kThreads, kSmemBytes>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) goto out;
        if ((e = cudaDeviceSynchronize()) != cudaSuccess) goto out;
        e = cudaMemcpy(status_host, d_status, sizeof(int), cudaMemcpyDeviceToHost);
    }
out:
    if (d_item) cudaFree(d_item);
    if (d_buf) cudaFree(d_buf);
    if (d_ck) cudaFree(d_ck);
    if (d_status) cudaFree(d_status);
    return e;
}
