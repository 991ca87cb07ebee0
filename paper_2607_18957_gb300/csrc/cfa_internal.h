/*
 * Internal structures shared by the host plan builder (cfa_plan.c), the kernels
 * (cfa_unpack.cu) and the runtime (cfa_runtime.cu).  Not part of the C ABI.
 */
#ifndef CFA_INTERNAL_H
#define CFA_INTERNAL_H

#include <stddef.h>
#include <stdint.h>

#include "cfa.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * One unit of GPU work: a contiguous run of elements of one piece (tensor x chunk).
 * 32 bytes, read once per work item.
 *   src   blob byte offset of the first source element (the launch adds its source base)
 *   dst   device address of the first destination element
 *   n     element count
 *   ck    checksum slot (the entry index), or CFA_NO_CK
 *   mode  bits 0-1: log2 of the source element size; bits 2-3: log2 of the destination element
 *         size; bit 4: fp32 -> bf16 round-to-nearest-even cast
 */
typedef struct cfa_work {
    uint64_t src;
    uint64_t dst;
    uint32_t n;
    uint32_t ck;
    uint32_t mode;
    uint32_t pad;
} cfa_work;

/*
 * A block of rows of a strided piece (a column slice of a larger checkpoint tensor): row k
 * starts at source blob offset src + k * stride * (source element size) and lands at
 * dst + k * cols * (destination element size).  40 bytes.
 */
/* Warp-level work items hold at most this many destination bytes (the plan cuts tiny pieces at
 * destination addresses that are multiples of it): one 8-lane warp segment copies one item. */
#define CFA_TINY_SEG_BYTES 512u

typedef struct cfa_swork {
    uint64_t src;
    uint64_t dst;
    uint32_t rows;
    uint32_t cols;   /* elements per row */
    uint32_t stride; /* source elements between row starts */
    uint32_t ck;
    uint32_t mode;
    uint32_t cls;    /* work class, used while the plan is built */
} cfa_swork;

/* Column slices whose rows hold at least this many bytes, and start and lie at multiples of 16,
 * go to the TMA kernel (one bulk load a row).  Shorter rows stay with the vector kernel's warps: a
 * tensor-parallel rank whose attention slices have rows of 2 KiB took 540 us with those rows
 * there and 556 with them loaded one by one; with rows of 14-28 KiB on the vector kernel another
 * took 135, and with TMA loads 110. */
#define CFA_BULK_ROW_BYTES 4096u

/* One of the item lists of a bulk launch: the contiguous runs (cfa_work), or the row blocks
 * (cfa_swork), of one element size. */
typedef struct cfa_bulk_range {
    const void *items;
    uint32_t n;
    uint32_t rows; /* 1: cfa_swork */
} cfa_bulk_range;
#define CFA_BULK_RANGES 8

/*
 * A host->device copy of one chunk: `rows` runs of `width` bytes, `pitch` bytes apart, the first
 * at blob offset `src`; it lands at the same offset inside the chunk's device slot.
 */
typedef struct cfa_copy {
    uint64_t src;
    uint64_t width;
    uint64_t pitch;
    uint64_t rows;
} cfa_copy;

#define CFA_NO_CK 0xFFFFFFFFu

/* Element conversions (cfa_work.mode bits 4-7, cfa_piece.conv). */
#define CFA_CONV_NONE 0
#define CFA_CONV_F32_BF16 1
#define CFA_CONV_F32_F16 2
#define CFA_CONV_F16_BF16 3
#define CFA_CONV_BF16_F32 4
#define CFA_CONV_F16_F32 5
#define CFA_N_CONV 6

/* Work classes: one specialised kernel each.  0..3 = plain copy of 1, 2, 4, 8-byte elements;
 * 3 + conv = conversion `conv`. */
#define CFA_N_CLASSES 9
#define CFA_CLASS_OF_CONV(conv) (3 + (conv))
#define CFA_MODE(src_log2, dst_log2, conv) \
    ((uint32_t)(src_log2) | ((uint32_t)(dst_log2) << 2) | ((uint32_t)(conv) << 4))
#define CFA_MODE_CONV(mode) (((mode) >> 4) & 15u)

/* Whether a work class reads twice what it writes. */
static inline int cfa_class_narrows(int cls)
{
    return cls == CFA_CLASS_OF_CONV(CFA_CONV_F32_BF16) ||
           cls == CFA_CLASS_OF_CONV(CFA_CONV_F32_F16);
}

/* Conversion for a (source, destination) dtype pair, 0 if the pair has none. */
static inline int cfa_conversion(int32_t src, int32_t dst)
{
    if (src == CFA_DTYPE_F32 && dst == CFA_DTYPE_BF16) return CFA_CONV_F32_BF16;
    if (src == CFA_DTYPE_F32 && dst == CFA_DTYPE_F16) return CFA_CONV_F32_F16;
    if (src == CFA_DTYPE_F16 && dst == CFA_DTYPE_BF16) return CFA_CONV_F16_BF16;
    if (src == CFA_DTYPE_BF16 && dst == CFA_DTYPE_F32) return CFA_CONV_BF16_F32;
    if (src == CFA_DTYPE_F16 && dst == CFA_DTYPE_F32) return CFA_CONV_F16_F32;
    return CFA_CONV_NONE;
}

/* Host side of a plan: everything cfa_plan_create computes before touching the GPU. */
typedef struct cfa_host_plan {
    cfa_plan_opts opts;
    uint64_t blob_bytes;
    uint64_t chunk_bytes;
    uint32_t n_chunks;
    uint32_t n_layers;
    size_t n_entries, n_dsts;
    cfa_tensor_entry *entries; /* copies; names point into `names` */
    char **names;
    cfa_dst *dsts;
    cfa_piece *pieces; /* sorted by (chunk, src offset) */
    size_t n_pieces;
    /* work items ordered by (class, chunk): class k of chunk c owns
     * [first[k * (n_chunks + 1) + c], first[k * (n_chunks + 1) + c + 1]) of each array, so the
     * items of one class over a run of chunks are contiguous; the `units` beside slabs, bulk and
     * brows count the bytes before each of those bounds (source or destination bytes, whichever
     * is more) in whole CFA_MIN_PART_BYTES */
    cfa_work *slabs; /* block-level, LSU vector path */
    size_t n_slabs;
    uint32_t *slab_first, *slab_units;
    cfa_work *bulk;  /* block-level, TMA bulk path (cast-free, 16-byte aligned) */
    size_t n_bulk;
    uint32_t *bulk_first, *bulk_units;
    cfa_work *tiny;  /* warp-level */
    size_t n_tiny;
    uint32_t *tiny_first;
    cfa_swork *strided; /* block-level, rows of column slices */
    size_t n_strided;
    uint32_t *strided_first;
    cfa_swork *brows; /* the same for the TMA path (cast-free, 16-byte aligned) */
    size_t n_brows;
    uint32_t *brows_first, *brows_units;
    int64_t *layer_last_chunk; /* n_layers; -1 = the group has no bytes */
    cfa_copy *copies;          /* what each chunk's pieces read: chunk c owns
                                  [copy_first[c], copy_first[c + 1]) */
    size_t n_copies;
    uint32_t *copy_first;
    uint64_t staged_bytes;
    uint32_t part_bytes; /* a launch over the whole load cuts its slabs to; 0: leaves them whole */
    uint64_t bytes_read, bytes_written;
    int any_cksum;
} cfa_host_plan;

/*
 * Block-level items are cut once more at launch: into 2^cfa_parts_log2 equal parts each, cut where
 * the destination is a multiple of CFA_PART_ALIGN, so that the parts of an item of the caller's usual
 * size, cut->item_bytes, hold part_bytes or more (source or destination bytes, whichever is more; a
 * smaller item has fewer parts, none below CFA_MIN_PART_BYTES).  The plan's slabs, and the no-alloc
 * entry point's 2 MiB items, are few and large for the sake of their descriptors; a launch over one
 * chunk or a small checkpoint would leave most CTAs without work, and large items spread the
 * addresses in flight over too much memory (cfa_auto_part).  A chunk's items go down to 32 KiB.
 * The no-alloc items stop at 64 KiB: fp32 -> bf16, 252 MB, 118 us so, 125 with 32 KiB parts; 945 MB
 * 417 and 429; bf16, 1.1 GB, 673 with 64 KiB, 680 with 128, 686 with 512.
 *
 * The kernels visit 2^k parts of every item, and the surplus parts of an item smaller than
 * item_bytes are empty: each costs a CTA a descriptor fetch and the checks.  So k also depends on
 * what the launch holds, n_items items of cut->bytes in all: visits beyond one per CTA of a full
 * grid stay within 3/2 of the parts that the bytes would fill.  Full items are cut as their size
 * says; items below the part size on average are not cut.  With k from item_bytes alone 16,000
 * tensors of 8 to 64 KiB took 1149 us through the no-alloc entry point (k = 5), 416 at k = 0, and
 * as many of 8 to 32 KiB, in chunks of a plan with 64 MiB slabs (k = 11), 37 ms and 0.13.
 */
#define CFA_MIN_PART_BYTES 32768u
#define CFA_PART_ALIGN 128u
#define CFA_MOST_VISITS (1ull << 31) /* the kernels count visits in 32 bits */
typedef struct cfa_cut {
    uint64_t item_bytes; /* of the caller's usual item */
    uint64_t bytes;      /* of all block-level items of the launch */
    uint32_t part_bytes; /* 0: whole items */
} cfa_cut;

static inline uint32_t cfa_parts_log2(const cfa_cut *cut, uint64_t n_items, uint32_t grid)
{
    const uint64_t part_bytes = cut->part_bytes;
    if (part_bytes == 0) return 0;
    const uint64_t filled = cut->bytes / part_bytes;
    uint64_t most = filled + filled / 2;
    uint32_t k = 0;
    if (most < grid) most = grid;
    if (most >= CFA_MOST_VISITS) most = CFA_MOST_VISITS - 1;
    while ((cut->item_bytes >> (k + 1)) >= part_bytes && (n_items << (k + 1)) <= most) ++k;
    return k;
}

/*
 * How a kernel launch follows the one before it on its stream (programmatic dependent launch),
 * and what it clears before its work.
 *   EARLY       may start once the kernel before it on the stream has released its dependents
 *               (launch attribute) instead of after it has ended
 *   WAIT_FIRST  the kernel waits for the end of everything before it on the stream before it reads
 *               a source, writes, or releases its own dependents
 *   WAIT_LAST   the kernel does not need the one before it (they write disjoint bytes and add
 *               checksums atomically) but ends only after it, so that whatever follows on the
 *               stream follows both
 *   RELEASE     the kernel releases its dependents as soon as its CTAs run; never set on the last
 *               kernel of a call, whose dependents are the caller's: a kernel of theirs with the
 *               launch attribute starts when the CTAs of a call's last kernel have ended, as after
 *               any kernel that does not release
 * clear: words set to zero by this launch (the checksum half of the next load), or NULL.
 */
#define CFA_LAUNCH_EARLY 1u
#define CFA_LAUNCH_WAIT_FIRST 2u
#define CFA_LAUNCH_WAIT_LAST 4u
#define CFA_LAUNCH_RELEASE 8u
typedef struct cfa_launch_ctl {
    unsigned long long *clear;
    uint64_t clear_words;
    uint32_t flags;
    uint32_t pad;
} cfa_launch_ctl;

/* Flags of kernel i of the n that a call launches one after the other on a stream, all independent
 * of one another.  early: the first is launched with the attribute as well, and waits inside. */
static inline uint32_t cfa_chain_flags(uint32_t i, uint32_t n, int early)
{
    uint32_t f = 0;
    if (i > 0) f |= CFA_LAUNCH_EARLY | CFA_LAUNCH_WAIT_LAST;
    else if (early) f |= CFA_LAUNCH_EARLY | CFA_LAUNCH_WAIT_FIRST;
    if (i + 1 < n) f |= CFA_LAUNCH_RELEASE;
    return f;
}

/* Sets the calling thread's detail string returned by cfa_last_error(NULL). */
void cfa_internal_set_error(const char *msg);

cfa_status cfa_host_plan_build(const cfa_tensor_entry *entries, size_t n_entries,
                               const cfa_dst *dsts, size_t n_dsts, uint64_t blob_bytes,
                               const cfa_plan_opts *opts, cfa_host_plan *out, char *err,
                               size_t errlen);
void cfa_host_plan_free(cfa_host_plan *hp);
int cfa_dtype_size(int32_t dtype);

#ifdef __cplusplus
}
#endif

#endif /* CFA_INTERNAL_H */
