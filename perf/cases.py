"""Loads that a user of the checkpoint loader makes, for measuring.

A case names a checkpoint (its tensors, their types, how they are packed in the blob, the part
of it that this GPU holds) and the way it is loaded.  Every case keeps the loader's plan in
`prepare`, as an engine that loads the same parameters again (new weights, another adapter, a
model swapped back in) does, and makes one load in `run`.

    kind      adapter   pairs of low-rank matrices per layer
              vectors   1-D tensors of log-uniform sizes, in a shuffled order
              dense     a decoder-only transformer: embedding, per layer q/k/v (fused), o,
                        gate/up (fused), down, two norms; final norm, head
              moe       the same attention, a router and experts stacked per layer (w1/w3 fused,
                        w2), and optionally small extra tensors
              fp8       dense with 8-bit weights and one fp32 scale per 128 x 128 block
    src, dst  element types in the checkpoint and of the parameters (different: converted)
    align     every tensor starts at a multiple of it in the blob, plus up to `gap` elements
    tp, rank  tensor-parallel rank: row ranges and column slices of the checkpoint's tensors
    ep, rank  expert-parallel rank: whole experts
    how       device    the blob is in device memory; the load is enqueued on the current stream
              verify    the same, and the caller waits and reads the checksums
              chunks    the blob is in device memory and is unpacked chunk by chunk, as by an
                        engine that stages the chunks itself
              noalloc   the C entry point that needs no plan and allocates nothing
              pinned    the blob is in page-locked host memory; the caller waits and reads the
                        checksums
              pageable  the same from ordinary host memory

Copied parameters are compared as the 64-bit words that they fill, converted ones as numbers.
"""
import ctypes
import functools
import math

import numpy as np
import torch

import paper_2607_18957_gb300 as cfa

SIZE = {"u8": 1, "bf16": 2, "f16": 2, "f32": 4}
TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}

# A decoder of 8 billion parameters and one of 70 billion, as the benchmark has them; cases set
# the number of layers.
DENSE_8B = {"hidden": 4096, "heads": 32, "kv": 8, "head_dim": 128, "inter": 14336,
            "vocab": 128256}
DENSE_70B = {"hidden": 8192, "heads": 64, "kv": 8, "head_dim": 128, "inter": 28672,
             "vocab": 128256}
MOE = {"hidden": 4096, "heads": 32, "kv": 8, "head_dim": 128, "inter": 14336, "vocab": 32000,
       "experts": 8}


def case(name, kind, how, src="bf16", dst=None, align=256, gap=0, **kw):
    c = {"kind": kind, "how": how, "src": src, "dst": dst or src, "align": align, "gap": gap}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # the smallest load: one adapter's rank-16 pairs for four projections are swapped in and
        # checked before the request that needs them starts
        case("adapter", "adapter", "verify", layers=1, targets=4, rank_dim=16, width=4096),
        # a checkpoint of 1,000 small tensors, 256 B to 1 MiB (about 130 MB): fits the L2 cache
        case("vectors_1000", "vectors", "device", n=1000, lo=256, hi=1 << 20),
        # the small extra tensors of an MoE checkpoint on their own: 200,000 of 4 B to 4 KiB
        case("vectors_200k", "vectors", "device", n=200_000, lo=4, hi=4096),
        # the whole 8B checkpoint, already in device memory (16 GB): weights handed over on the GPU
        case("dense_bf16", "dense", "device", layers=32, **DENSE_8B),
        # an fp32 checkpoint converted on the way in, tensors at 256-byte offsets
        case("dense_f32_bf16", "dense", "device", "f32", "bf16", layers=8, **DENSE_8B),
        # fp32 tensors back to back at 4-byte offsets, as a file whose tensors have odd sizes
        case("dense_f32_bf16_odd", "dense", "device", "f32", "bf16", align=4, gap=3, layers=4,
             **DENSE_8B),
        # bf16 tensors back to back at 2-byte offsets
        case("dense_bf16_odd", "dense", "device", align=2, gap=7, layers=8, **DENSE_8B),
        # rank 3 of 8 of a tensor-parallel engine: row ranges and column slices
        case("dense_tp8", "dense", "device", layers=6, tp=8, rank=3, **DENSE_70B),
        # rank 5 of 8 of an expert-parallel engine, with small extra tensors replicated
        case("moe_ep8", "moe", "device", layers=6, ep=8, rank=5, extras=30_000, **MOE),
        # 8-bit weights and block scales, unpacked chunk by chunk from the engine's own staging
        case("fp8_chunks", "fp8", "chunks", "u8", chunk_mib=64, layers=6, **DENSE_8B),
        # a cold start from page-locked memory with the default chunks, checked at the end
        case("dense_pinned", "dense", "pinned", chunk_mib=512, layers=4,
             **dict(DENSE_8B, vocab=32000)),
        # an engine that may not allocate: the blob is on the GPU, its own memory is all taken
        case("dense_noalloc", "dense", "noalloc", layers=4, **dict(DENSE_8B, vocab=32000)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    packed = rng.choice([{"align": 256, "gap": 0}, {"align": 256, "gap": 0},
                         {"align": 16, "gap": 0}, {"align": 8, "gap": 0},
                         {"align": 4, "gap": 3}])
    kind = rng.choice(["adapter", "vectors", "dense", "dense", "convert", "convert", "tp", "moe",
                       "fp8", "staged", "noalloc"])
    head_dim = rng.choice([64, 80, 96, 128])
    kv = rng.choice([1, 2, 4, 8])
    heads = kv * rng.choice([1, 2, 4, 8])
    shape = {"hidden": 8 * _log(rng, 64, 1024), "heads": heads, "kv": kv, "head_dim": head_dim,
             "inter": 8 * _log(rng, 128, 3584), "vocab": _log(rng, 1000, 128256)}

    def layers(most_bytes, es=2, **kw):
        """As many layers, up to 32, as a random share of most_bytes of checkpoint holds."""
        budget = most_bytes * math.exp(rng.uniform(math.log(0.02), 0.0))
        h, per = shape["hidden"], (2 * heads + 2 * kv) * head_dim
        mats = 3 * shape["inter"] * kw.get("experts", 1)
        return max(1, min(32, int((budget / es - 2 * h * shape["vocab"]) / (h * (per + mats)))))

    if kind == "adapter":
        return case(None, "adapter", rng.choice(["verify", "device"]), src=rng.choice(["bf16", "f16"]),
                    layers=_log(rng, 1, 64), targets=rng.randint(1, 7),
                    rank_dim=rng.choice([4, 8, 16, 32, 64, 11]), width=_log(rng, 512, 8192),
                    **packed)
    if kind == "vectors":
        hi = _log(rng, 1 << 10, 1 << 20)
        return case(None, "vectors", rng.choice(["device", "device", "verify"]),
                    src=rng.choice(["bf16", "bf16", "f32"]),
                    n=min(_log(rng, 100, 200_000), (200 << 20) // hi * 8), lo=rng.choice([4, 64, 256]),
                    hi=hi, **packed)
    if kind == "dense":
        return case(None, "dense", "device", layers=layers(16e9), **packed, **shape)
    if kind == "convert":
        src, dst = rng.choice([("f32", "bf16"), ("f32", "bf16"), ("f32", "f16"), ("f16", "bf16"),
                               ("bf16", "f32")])
        return case(None, "dense", "device", src, dst, layers=layers(8e9, SIZE[src]), **packed,
                    **shape)
    if kind == "tp":
        tp = rng.choice([2, 4, 8])
        s = dict(shape, heads=8 * rng.choice([2, 4, 8]), kv=8, inter=shape["inter"] // 8 * 8 * 8,
                 vocab=shape["vocab"] // 8 * 8)
        s["inter"] = min(s["inter"], 28672)
        return case(None, "dense", "device", layers=rng.randint(1, 6), tp=tp,
                    rank=rng.randrange(tp), **packed, **s)
    if kind == "moe":
        ep = rng.choice([1, 2, 4, 8])
        e = 8 * rng.choice([1, 2])
        s = dict(shape, inter=min(shape["inter"], 8192), experts=e)
        return case(None, "moe", "device", layers=min(6, layers(8e9, experts=e)), ep=ep,
                    rank=rng.randrange(ep), extras=rng.choice([0, _log(rng, 100, 50_000)]),
                    **packed, **s)
    if kind == "fp8":
        s = dict(shape, head_dim=128)
        s["inter"] = max(128, s["inter"] // 128 * 128)
        return case(None, "fp8", rng.choice(["device", "chunks"]), "u8", align=256,
                    layers=layers(6e9, 1), chunk_mib=_log(rng, 16, 512), **s)
    if kind == "staged":
        return case(None, "dense", rng.choice(["pinned", "pinned", "pageable"]),
                    chunk_mib=rng.choice([16, 64, 128, 512, 512]), layers=layers(2e9), **packed,
                    **dict(shape, vocab=min(shape["vocab"], 32000)))
    src, dst = rng.choice([("bf16", "bf16"), ("bf16", "bf16"), ("f32", "bf16")])
    return case(None, "dense", "noalloc", src, dst, layers=layers(2e9, SIZE[src]), **packed, **shape)


# ---- the checkpoint and the parameters ---------------------------------------------------------

class Layout:
    """Where every tensor lies in the blob and in the engine's parameters, by column.  The
    parameters lie in one buffer, each at a multiple of 256 bytes."""

    def __init__(self, c):
        self.rng = np.random.default_rng(17)
        self.align, self.gap, self.blob = c["align"], c["gap"], 0
        self.src, self.dst = c["src"], c["dst"]
        self.rows = []      # (dtype, shape, offset, dst, row, stride, layer)
        self.params = []    # (dtype, shape)
        getattr(self, c["kind"])(c)
        if c["kind"] != "vectors":
            dts, shapes, off, d, row, stride, layer = zip(*self.rows)
            self.dtype, self.offset, self.d = list(dts), np.array(off, np.uint64), np.array(d)
            self.row, self.stride, self.layer = np.array(row), np.array(stride), np.array(layer)
            self.shape = (np.zeros((len(shapes), 8), np.int64),
                          np.array([len(s) for s in shapes], np.int32))
            for i, s in enumerate(shapes):
                self.shape[0][i, :len(s)] = s
            self.p_dtype = [p[0] for p in self.params]
            self.p_shape = (np.zeros((len(self.params), 8), np.int64),
                            np.array([len(p[1]) for p in self.params], np.int32))
            for i, p in enumerate(self.params):
                self.p_shape[0][i, :len(p[1])] = p[1]
        dims = np.arange(8)[None, :]
        self.numel = np.where(dims < self.shape[1][:, None], self.shape[0], 1).prod(axis=1)
        p_numel = np.where(dims < self.p_shape[1][:, None], self.p_shape[0], 1).prod(axis=1)
        p_bytes = p_numel * np.array([SIZE[t] for t in self.p_dtype])
        room = (p_bytes + 255) // 256 * 256
        self.p_offset = np.cumsum(room) - room
        self.out_bytes = int(room.sum())
        self.blob_bytes = (self.blob + 255) // 256 * 256
        self.read_bytes = int((self.numel * np.array([SIZE[t] for t in self.dtype])).sum())
        self.written_bytes = int(p_bytes.sum())

    def param(self, dtype, *shape):
        self.params.append((dtype, shape))
        return len(self.params) - 1

    def tensor(self, dtype, shape, dst, row=0, layer=0, rows=None, cols=None):
        """A checkpoint tensor of `shape`, loaded into parameter dst at `row`: all of it, its
        rows [a, b) or its columns [a, b).  dst None: in the blob, but not loaded here."""
        es = SIZE[dtype]
        at = -(-self.blob // max(self.align, es)) * max(self.align, es)
        at += es * int(self.rng.integers(0, self.gap + 1)) if self.gap else 0
        self.blob = at + es * int(np.prod(shape, dtype=np.int64))
        if dst is None:
            return
        stride = 0
        if rows:
            at += es * rows[0] * int(np.prod(shape[1:], dtype=np.int64))
            shape = (rows[1] - rows[0],) + tuple(shape[1:])
        elif cols:
            at += es * cols[0]
            stride = shape[-1] if shape[0] > 1 else 0
            shape = tuple(shape[:-1]) + (cols[1] - cols[0],)
        self.rows.append((dtype, tuple(shape), at, dst, row, stride, layer))

    def adapter(self, c):
        for l in range(c["layers"]):
            for _ in range(c["targets"]):
                for shape in ((c["rank_dim"], c["width"]), (c["width"], c["rank_dim"])):
                    self.tensor(self.src, shape, self.param(self.dst, *shape), layer=l)

    def vectors(self, c):
        """Columns made at once: there can be 200,000 of them."""
        n, es = c["n"], SIZE[self.src]
        sizes = np.exp(self.rng.uniform(math.log(c["lo"]), math.log(c["hi"]), size=n))
        nel = np.maximum(1, sizes.astype(np.int64) // es)
        order = self.rng.permutation(n)
        a = max(self.align, es)
        room = (nel[order] * es + self.gap * es + a - 1) // a * a
        shift = es * self.rng.integers(0, self.gap + 1, size=n) if self.gap else 0
        self.offset = np.zeros(n, np.uint64)
        self.offset[order] = (np.cumsum(room) - room + shift).astype(np.uint64)
        self.blob = int(room.sum())
        self.dtype, self.p_dtype = [self.src] * n, [self.dst] * n
        one = np.zeros((n, 8), np.int64)
        one[:, 0] = nel
        self.shape = self.p_shape = (one, np.ones(n, np.int32))
        self.d, zero = np.arange(n), np.zeros(n, np.int64)
        self.row = self.stride = self.layer = zero

    def attention(self, c, l, w):
        """q/k/v (row ranges) and o (a column range) of layer l; fewer kv heads than ranks:
        each rank holds a replica of its head."""
        h, hd, tp, r = c["hidden"], c["head_dim"], c.get("tp", 1), c.get("rank", 0)
        q = c["heads"] * hd
        qr = (r * q // tp, (r + 1) * q // tp) if tp > 1 else (0, q)
        k0 = r * c["kv"] // tp
        kr = (k0 * hd, (k0 + max(1, c["kv"] // tp)) * hd) if tp > 1 else (0, c["kv"] * hd)
        nq, nk = qr[1] - qr[0], kr[1] - kr[0]
        d = self.param(w(self.dst), nq + 2 * nk, h)
        self.weight(w, (q, h), d, 0, l, rows=qr if tp > 1 else None)
        for i in range(2):
            self.weight(w, (c["kv"] * hd, h), d, nq + i * nk, l, rows=kr if tp > 1 else None)
        self.weight(w, (h, q), self.param(w(self.dst), h, nq), 0, l, cols=qr if tp > 1 else None)

    def weight(self, w, shape, dst, row, layer, **kw):
        self.tensor(w(self.src), shape, dst, row, layer, **kw)

    def dense(self, c, same=lambda t: t):
        h, i, v, tp, r = c["hidden"], c["inter"], c["vocab"], c.get("tp", 1), c.get("rank", 0)
        vr = (r * v // tp, (r + 1) * v // tp)
        ir = (r * i // tp, (r + 1) * i // tp)
        part = tp > 1
        last = c["layers"] + 1
        self.tensor(self.src, (v, h), self.param(self.dst, vr[1] - vr[0], h), 0, 0,
                    rows=vr if part else None)
        for l in range(1, last):
            self.attention(c, l, same)
            n = ir[1] - ir[0]
            d = self.param(self.dst, 2 * n, h)
            for k in range(2):
                self.tensor(self.src, (i, h), d, k * n, l, rows=ir if part else None)
            self.tensor(self.src, (h, i), self.param(self.dst, h, n), 0, l,
                        cols=ir if part else None)
            for _ in range(2):
                self.tensor(self.src, (h,), self.param(self.dst, h), 0, l)
        self.tensor(self.src, (h,), self.param(self.dst, h), 0, last)
        self.tensor(self.src, (v, h), self.param(self.dst, vr[1] - vr[0], h), 0, last,
                    rows=vr if part else None)

    def moe(self, c, same=lambda t: t):
        h, i, v, e, ep = c["hidden"], c["inter"], c["vocab"], c["experts"], c.get("ep", 1)
        mine = range(c.get("rank", 0) * e // ep, (c.get("rank", 0) + 1) * e // ep)
        last = c["layers"] + 1
        self.tensor(self.src, (v, h), self.param(self.dst, v, h), 0, 0)
        for l in range(1, last):
            self.attention(c, l, same)
            self.tensor(self.src, (e, h), self.param(self.dst, e, h), 0, l)
            d13 = self.param(self.dst, len(mine), 2 * i, h)
            d2 = self.param(self.dst, len(mine), h, i)
            for x in range(e):
                k = x - mine[0] if x in mine else None
                here = k is not None
                self.tensor(self.src, (i, h), d13 if here else None, (k or 0) * 2 * i, l)
                self.tensor(self.src, (h, i), d2 if here else None, (k or 0) * h, l)
                self.tensor(self.src, (i, h), d13 if here else None, (k or 0) * 2 * i + i, l)
            for _ in range(2):
                self.tensor(self.src, (h,), self.param(self.dst, h), 0, l)
        self.tensor(self.src, (h,), self.param(self.dst, h), 0, last)
        self.tensor(self.src, (v, h), self.param(self.dst, v, h), 0, last)
        sizes = np.exp(self.rng.uniform(math.log(4), math.log(4096), size=c.get("extras", 0)))
        for n in np.maximum(1, sizes.astype(np.int64) // 2).tolist():
            self.tensor(self.src, (n,), self.param(self.dst, n), 0, last)

    def fp8(self, c):
        h, i, v, hd = c["hidden"], c["inter"], c["vocab"], c["head_dim"]
        q, kv, last = c["heads"] * hd, c["kv"] * hd, c["layers"] + 1
        blocks = lambda n: -(-n // 128)  # noqa: E731
        self.tensor("bf16", (v, h), self.param("bf16", v, h), 0, 0)
        for l in range(1, last):
            for parts, cols in (((q, kv, kv), h), ((h,), q), ((i, i), h), ((h,), i)):
                d = self.param("u8", sum(parts), cols)
                s = self.param("f32", sum(blocks(p) for p in parts), blocks(cols))
                at = at_s = 0
                for p in parts:
                    self.tensor("u8", (p, cols), d, at, l)
                    self.tensor("f32", (blocks(p), blocks(cols)), s, at_s, l)
                    at, at_s = at + p, at_s + blocks(p)
            for _ in range(2):
                self.tensor("bf16", (h,), self.param("bf16", h), 0, l)
        self.tensor("bf16", (h,), self.param("bf16", h), 0, last)
        self.tensor("bf16", (v, h), self.param("bf16", v, h), 0, last)


@functools.lru_cache(maxsize=2)
def _layout(key):
    return Layout(dict(key))


def layout(c):
    return _layout(tuple(sorted((k, v) for k, v in c.items() if k != "name")))


def _values(c, lay, seed):
    """The checkpoint's bytes: weights with a standard deviation of 0.02 where they are converted
    (among them ties and subnormals of the narrower type), any bytes where they are copied."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    blob = torch.empty(lay.blob_bytes, dtype=torch.uint8, device="cuda")
    if c["src"] == c["dst"]:
        blob.view(torch.int64).random_(generator=g)
        return blob
    x = blob.view(TORCH[c["src"]])
    for part in x.split(1 << 28):
        part.normal_(0.0, 0.02, generator=g)
        if c["src"] == "f32":
            bits = part.view(torch.int32)
            bits[::199] = bits[::199] & -65536 | 0x8000
            part[::211] *= 1e-37
    return blob


class State:
    pass


def prepare(case, seed):
    s = State()
    lay = layout(case)
    s.how, s.typed = case["how"], case["src"] != case["dst"]
    s.blob = _values(case, lay, seed)
    s.out = torch.zeros(lay.out_bytes, dtype=torch.uint8, device="cuda")
    s.result = s.out.view(TORCH[case["dst"]] if s.typed else torch.int64)
    dsts = np.zeros(len(lay.p_dtype), dtype=cfa.DST_DTYPE)
    dsts["dev_ptr"] = np.uint64(s.out.data_ptr()) + lay.p_offset.astype(np.uint64)
    dsts["dtype"] = [cfa.DTYPE[t] for t in lay.p_dtype]
    dsts["shape"], dsts["ndim"] = lay.p_shape
    entries = cfa.make_entries(dtype=lay.dtype, shape=lay.shape, offset=lay.offset, dst=lay.d,
                               row=lay.row, cast=np.full(len(lay.dtype), s.typed),
                               layer=lay.layer, src_row_stride=lay.stride)
    if s.how == "noalloc":
        s.entries, s.dsts, s.blob_bytes = entries, dsts, lay.blob_bytes
        s.cksum = torch.zeros(len(lay.dtype), dtype=torch.int64, device="cuda")
        s.call = ctypes.CDLL(cfa.library_path()).cfa_unpack_noalloc
        s.call.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_size_t,
                           ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p,
                           ctypes.c_void_p, ctypes.c_char_p, ctypes.c_size_t]
        return s
    staged = s.how in ("pinned", "pageable")
    s.plan = cfa.Plan(entries, dsts, lay.blob_bytes,
                      chunk_bytes=case.get("chunk_mib", 512) << 20, host_slots=0,
                      dev_slots=3 if staged else 0)
    if staged:
        host = torch.empty(lay.blob_bytes, dtype=torch.uint8, pin_memory=s.how == "pinned")
        host.copy_(s.blob)
        s.blob = host
        kind = cfa.Source.pinned if s.how == "pinned" else cfa.Source.host
        s.source = kind(host.data_ptr(), size=lay.blob_bytes)
    elif s.how == "chunks":
        step = s.plan.chunk_bytes
        s.chunks = [(k, s.blob.data_ptr() + k * step) for k in range(s.plan.info()["n_chunks"])]
    else:
        s.source = cfa.Source.device(s.blob.data_ptr(), size=lay.blob_bytes)
    return s


def run(s):
    if s.how == "noalloc":
        err = ctypes.create_string_buffer(256)
        st = s.call(s.entries.arr.ctypes.data, len(s.entries), s.dsts.ctypes.data, len(s.dsts),
                    s.blob.data_ptr(), s.blob_bytes, s.cksum.data_ptr(), None,
                    torch.cuda.current_stream().cuda_stream, err, len(err))
        if st:
            raise RuntimeError(err.value.decode())
        return {"params": s.result, "checksums": s.cksum}
    if s.how == "chunks":
        s.plan.reset_checksums()
        for k, at in s.chunks:
            s.plan.unpack_chunks_async(k, k + 1, at)
        return {"params": s.result}
    s.plan.load_async(s.source)
    if s.how == "device":
        return {"params": s.result}
    s.plan.wait_layer()
    return {"params": s.result, "checksums": s.plan.checksums().view(np.int64)}


def work(case):
    lay = layout(case)
    return {"bytes": lay.read_bytes + lay.written_bytes, "flops": 0}


def tolerance(case):
    # copies move bytes, conversions round to nearest even: there is one right answer
    return "exact"


def exact(case, seed):
    """Converted parameters: the checkpoint's numbers in 64 bits, where each belongs."""
    if case["src"] == case["dst"]:
        return None
    lay = layout(case)
    x = _values(case, lay, seed).view(TORCH[case["src"]])
    es, ds = SIZE[case["src"]], SIZE[case["dst"]]
    out = torch.zeros(lay.out_bytes // ds, dtype=torch.float64, device="cuda")
    for i, n in enumerate(lay.numel.tolist()):
        cols = int(lay.shape[0][i, lay.shape[1][i] - 1])
        a = int(lay.offset[i]) // es
        first = int(lay.p_offset[lay.d[i]]) // ds + int(lay.row[i]) * (
            cols if lay.p_shape[1][lay.d[i]] > 1 else 1)
        stride = int(lay.stride[i]) or cols
        out[first:first + n] = x.as_strided((n // cols, cols), (stride, 1), a).reshape(-1)
    v = {"params": out}
    if case["how"] in ("verify", "pinned", "pageable", "noalloc"):
        v["checksums"] = None
    return v
