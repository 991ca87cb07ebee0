"""How launches are cut and chained: block-level items cut into parts (sizes around the parts,
sources and destinations at odd phases), one TMA launch over several element sizes, the no-alloc
entry point's upload, and chunks unpacked one after the other from a staging slot that the caller,
or the kernel before, overwrites in between, on a stream and in a CUDA graph.  Checked against
slices of the blob, and against the oracle where elements are converted."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2607_18957_gb300 as cfa
from paper_2607_18957_gb300 import _lib

pytestmark = pytest.mark.gpu

ES = {"u8": 1, "bf16": 2, "f32": 4, "i64": 8}
PART = 32768  # least bytes of a part


@pytest.fixture(scope="module", autouse=True)
def cuda_device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


class Copies:
    """Plain copies: tensors of (dtype, bytes, source phase, destination phase) in one blob."""

    def __init__(self, tensors, seed=3):
        self.runs, at, to = [], 0, 0
        for dtype, nbytes, sp, dp in tensors:
            es = ES[dtype]
            at, to = (at + 255) // 256 * 256 + sp * es, (to + 255) // 256 * 256 + 256 + dp * es
            self.runs.append((dtype, at, to, nbytes // es * es))
            at, to = at + nbytes, to + nbytes
        self.blob_bytes = (at + 255) // 256 * 256
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.blob = torch.randint(0, 256, (self.blob_bytes,), dtype=torch.uint8, device="cuda",
                                  generator=g)
        self.out = torch.full((to + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        self.want = self.out.clone()
        for _, a, t, n in self.runs:
            self.want[t:t + n] = self.blob[a:a + n]
        shapes = [(n // ES[d],) for d, _, _, n in self.runs]
        self.entries = cfa.make_entries(dtype=[r[0] for r in self.runs], shape=shapes,
                                        offset=[r[1] for r in self.runs],
                                        dst=list(range(len(self.runs))))
        self.dsts = [(self.out.data_ptr() + r[2], r[0], s) for r, s in zip(self.runs, shapes)]

    def checksums(self):
        blob = self.blob.cpu().numpy()
        u = {1: np.uint8, 2: np.uint16, 4: np.uint32, 8: np.uint64}
        return np.array([blob[a:a + n].view(u[ES[d]]).astype(np.uint64).sum(dtype=np.uint64)
                         for d, a, _, n in self.runs])


def tensors(sizes, phases):
    return [(d, n, p, q) for n in sizes for d in ES for p, q in phases]


SIZES = [8192, PART - 16, PART, PART + 16, 2 * PART + 48, 7 * PART + 8, 300 * 1024, (2 << 20) + 24]


@pytest.mark.parametrize("phases", [[(0, 0)], [(0, 0), (1, 0), (0, 1), (1, 3)]])
@pytest.mark.parametrize("slab_kib,filler_mib", [(0, 0), (0, 600), (256, 0), (4096, 0)])
def test_planned_items_are_cut_into_parts(phases, slab_kib, filler_mib):
    """Whole loads.  The plan's own slabs are 32 KiB here, or 128 KiB with 600 MiB more in the load,
    and those of aligned copies are then cut into four parts; the caller's slabs stay whole."""
    c = Copies(tensors(SIZES, phases) + [("bf16", filler_mib << 20, 0, 0)] * (filler_mib > 0))
    with cfa.Plan(c.entries, c.dsts, c.blob_bytes, dev_slots=0, host_slots=0,
                  slab_bytes=slab_kib << 10) as plan:
        plan.load_async(cfa.Source.device(c.blob.data_ptr()))
        plan.wait_layer()
        ck = plan.checksums()
    assert torch.equal(c.out, c.want)
    assert np.array_equal(ck, c.checksums())


def test_noalloc_items_are_cut_into_parts():
    c = Copies(tensors(SIZES + [(4 << 20) + 8], [(0, 0), (1, 0), (1, 3)]))
    ck = torch.full((len(c.runs),), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    dsts = cfa.make_dsts(c.dsts)
    err = ctypes.create_string_buffer(256)
    st = _lib.load().cfa_unpack_noalloc(
        c.entries.arr.ctypes.data, len(c.entries), dsts.ctypes.data, len(dsts),
        c.blob.data_ptr(), c.blob_bytes, ck.data_ptr(), status.data_ptr(),
        torch.cuda.current_stream().cuda_stream, err, len(err))
    assert st == 0, err.value
    assert int(status.item()) == 0
    assert torch.equal(c.out, c.want)
    assert np.array_equal(ck.cpu().numpy().view(np.uint64), c.checksums())


@pytest.mark.parametrize("n", [1, 112, 113, 1000, 1001, 1112, 2113, 16384])
def test_noalloc_uploads_any_number_of_items(n):
    """Item counts around what one launch of the upload carries, up to the most; twice, since a
    call reads its descriptors where the one before left its own."""
    per, es = 8192, 2
    blob = torch.randint(0, 256, (n * per,), dtype=torch.uint8, device="cuda")
    flip = torch.empty_like(blob)
    ck = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    err = ctypes.create_string_buffer(256)
    for order in (np.arange(n), np.arange(n)[::-1].copy()):
        flip.fill_(0xA5)
        ents = cfa.make_entries(dtype=["bf16"] * n, shape=[(per // es,)] * n,
                                offset=np.arange(n) * per, dst=np.zeros(n, np.int64),
                                row=order * (per // es))
        dsts = cfa.make_dsts([(flip.data_ptr(), "bf16", (n * per // es,))])
        st = _lib.load().cfa_unpack_noalloc(
            ents.arr.ctypes.data, n, dsts.ctypes.data, 1, blob.data_ptr(), blob.numel(),
            ck.data_ptr(), None, torch.cuda.current_stream().cuda_stream, err, len(err))
        assert st == 0, err.value
        to = torch.from_numpy(order).cuda()
        assert torch.equal(flip.view(n, per)[to], blob.view(n, per))
        sums = blob.view(torch.int16).view(n, -1).to(torch.int64).bitwise_and_(0xFFFF).sum(1)
        assert torch.equal(ck, sums)


def test_noalloc_checksum_array_off_the_8_byte_grid():
    """It is zeroed for entries without a checksum, and refused on the host for one with."""
    c = Copies(tensors([9000], [(0, 0)]))
    n = len(c.runs)
    room = torch.full((8 * n + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    dsts, err = cfa.make_dsts(c.dsts), ctypes.create_string_buffer(256)

    def call(flag):
        c.entries.arr["flags"] = flag
        return _lib.load().cfa_unpack_noalloc(
            c.entries.arr.ctypes.data, n, dsts.ctypes.data, n, c.blob.data_ptr(), c.blob_bytes,
            room.data_ptr() + 4, None, torch.cuda.current_stream().cuda_stream, err, len(err))

    assert call(_lib.ENTRY_CKSUM) == -11 and b"8-byte" in err.value
    assert bool((room == 0xA5).all()) and bool((c.out == 0xA5).all())
    assert call(0) == 0
    assert torch.equal(c.out, c.want)
    assert not room[4:4 + 8 * n].any() and bool((room[:4] == 0xA5).all())
    assert bool((room[4 + 8 * n:] == 0xA5).all())


def chunk_plan(c, chunk, slab_kib=0):
    return cfa.Plan(c.entries, c.dsts, c.blob_bytes, chunk_bytes=chunk, slab_bytes=slab_kib << 10,
                    dev_slots=0, host_slots=0)


def test_a_chunk_of_very_many_small_items_under_large_slabs():
    """2^20 block-level items in one chunk launch of a plan whose slabs are 64 MiB: the cut into
    parts gives way, the call is not refused."""
    n, es = 1 << 20, 2
    per = 64 // es
    entries = cfa.make_entries(dtype=["bf16"] * (n + 1),
                               shape=[(per,)] * (n + 1), offset=np.arange(n + 1) * 64,
                               dst=np.zeros(n + 1, np.int64), row=np.arange(n + 1) * per)
    blob = torch.randint(0, 256, ((n + 1) * 64,), dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(blob)
    with cfa.Plan(entries, [(out.data_ptr(), "bf16", ((n + 1) * per,))], blob.numel(),
                  chunk_bytes=n * 64, slab_bytes=64 << 20, tiny_bytes=0, dev_slots=0,
                  host_slots=0) as plan:
        assert plan.stats()["n_bulk"] == n + 1
        for k in range(2):
            plan.unpack_chunks_async(k, k + 1, blob.data_ptr() + k * n * 64)
        assert torch.equal(out, blob)


def unpack_through_one_slot(c, plan, chunk, slot):
    for k in range(plan.info()["n_chunks"]):
        part = c.blob[k * chunk:(k + 1) * chunk]
        slot[:part.numel()].copy_(part)  # a kernel or a copy that the unpack has to wait for
        slot[:part.numel()].bitwise_xor_(0xFF).bitwise_xor_(0xFF)
        plan.unpack_chunks_async(k, k + 1, slot.data_ptr())


@pytest.mark.parametrize("chunk,slab_kib", [(1 << 20, 0), (8 << 20, 0), (8 << 20, 256),
                                            (8 << 20, 4096)])
def test_chunks_through_one_slot_that_is_overwritten(chunk, slab_kib):
    """The plan's own slabs hold one part here; slabs of 256 KiB and 4 MiB are cut into several."""
    c = Copies(tensors(SIZES + [96, 5000], [(0, 0), (1, 3)]))
    slot = torch.empty(chunk, dtype=torch.uint8, device="cuda")
    with chunk_plan(c, chunk, slab_kib) as plan:
        plan.load_async(cfa.Source.device(c.blob.data_ptr()))  # checksums are those of a load
        for _ in range(3):
            c.out.fill_(0xA5)
            plan.reset_checksums()
            unpack_through_one_slot(c, plan, chunk, slot)
            torch.cuda.synchronize()
            assert torch.equal(c.out, c.want)
            assert np.array_equal(plan.checksums(), c.checksums())


PAIRS = [("f32", "bf16"), ("f32", "f16"), ("f16", "bf16"), ("bf16", "f32"), ("f16", "f32")]
UINT = {1: np.uint8, 2: np.uint16, 4: np.uint32, 8: np.uint64}


@pytest.mark.parametrize("chunk,slab_kib", [(1 << 20, 0), (8 << 20, 256), (8 << 20, 4096)])
def test_converted_chunks_and_column_slices_through_one_slot(chunk, slab_kib):
    """Every conversion, and column slices on both of their kernels and with a conversion, by
    chunks from a slot that is overwritten in between; the larger slabs are cut into parts, row
    blocks in the middle of rows."""
    rng = np.random.default_rng(11)
    es = {**ES, "f16": 2}
    jobs = [(s, d, None, n) for s, d in PAIRS for n in (5000, 33_000, 400_003)]
    jobs += [(s, d, 70, n // es[s]) for n in (1000, 4112, 7168, 32_784, 100_000)
             for s, d in (("u8", "u8"), ("f32", "f32"), ("f32", "bf16"), ("bf16", "f32"))]
    rows, at, to = [], 0, 0
    for i, (s, d, r, n) in enumerate(jobs):
        off = es[s] * (i % 3) if r is None else 64 + 16 * (i % 2)
        at, to = (at + 255) // 256 * 256, (to + 255) // 256 * 256 + 16 * (i % 5)
        pitch = 0 if r is None else -(-n * es[s] // 16) * 16 + 128  # source bytes between rows
        rows.append((at + off, to, pitch))
        at += off + (n * es[s] if r is None else pitch * r)
        to += n * (r or 1) * es[d]
    blob = rng.integers(0, 256, -(-at // 256) * 256, dtype=np.uint8)
    dev = torch.from_numpy(blob).cuda()
    out = torch.full((to + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    want, sums = np.full(to + 256, 0xA5, np.uint8), []
    for (s, d, r, n), (a, t, pitch) in zip(jobs, rows):
        cut = blob[a:a + n * es[s]] if r is None else np.stack(
            [blob[a + k * pitch:a + k * pitch + n * es[s]] for k in range(r)])
        bits = np.ascontiguousarray(cut).reshape(-1).view(UINT[es[s]])
        y = bits if s == d else oracle.convert(s, d, bits)
        want[t:t + y.nbytes] = y.view(np.uint8)
        sums.append(y.astype(np.uint64).sum(dtype=np.uint64))
    shapes = [(n,) if r is None else (r, n) for _, _, r, n in jobs]
    ents = cfa.make_entries(dtype=[j[0] for j in jobs], shape=shapes, offset=[x[0] for x in rows],
                            dst=list(range(len(jobs))), cast=[j[0] != j[1] for j in jobs],
                            src_row_stride=[x[2] // es[j[0]] for x, j in zip(rows, jobs)])
    dsts = [(out.data_ptr() + x[1], j[1], s) for x, j, s in zip(rows, jobs, shapes)]
    slot = torch.empty(chunk, dtype=torch.uint8, device="cuda")
    with cfa.Plan(ents, dsts, blob.nbytes, chunk_bytes=chunk, slab_bytes=slab_kib << 10,
                  dev_slots=0, host_slots=0) as plan:
        plan.load_async(cfa.Source.device(dev.data_ptr()))
        for _ in range(2):
            out.fill_(0xA5)
            plan.reset_checksums()
            for k in range(plan.info()["n_chunks"]):
                part = dev[k * chunk:(k + 1) * chunk]
                slot[:part.numel()].copy_(part).bitwise_xor_(0xFF).bitwise_xor_(0xFF)
                plan.unpack_chunks_async(k, k + 1, slot.data_ptr())
            torch.cuda.synchronize()
            bad = np.nonzero(out.cpu().numpy() != want)[0]
            assert bad.size == 0, [j for j, x in zip(jobs, rows) if x[1] <= bad[0]][-1]
            assert np.array_equal(plan.checksums(), np.array(sums))


@pytest.mark.parametrize("kind", ["aligned", "phases", "tiny"])
def test_chunks_that_the_kernel_before_writes(kind):
    """Chunks whose source is written by the kernel right before on the stream, an unpack of
    another plan, with new contents each time: bytes and sums."""
    chunk = 2 << 20
    c = Copies({"aligned": tensors(SIZES, [(0, 0)]), "phases": tensors(SIZES, [(1, 0), (1, 3)]),
                "tiny": tensors([96, 1000, 5000] * 60, [(0, 0), (1, 3)])}[kind])
    n = c.blob_bytes
    mid = torch.zeros(n, dtype=torch.uint8, device="cuda")
    copy = cfa.make_entries(dtype=["u8"], shape=[(n,)], offset=[0], dst=[0])
    with cfa.Plan(copy, [(mid.data_ptr(), "u8", (n,))], n, chunk_bytes=chunk, dev_slots=0,
                  host_slots=0) as first, chunk_plan(c, chunk) as second:
        second.load_async(cfa.Source.device(mid.data_ptr()))  # checksums are those of a load
        for r in range(4):
            c.blob.bitwise_xor_(0x5A + r)
            c.out.fill_(0xA5)
            second.reset_checksums()
            for k in range(second.info()["n_chunks"]):
                first.unpack_chunks_async(k, k + 1, c.blob.data_ptr() + k * chunk)
                second.unpack_chunks_async(k, k + 1, mid.data_ptr() + k * chunk)
            torch.cuda.synchronize()
            for _, a, t, m in c.runs:
                c.want[t:t + m] = c.blob[a:a + m]
            assert torch.equal(c.out, c.want)
            assert np.array_equal(second.checksums(), c.checksums())


def test_consecutive_chunks_in_a_cuda_graph():
    chunk = 4 << 20
    c = Copies(tensors(SIZES + [96, 5000], [(0, 0), (1, 3)]))
    slot = torch.empty(chunk, dtype=torch.uint8, device="cuda")
    with chunk_plan(c, chunk) as plan:
        unpack_through_one_slot(c, plan, chunk, slot)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            plan.reset_checksums()
            unpack_through_one_slot(c, plan, chunk, slot)
            for k in range(plan.info()["n_chunks"]):  # and with nothing in between
                plan.unpack_chunks_async(k, k + 1, c.blob.data_ptr() + k * chunk)
        for _ in range(2):
            c.out.fill_(0xA5)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(c.out, c.want)
        del graph


@pytest.mark.parametrize("before", ["nothing", "memset", "copy_from_host", "other_stream", "kernel"])
@pytest.mark.parametrize("kind", ["aligned", "phases"])
def test_chunks_in_a_cuda_graph_behind_other_work(kind, before):
    """A captured chunk call whose predecessor in the graph is no kernel, or not on its stream."""
    chunk = 4 << 20
    c = Copies(tensors(SIZES, [(0, 0)] if kind == "aligned" else [(1, 0), (1, 3)]))
    host = c.blob.cpu().pin_memory()
    slot = torch.zeros(chunk, dtype=torch.uint8, device="cuda")
    other, joined = torch.cuda.Stream(), torch.cuda.Event()
    with chunk_plan(c, chunk) as plan:
        chunks = [(k, host[k * chunk:(k + 1) * chunk]) for k in range(plan.info()["n_chunks"])]

        def load():
            for k, part in chunks:
                if before in ("nothing", "memset"):
                    if before == "memset":
                        plan.reset_checksums()
                    plan.unpack_chunks_async(k, k + 1, c.blob.data_ptr() + k * chunk)
                    continue
                if before == "other_stream":
                    other.wait_stream(torch.cuda.current_stream())
                    with torch.cuda.stream(other):
                        slot[:part.numel()].copy_(part, non_blocking=True)
                        joined.record()
                    torch.cuda.current_stream().wait_event(joined)
                else:
                    slot[:part.numel()].copy_(part, non_blocking=True)
                    if before == "kernel":
                        slot[:part.numel()].bitwise_xor_(0xFF).bitwise_xor_(0xFF)
                plan.unpack_chunks_async(k, k + 1, slot.data_ptr())

        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            load()
        torch.cuda.synchronize()
        assert torch.equal(c.out, c.want)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            load()
        for _ in range(2):
            c.out.fill_(0xA5)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(c.out, c.want)
        del graph


@pytest.mark.parametrize("row_bytes", [16, 1008, 1024, 1040, 4080, 4096, 4112, 7168, 8176, 8192,
                                       8208, 32768, 32784, 300_000])
def test_column_slices_by_row_length(row_bytes):
    """Rows below, at and above the shortest that go to the TMA kernel (4096), the shortest that
    are cut into segments off it (8192), the stage and a slab, at column offsets on and off the
    16-byte grid and destinations at several offsets within 128 bytes, from device memory and (in
    place) pinned memory."""
    rows, lead = 37, 6
    cases = [(d, off, to) for d in ES for off, to in ((0, 0), (16, 16), (16 + ES[d], 0),
                                                      (16, 112), (0, 48 + ES[d]), (ES[d], 120))]
    entries, outs, want = [], [], []
    g = torch.Generator(device="cuda").manual_seed(9)
    pitch = row_bytes + 64
    blob = torch.randint(0, 256, (rows * pitch + 256,), dtype=torch.uint8, device="cuda",
                         generator=g)
    grid = blob[:rows * pitch].view(rows, pitch)
    for d, off, _ in cases:
        entries.append((d, (rows, row_bytes // ES[d]), off, pitch // ES[d]))
        outs.append(torch.zeros(rows * row_bytes + 256 * lead, dtype=torch.uint8, device="cuda"))
        want.append(grid[:, off:off + row_bytes].contiguous().view(-1))
    ents = cfa.make_entries(dtype=[e[0] for e in entries], shape=[e[1] for e in entries],
                            offset=[e[2] for e in entries], dst=list(range(len(entries))),
                            src_row_stride=[e[3] for e in entries])
    dsts = [(o.data_ptr() + q[2], e[0], e[1]) for o, e, q in zip(outs, entries, cases)]
    host = blob.cpu().pin_memory()
    with cfa.Plan(ents, dsts, blob.numel(), dev_slots=2, host_slots=0,
                  chunk_bytes=1 << 20) as plan:
        for src in (cfa.Source.device(blob.data_ptr()), cfa.Source.pinned(host.data_ptr())):
            for o in outs:
                o.zero_()
            torch.cuda.synchronize()
            plan.load_async(src)
            plan.wait_layer()
            ck = plan.checksums()
            for i, (o, w) in enumerate(zip(outs, want)):
                to = cases[i][2]
                assert torch.equal(o[to:to + w.numel()], w), (i, cases[i])
                assert not o[:to].any() and not o[to + w.numel():].any()
                u = UINT[ES[cases[i][0]]]
                total = w.cpu().numpy().view(u).astype(np.uint64).sum(dtype=np.uint64)
                assert int(ck[i]) == int(total)


@pytest.mark.parametrize("dtype,n_tiny,launches", [
    ("bf16", 0, 1), ("bf16", 3, 1), ("bf16", 40, 2), ("f32", 3, 1), ("i64", 3, 1), ("u8", 3, 2)])
def test_whole_loads_of_one_plain_type(dtype, n_tiny, launches):
    """Aligned copies of one 2-, 4- or 8-byte type with few tiny pieces are one launch of the
    vector kernel; with many, or of bytes, the TMA kernel and the tiny kernel; chunk by chunk, the
    TMA kernel.  All give the blob's bytes and sums."""
    c = Copies([(dtype, n, 0, 0) for n in [8192, 65536, 4 << 20, 300 * 1024]] +
               [(dtype, 40 + 8 * k, 0, 0) for k in range(n_tiny)])
    with cfa.Plan(c.entries, c.dsts, c.blob_bytes, dev_slots=0, host_slots=0,
                  chunk_bytes=1 << 20) as plan:
        for _ in range(3):
            c.out.fill_(0xA5)
            plan.load_async(cfa.Source.device(c.blob.data_ptr()))
            plan.wait_layer()
            assert torch.equal(c.out, c.want)
            assert np.array_equal(plan.checksums(), c.checksums())
            assert plan.stats()["kernel_launches"] == launches
        c.out.fill_(0xA5)
        for k in range(plan.info()["n_chunks"]):
            plan.unpack_chunks_async(k, k + 1, c.blob.data_ptr() + k * (1 << 20))
        assert torch.equal(c.out, c.want)
