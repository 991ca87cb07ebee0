"""Every dtype conversion at the edges of its groups of eight elements: run lengths around the
group and around a CTA's round of groups, sources at every element phase within 16 bytes and
destinations at every element phase within 32 bytes, on random bit patterns (NaNs with either
sign, infinities and subnormals among them), as block-level items, warp-level items and column
slices, against the oracle bit for bit and checksum for checksum."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_18957_gb300 as cfa

pytestmark = pytest.mark.gpu

ES = {"f32": 4, "f16": 2, "bf16": 2}
UINT = {4: np.uint32, 2: np.uint16}
PAIRS = [("f32", "bf16"), ("f32", "f16"), ("f16", "bf16"), ("bf16", "f32"), ("f16", "f32")]
LENGTHS = [1, 7, 8, 9, 15, 16, 17, 255, 2047, 2048, 8191, 8192 + 3, 16384 + 13]


@pytest.fixture(scope="module", autouse=True)
def cuda_device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def patterns(dtype, n, rng):
    """Random bit patterns, every eighth one a NaN, an infinity or a subnormal."""
    es = ES[dtype]
    x = rng.integers(0, 1 << (8 * es), size=n, dtype=np.uint64).astype(UINT[es])
    exp = {"f32": 0x7F800000, "f16": 0x7C00, "bf16": 0x7F80}[dtype]
    pick = rng.integers(0, 8, size=n)
    x = np.where(pick == 0, x | UINT[es](exp), x)
    x = np.where(pick == 1, x & UINT[es](~exp & ((1 << (8 * es)) - 1)), x)
    return x.astype(UINT[es])


@pytest.mark.parametrize("tiny_bytes", [0, 8192])
@pytest.mark.parametrize("src_dtype,dst_dtype", PAIRS)
def test_runs_at_every_phase(src_dtype, dst_dtype, tiny_bytes):
    rng = np.random.default_rng(5)
    ss, ds = ES[src_dtype], ES[dst_dtype]
    runs, at, to = [], 0, 0  # (source byte, destination byte, elements)
    for k, n in enumerate(LENGTHS * 3):
        for q in range(max(16 // ss, 32 // ds)):
            at = (at + 31) // 32 * 32 + ss * ((q + k) % (32 // ss))
            to = (to + 31) // 32 * 32 + ds * q + 32
            runs.append((at, to, n))
            at += n * ss
            to += n * ds
    bits = patterns(src_dtype, -(-at // ss), rng)
    blob = torch.from_numpy(bits.view(np.uint8)).to("cuda")
    out = torch.full((to + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    ents = cfa.make_entries(dtype=[src_dtype] * len(runs), shape=[(n,) for _, _, n in runs],
                            offset=[a for a, _, _ in runs], dst=list(range(len(runs))),
                            cast=[True] * len(runs))
    dsts = [(out.data_ptr() + t, dst_dtype, (n,)) for _, t, n in runs]
    with cfa.Plan(ents, dsts, bits.nbytes, dev_slots=0, host_slots=0,
                  tiny_bytes=tiny_bytes) as plan:
        plan.load_async(cfa.Source.device(blob.data_ptr()))
        plan.wait_layer()
        ck = plan.checksums()
    want = np.full(out.numel(), 0x5A, dtype=np.uint8)
    for i, (a, t, n) in enumerate(runs):
        y = oracle.convert(src_dtype, dst_dtype, bits[a // ss:a // ss + n])
        want[t:t + n * ds] = y.view(np.uint8)
        assert int(ck[i]) == int(y.astype(np.uint64).sum(dtype=np.uint64)), (i, a, t, n)
    got = out.cpu().numpy()
    bad = np.nonzero(got != want)[0]
    assert bad.size == 0, [r for r in runs if r[1] <= bad[0]][-1]


@pytest.mark.parametrize("src_dtype,dst_dtype", PAIRS)
def test_column_slices_at_every_phase(src_dtype, dst_dtype):
    rng = np.random.default_rng(6)
    ss, ds = ES[src_dtype], ES[dst_dtype]
    rows, stride = 5, 1237
    bits = patterns(src_dtype, rows * stride, rng)
    blob = torch.from_numpy(bits.view(np.uint8)).to("cuda")
    cuts = [(q, n) for q in range(16 // ss) for n in (1, 8, 15, 264, 1200)]
    outs = [torch.full((rows * n + 32,), 0, dtype=torch.int32, device="cuda") for _, n in cuts]
    ents = cfa.make_entries(dtype=[src_dtype] * len(cuts), shape=[(rows, n) for _, n in cuts],
                            offset=[q * ss for q, _ in cuts], dst=list(range(len(cuts))),
                            cast=[True] * len(cuts), src_row_stride=[stride] * len(cuts))
    lead = [ds * (i % 9) for i in range(len(cuts))]
    dsts = [(o.data_ptr() + b, dst_dtype, (rows, n)) for o, b, (_, n) in zip(outs, lead, cuts)]
    with cfa.Plan(ents, dsts, bits.nbytes, dev_slots=0, host_slots=0) as plan:
        plan.load_async(cfa.Source.device(blob.data_ptr()))
        plan.wait_layer()
        ck = plan.checksums()
    for i, (o, b, (q, n)) in enumerate(zip(outs, lead, cuts)):
        part = np.ascontiguousarray(bits.reshape(rows, stride)[:, q:q + n]).reshape(-1)
        y = oracle.convert(src_dtype, dst_dtype, part)
        got = o.cpu().numpy().view(np.uint8)[b:b + rows * n * ds]
        assert np.array_equal(got, y.view(np.uint8)), (q, n)
        assert int(ck[i]) == int(y.astype(np.uint64).sum(dtype=np.uint64)), (q, n)
