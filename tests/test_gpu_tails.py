"""Ragged batches read in place: full tiles straight from the caller's tensors, each sequence's last tile from the packed
streams.  Against the packed path (every tile from the streams), bit for bit: the same tiles reach the same kernels."""
import random

import pytest
import torch

from paper_2604_24432_b200 import binding as ksa
from paper_2604_24432_b200 import build as ksa_build

pytestmark = pytest.mark.gpu

# every tile from the streams, as the CTA-pair kernel wants them, in the same kernels as without flags
PACKED = ksa.KSA_FLAG_CTA_PAIR_KERNEL | ksa.KSA_FLAG_SINGLE_CTA_KERNEL


@pytest.fixture(scope="module")
def ctx():
    ksa_build.build()
    c = ksa.Context(0)
    yield c
    c.close()


def _rows(total, H, D, gen, layout="dense", gap=8):
    """bf16 rows [total, H, D]; "gaps": heads with `gap` elements between them, rows with more; "heads first": [H, total, D] in memory."""
    if layout == "heads first":
        return torch.randn((H, total, D), generator=gen, device="cuda").bfloat16().transpose(0, 1)
    if layout == "gaps":
        return torch.randn((total, H + 1, D + gap), generator=gen, device="cuda").bfloat16()[:, 1:, :D]
    return torch.randn((total, H, D), generator=gen, device="cuda").bfloat16()


def _like(t):
    return torch.empty_strided(t.shape, t.stride(), dtype=t.dtype, device=t.device).fill_(7.0)


def _assert_same_bits(a, b, what=None):
    as_int = {torch.bfloat16: torch.int16, torch.float32: torch.int32}[a.dtype]
    assert torch.equal(a.view(as_int), b.view(as_int)), what


def _assert_one_rounding_apart(a, b, what=None):
    """dk, dv: sums of fp32 atomics in either order, then bf16."""
    a, b = a.float(), b.float()
    assert ((a - b).abs() <= 2 ** -7 * b.abs() + 1e-6 * b.abs().max()).all(), what


@pytest.mark.parametrize("lens,k,m,C,Hq,Hkv,D", [
    ([129, 127, 1, 257], 8, 1, 4, 4, 2, 128),            # a last tile of one row, of 127, no full tile
    ([1027, 5, 130, 643], 8, 1, 16, 8, 2, 64),           # sequences that start at every row of a chunk
    ([1153, 2175], 8, 1, 16, 4, 4, 128),                 # 144 and 271 summary rows: full tiles and last ones
    ([4097, 70], 64, 8, 4, 8, 2, 128),                   # 64 chunks of eight summaries: four full tiles, none left over
    ([300, 1011], 8, 0, 1 << 20, 4, 2, 128),             # no summaries
    ([513, 255, 771], 1, 1, 100, 4, 2, 64),              # chunks of one token: never ragged, read in place either way
    ([513, 255, 771], 2, 2, 50, 4, 2, 64),               # chunks of two
    ([400, 999], 128, 2, 1, 6, 2, 128),                  # a chunk fills a tile; head pairs across KV heads
])
@pytest.mark.parametrize("layout", ["dense", "gaps", "heads first"])
def test_tails_equal_the_packed_path(ctx, lens, k, m, C, Hq, Hkv, D, layout):
    gen = torch.Generator("cuda").manual_seed(11)
    packed = ksa.Problem(lens, k, m, C, Hq, Hkv, D, D ** -0.5, PACKED)
    prob = ksa.Problem(lens, k, m, C, Hq, Hkv, D, D ** -0.5)
    total = ksa.total_aug_len(prob)
    # (strides of their own for q, k, v and for out and dout)
    q, kk, v, dout = (_rows(total, H, D, gen, layout, gap) for H, gap in ((Hq, 8), (Hkv, 16), (Hkv, 24), (Hq, 40)))
    got = []
    for p in (packed, prob):
        out, dq, dk, dv = (_like(t) for t in (dout, q, kk, v))
        lse = torch.empty((Hq, total), dtype=torch.float32, device="cuda")
        ws = torch.full((max(256, ksa.workspace_bytes(p)),), 0xFF, dtype=torch.uint8, device="cuda")   # NaN patterns
        wsb = torch.full((ksa.bwd_workspace_bytes(p),), 0xFF, dtype=torch.uint8, device="cuda")
        ctx.clear_device_status()
        ctx.attn_fwd(p, q, kk, v, out, lse, ws)
        ctx.attn_bwd(p, q, kk, v, out, lse, dout, dq, dk, dv, wsb)
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        got.append((out, lse, dq, dk, dv))
    for a, b in zip(got[0][:3], got[1][:3]):
        _assert_same_bits(a, b)
    for a, b in zip(got[0][3:], got[1][3:]):
        _assert_one_rounding_apart(a, b)


def test_the_forward_pass_ignores_the_backward_flag(ctx):
    """What stands in the workspace behind a ragged call: with full tiles read in place the streams' last tiles, whether the
    backward pass is to run on mma.sync kernels, which want whole streams, or not."""
    left = []
    for flags in (0, ksa.KSA_FLAG_BWD_MMA_SYNC_KERNELS, PACKED):
        prob = ksa.Problem([1027, 333], 8, 1, 4, 4, 2, 128, 128 ** -0.5, flags)
        total = ksa.total_aug_len(prob)
        gen = torch.Generator("cuda").manual_seed(14)
        q, kk, v = (_rows(total, H, 128, gen) for H in (4, 2, 2))
        lse = torch.empty((4, total), dtype=torch.float32, device="cuda")
        left.append(torch.full((ksa.workspace_bytes(prob),), 0xFF, dtype=torch.uint8, device="cuda"))
        ctx.attn_fwd(prob, q, kk, v, torch.empty_like(q), lse, left[-1])
    assert torch.equal(left[0], left[1]) and not torch.equal(left[0], left[2])


def test_a_sequence_does_not_see_its_neighbour(ctx):
    """NaN and infinities in one sequence of a ragged batch leave the others' outputs and gradients finite."""
    lens, k, m, C, Hq, Hkv, D = [333, 258, 131], 8, 1, 4, 4, 2, 128
    gen = torch.Generator("cuda").manual_seed(12)
    prob = ksa.Problem(lens, k, m, C, Hq, Hkv, D, D ** -0.5)
    total = ksa.total_aug_len(prob)
    q, kk, v, dout = (_rows(total, H, D, gen) for H in (Hq, Hkv, Hkv, Hq))
    lo, hi = ksa.aug_len(333, k, m), ksa.aug_len(333, k, m) + ksa.aug_len(258, k, m)
    for t in (kk, v, dout):
        t[lo:hi] = float("nan")
        t[lo:lo + 3] = float("inf")
    out, dq = torch.empty_like(q), torch.empty_like(q)
    dk, dv = torch.empty_like(kk), torch.empty_like(v)
    lse = torch.empty((Hq, total), dtype=torch.float32, device="cuda")
    ws = torch.full((ksa.workspace_bytes(prob),), 0xFF, dtype=torch.uint8, device="cuda")
    wsb = torch.full((ksa.bwd_workspace_bytes(prob),), 0xFF, dtype=torch.uint8, device="cuda")
    ctx.clear_device_status()
    ctx.attn_fwd(prob, q, kk, v, out, lse, ws)
    ctx.attn_bwd(prob, q, kk, v, out, lse, dout, dq, dk, dv, wsb)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    for t in (out, dq, dk, dv):
        assert torch.isfinite(t[:lo].float()).all() and torch.isfinite(t[hi:].float()).all()


@pytest.mark.parametrize("wide", ["q", "k", "v", "o"])
def test_a_head_stride_that_no_tensor_map_holds(ctx, wide):
    """The head stride of a tensor with one head is never used, and may be any number: a ragged batch gives the same with 2^40
    bytes, more than a tensor map's stride may be."""
    lens, k, m, C, D = [333, 130, 8], 8, 1, 4, 128
    Hq = 1 if wide in "qo" else 4
    total = sum(ksa.aug_len(n, k, m) for n in lens)
    prob = ksa.Problem(lens, k, m, C, Hq, 1, D, D ** -0.5)
    gen = torch.Generator("cuda").manual_seed(13)
    q, kk, v, dout = (_rows(total, H, D, gen) for H in (Hq, 1, 1, Hq))

    def view(t, name):
        return t.as_strided(t.shape, (t.stride(0), 1 << 39, 1)) if name == wide else t

    got = []
    for shape in (lambda t, name: t, view):
        out, dq, dk, dv = (shape(torch.full_like(t, 7.0), n) for t, n in ((q, "o"), (q, "q"), (kk, "k"), (v, "v")))
        lse = torch.empty((Hq, total), dtype=torch.float32, device="cuda")
        ws = torch.full((ksa.workspace_bytes(prob),), 0xFF, dtype=torch.uint8, device="cuda")
        wsb = torch.full((ksa.bwd_workspace_bytes(prob),), 0xFF, dtype=torch.uint8, device="cuda")
        args = shape(q, "q"), shape(kk, "k"), shape(v, "v"), out, lse
        ctx.clear_device_status()
        ctx.attn_fwd(prob, *args, ws)
        ctx.attn_bwd(prob, *args, shape(dout, "o"), dq, dk, dv, wsb)
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        got.append((out, lse, dq, dk, dv))
    for a, b in zip(got[0][:3], got[1][:3]):
        _assert_same_bits(a, b)
    for a, b in zip(got[0][3:], got[1][3:]):
        _assert_one_rounding_apart(a, b)


@pytest.mark.parametrize("k,m", [(8, 1), (24, 8)])
def test_schedules_that_share_memory(ctx, k, m):
    """One context, another split of the same rows into sequences in every call: the schedules' memory goes round several times,
    and the kernels that start beside the one in front of them read the table of this call.  Against contexts of one call each."""
    Hq, Hkv, D, n = 8, 4, 64, 1536
    rng = random.Random(15)
    gen = torch.Generator("cuda").manual_seed(15)
    q, kk, v, dout = (_rows(n + n // k * m, H, D, gen) for H in (Hq, Hkv, Hkv, Hq))
    once = ksa.Context(0)
    own = ksa.Context(0)
    for call in range(150):
        cuts = sorted(rng.sample(range(1, n), rng.randrange(1, 8)))
        lens = [b - a for a, b in zip([0] + cuts, cuts + [n])]
        prob = ksa.Problem(lens, k, m, 4, Hq, Hkv, D, D ** -0.5)
        total = ksa.total_aug_len(prob)
        args = q[:total], kk[:total], v[:total]
        ws = torch.empty(max(256, ksa.workspace_bytes(prob)), dtype=torch.uint8, device="cuda")
        wsb = torch.empty(ksa.bwd_workspace_bytes(prob), dtype=torch.uint8, device="cuda")
        got = []
        for c in (own, once):
            out, dq, dk, dv = (torch.full_like(t, 7.0) for t in (args[0], *args))
            lse = torch.empty((Hq, total), dtype=torch.float32, device="cuda")
            c.attn_fwd(prob, *args, out, lse, ws)
            c.attn_bwd(prob, *args, out, lse, dout[:total], dq, dk, dv, wsb)
            got.append((out, lse, dq, dk, dv))
        torch.cuda.synchronize()
        once.close()
        once = ksa.Context(0)
        for a, b in zip(got[0][:3], got[1][:3]):
            _assert_same_bits(a, b, (call, lens))
        for a, b in zip(got[0][3:], got[1][3:]):
            _assert_one_rounding_apart(a, b, (call, lens))
    once.close()
    own.close()
