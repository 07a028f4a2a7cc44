"""The calls a user of this library makes, as measured cases.

Every case runs through the public entry points of ``paper_2604_24432_b200.binding``: the forward pass (training and
prefill), forward plus backward (one attention layer of a training step), the preparation of q, k, v upstream of it,
the decode steps over the Summary KV cache and the forward pass on host tensors.  Layouts and heads are those of the
repository's workloads (``synth.py``: layouts P, G and F, 32/8, 32/4 and 16/16 heads of 128, 4/4 heads of 64).

A case is a flat dict; text lengths of a packed batch stand in one text, "4096,517".
"""
import random

import numpy as np
import torch

from paper_2604_24432_b200 import binding as ksa
from paper_2604_24432_b200 import synth

DEV = "cuda:0"

LAYOUTS = {"P": (8, 1, 128), "G": (64, 8, 16), "F": (8, 0, 1 << 20)}        # k, m, C (synth.py)


def listed():
    return [
        # The smallest call: one short sequence, four heads of 64.  Latency of the call itself.
        dict(name="fwd_1k", op="fwd", lens="1024", layout="P", hq=4, hkv=4, d=64, kscale=1.0, peaked=0.0),
        # An ordinary training or prefill sequence of the shortest stage.
        dict(name="fwd_8k", op="fwd", lens="8192", layout="P", hq=32, hkv=8, d=128, kscale=0.5, peaked=0.0),
        # The longest context: 131,072 tokens, eight query heads per KV head, 1 % of the keys four times larger.
        dict(name="fwd_128k", op="fwd", lens="131072", layout="P", hq=32, hkv=4, d=128, kscale=1.0, peaked=0.01),
        # A packed training batch of ragged lengths (no length a whole number of chunks).
        dict(name="fwd_packed", op="fwd", lens="30125,5189,61027,4711,9043,17390", layout="P", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
        # A server prefills the prompts that are waiting, one call each, through one context: every call has other lengths.
        dict(name="prefill_prompts", op="prompts", lens="517,3001,1290,6007", layout="P", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
        # One attention layer of a training step, two sequences of 32,768 tokens: forward and backward.
        dict(name="train_32k", op="train", lens="32768,32768", layout="P", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
        # The same with long chunks (64 tokens and 8 summaries) at a shorter stage.
        dict(name="train_8k_long_chunks", op="train", lens="8192,8192", layout="G", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
        # A small ragged fine-tuning batch of the multi-head model.
        dict(name="train_ragged_mha", op="train", lens="3001,777,2214,1950", layout="P", hq=16, hkv=16, d=128, kscale=1.0, peaked=0.0),
        # The projections of a continued-pretraining step: position ids, interpolation, rotation, then the attention.
        dict(name="prepared_packed", op="prepared", lens="11003,4999,16411", layout="P", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
        # Interactive decoding: one sequence, one token.
        dict(name="decode_one", op="decode", ctx=8195, batch=1, hq=32, hkv=8, d=128, chunk=False),
        # A serving batch at a long context: the eight tokens of a chunk and its summary.
        dict(name="decode_batch", op="decode", ctx=131072, batch=32, hq=32, hkv=4, d=128, chunk=True),
        # Host tensors in, host tensors out: the upload, compute, download pipeline.
        dict(name="host_32k", op="host", lens="32768", layout="P", hq=32, hkv=8, d=128, kscale=1.0, peaked=0.0),
    ]


def draw(rng: random.Random):
    op = rng.choice(["fwd", "fwd", "prompts", "train", "train", "prepared", "decode", "decode", "host"])
    log = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    hq, hkv, d = rng.choice([(32, 8, 128), (32, 8, 128), (32, 4, 128), (16, 16, 128), (4, 4, 64), (32, 8, 64)])
    if op == "decode":
        chunk = rng.random() < 0.5
        batch = log(1, 48)
        ctx = log(64, 131072)
        if batch * ctx > 32 * 131072:
            ctx = 32 * 131072 // batch
        return dict(op=op, ctx=max(8, ctx // 8 * 8) if chunk else ctx // 8 * 8 + rng.randrange(8), batch=batch, hq=hq, hkv=hkv, d=d, chunk=chunk)
    layout = rng.choice(["P", "P", "P", "G", "G", "F"])
    total = log(300, {"fwd": 65536, "train": 32768, "prepared": 32768, "prompts": 12000, "host": 32768}[op])
    if layout == "F":
        total = min(total, 16384)                                  # plain causal layers: quadratic work
    n = rng.choice([1, 1, 2, 3, 5, 9])
    n = max(1, min(n, total // 64))
    cuts = sorted(rng.random() for _ in range(n - 1))
    parts = [max(1, int(total * (b - a))) for a, b in zip([0.0] + cuts, cuts + [1.0])]
    if rng.random() < 0.4:                                         # whole chunks: the batches that are read in place
        k = LAYOUTS[layout][0]
        parts = [max(k, p // k * k) for p in parts]
    peaked = rng.choice([0.0, 0.0, 0.01])
    return dict(op=op, lens=",".join(map(str, parts)), layout=layout, hq=hq, hkv=hkv, d=d, kscale=rng.choice([0.5, 1.0]), peaked=peaked)


def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _problem(case, lens):
    k, m, C = LAYOUTS[case["layout"]]
    return ksa.Problem(lens, k, m, C, case["hq"], case["hkv"], case["d"], float(np.float32(1.0 / np.sqrt(case["d"]))))


def _problems(case):
    lens = _lens(case)
    return [_problem(case, [n]) for n in lens] if case["op"] == "prompts" else [_problem(case, lens)]


def _normal(shape, gen):
    """bf16 standard normal values, drawn in slabs."""
    out = torch.empty(shape, dtype=torch.bfloat16, device=DEV)
    flat = out.view(-1)
    for i in range(0, flat.numel(), 1 << 28):
        part = flat[i:i + (1 << 28)]
        part.copy_(torch.randn(part.shape, generator=gen, device=DEV))
    return out


def _qkv(case, prob, gen):
    """q, k, v as synth.py draws them: normal, keys scaled, a share of the key rows four times larger."""
    L = ksa.total_aug_len(prob)
    q = _normal((L, prob.Hq, prob.D), gen)
    k = _normal((L, prob.Hkv, prob.D), gen)
    v = _normal((L, prob.Hkv, prob.D), gen)
    if case["kscale"] != 1.0:
        k *= case["kscale"]
    if case["peaked"] > 0.0:
        k[torch.rand(L, generator=gen, device=DEV) < case["peaked"]] *= 4.0
    return q, k, v


def _fwd_buffers(prob, L):
    out = torch.empty((L, prob.Hq, prob.D), dtype=torch.bfloat16, device=DEV)
    lse = torch.empty((prob.Hq, L), dtype=torch.float32, device=DEV)
    return out, lse


def _bytes_u8(n):
    return torch.empty(max(256, n), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    ctx = ksa.Context(0)
    s = dict(case=case, ctx=ctx)
    op = case["op"]
    if op == "decode":
        B, Hq, Hkv, D, k, C = case["batch"], case["hq"], case["hkv"], case["d"], 8, 128
        spec = ksa.CacheSpec(B, k, C, case["ctx"] // k + 64, Hq, Hkv, D, float(np.float32(1.0 / np.sqrt(D))))
        cache = ksa.DecodeCache(ctx, spec)
        cache.kcache.copy_(_normal(cache.kcache.shape, gen))
        cache.vcache.copy_(_normal(cache.vcache.shape, gen))
        # Where a chunk is decoded, its tokens are those that already stand in Current Chunk (token o in row k - o), so
        # that a pass leaves the cache as it found it; state: a full chunk that waits for its summary.
        steps = k if case["chunk"] else 1
        s["q"] = _normal((steps + 1, B, Hq, D), gen)
        s["kn"], s["vn"] = _normal((steps + 1, B, Hkv, D), gen), _normal((steps + 1, B, Hkv, D), gen)
        pos = torch.full((B,), case["ctx"], dtype=torch.int32, device=DEV)
        if case["chunk"]:
            for o in range(k):
                cache.kcache[:, :, k - o] = s["kn"][o + 1]
                cache.vcache[:, :, k - o] = s["vn"][o + 1]
            nsum = pos // k - 1
        else:
            nsum = pos // k
        s["state"] = torch.stack([pos, nsum], dim=1).contiguous()
        s["out"] = torch.empty((steps + 1, B, Hq, D), dtype=torch.bfloat16, device=DEV)
        s["lse"] = torch.empty((steps + 1, B, Hq), dtype=torch.float32, device=DEV)
        s["cache"] = cache
        return s
    s["calls"] = []
    for prob in _problems(case):
        L = ksa.total_aug_len(prob)
        q, k, v = _qkv(case, prob, gen)
        if op == "host":
            host = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (q, k, v)]
            out = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
            lse = torch.empty((prob.Hq, L), dtype=torch.float32, pin_memory=True)
            s["calls"].append(dict(prob=prob, q=host[0], k=host[1], v=host[2], out=out, lse=lse, ws=_bytes_u8(ksa.host_staging_bytes(prob))))
            continue
        out, lse = _fwd_buffers(prob, L)
        c = dict(prob=prob, q=q, k=k, v=v, out=out, lse=lse)
        if op == "prepared":
            S = ksa.total_summary_rows(prob)
            for n, H in (("qs", prob.Hq), ("ks", prob.Hkv), ("vs", prob.Hkv)):
                c[n] = _normal((S, H, prob.D), gen)
            c["ws"] = _bytes_u8(ksa.prepared_workspace_bytes(prob))
        else:
            c["ws"] = _bytes_u8(ksa.workspace_bytes(prob))
        if op == "train":
            c["dout"] = _normal(q.shape, gen)
            c["dq"], c["dk"], c["dv"] = torch.empty_like(q), torch.empty_like(k), torch.empty_like(v)
            c["wsb"] = _bytes_u8(ksa.bwd_workspace_bytes(prob))
        s["calls"].append(c)
    return s


def run(s):
    ctx, op = s["ctx"], s["case"]["op"]
    if op == "decode":
        cache = s["cache"]
        cache.state.copy_(s["state"])                              # back to the prompt: every pass decodes the same tokens
        if s["case"]["chunk"]:
            cache.decode_summary(s["q"][0], s["kn"][0], s["vn"][0], s["out"][0], s["lse"][0])
            for o in range(1, s["q"].shape[0]):
                cache.decode_text(s["q"][o], s["kn"][o], s["vn"][o], s["out"][o], s["lse"][o])
            return s["out"], s["lse"], cache.state, cache.kcache, cache.vcache
        cache.decode_text(s["q"][0], s["kn"][0], s["vn"][0], s["out"][0], s["lse"][0])
        return s["out"][0], s["lse"][0], cache.state, cache.kcache, cache.vcache
    outs = []
    for c in s["calls"]:
        if op == "host":
            ctx.attn_fwd_host(c["prob"], c["q"], c["k"], c["v"], c["out"], c["lse"], c["ws"])
        elif op == "prepared":
            ctx.attn_fwd_prepared(c["prob"], c["q"], c["k"], c["v"], c["qs"], c["ks"], c["vs"], 0.5, 1e6, c["out"], c["lse"], c["ws"])
        else:
            ctx.attn_fwd(c["prob"], c["q"], c["k"], c["v"], c["out"], c["lse"], c["ws"])
        outs += [c["out"], c["lse"]]
        if op == "train":
            ctx.attn_bwd(c["prob"], c["q"], c["k"], c["v"], c["out"], c["lse"], c["dout"], c["dq"], c["dk"], c["dv"], c["wsb"])
            outs += [c["dq"], c["dk"], c["dv"]]
    return outs


def work(case):
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    if case["op"] == "decode":
        B, k, C = case["batch"], 8, 128
        spec = ksa.CacheSpec(B, k, C, case["ctx"] // k + 64, hq, hkv, d, 1.0)
        rows = 0
        steps = k if case["chunk"] else 1
        for i in range(steps):
            lo, hi = ksa.cache_slice(spec, case["ctx"] + i, False)
            rows += hi - lo
        if case["chunk"]:
            rows += k + 1
            steps += 1
        # the slices of K and V, the new rows in and into the cache, q in, out and lse out
        return {"bytes": B * (rows * hkv * d * 4 + steps * (hkv * d * 8 + hq * d * 4 + hq * 4)), "flops": 4 * d * B * hq * rows}
    nbytes = flops = 0
    for prob in _problems(case):
        L = ksa.total_aug_len(prob)
        q, kv, lse = L * hq * d * 2, L * hkv * d * 2, L * hq * 4
        f = 4 * d * hq * ksa.visible_pairs(prob)
        nbytes += 2 * q + 2 * kv + lse                             # q, k, v in; out, lse out
        if case["op"] == "train":
            nbytes += 2 * q + 2 * kv                               # dout in; dq, dk, dv out
            f = f * 7 // 2                                         # two products forward, five backward
        if case["op"] == "prepared":
            nbytes += ksa.total_summary_rows(prob) * (hq + 2 * hkv) * d * 2
        flops += f
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # bf16 operands, probabilities and results, fp32 sums.  Measured: decode against 64-bit sums 2.2e-3 (2-norm); forward on
    # the tensor cores against the CUDA-core kernel up to 1.5e-3, largest difference 0.025; gradients against the mma.sync
    # kernels up to 9e-5, largest 0.016.  Four times the largest of each.
    return {"rel": 8e-3, "max": 0.1}
