"""Measured cases of the mixed prefill/decode attention step.

A case is one call, or one short sequence of calls, that a serving program
makes per layer and step through the package's public entry points:

* ``step``: ``mixed_step`` of a plan (KV append of the step's new rows, then
  attention of every query over the paged cache). The plan is kept, as all
  layers of a model share one plan per step; with ``replan`` the pass also
  plans the step anew from the host metadata, as the first layer's call does.
* ``noalloc``: ``kv_append`` and ``decode_attn_noalloc``, for callers that may
  not allocate device memory.
* ``expand``: ``kv_append`` of latent rows, ``mla_expand`` into per-head keys
  and values, and multi-head attention of the chunk over them.

Head shapes, block sizes and lengths are those of the repository's workloads
and tests. Queries are N(0, 4) and cache rows N(0, 1), so that scaled scores
have a spread of about 2 and rows differ in where their weight lies. Sequence
lengths depend on the case alone (``lens`` seeds them); values and the places
of the blocks in the pool depend on the seed.
"""
import math

import numpy as np
import torch

import paper_2606_04415_gb300 as fnpu

# (query heads, kv heads, key width, value width, latent cache)
HEADS = {
    "4x2": (4, 2, 64, 64, False),          # the small exhaustive-check shape
    "28x4": (28, 4, 128, 128, False),      # Qwen2.5-7B
    "32x8": (32, 8, 128, 128, False),      # R1-Distill-Llama-8B
    "latent": (128, 1, 576, 512, True),    # DeepSeek-R1, absorbed
}
FP8_BLOCK = 16 * 4 * 128 + 16 * 4 * 4       # bytes of one block of the FP8 format
NOALLOC_SPLIT = 512                         # the entry point's default split


def _case(path, heads, bs, chunks, chunk, prefix, decodes, ctx_lo, ctx_hi, tokens=1, fp8=False, replan=False, lens=0):
    """``chunks`` prefill chunks of up to ``chunk`` tokens on prefixes of up to
    ``prefix`` and ``decodes`` decodes of ``tokens`` tokens each with contexts
    of ``ctx_lo`` .. ``ctx_hi``."""
    return dict(path=path, heads=heads, bs=bs, chunks=chunks, chunk=chunk, prefix=prefix, decodes=decodes, ctx_lo=ctx_lo,
                ctx_hi=ctx_hi, tokens=tokens, fp8=fp8, replan=replan, lens=lens)


def listed():
    return [
        # the smallest step: two short prompts and six decodes of a small
        # model, planned anew; launches and host calls count
        dict(_case("step", "4x2", 16, 2, 128, 0, 6, 64, 512, replan=True), name="step_small"),
        # a lightly loaded server: four decodes, a latency-bound call
        dict(_case("step", "28x4", 16, 0, 0, 0, 4, 300, 2500), name="decode_4"),
        # an ordinary decode batch, bound by cache reads
        dict(_case("step", "28x4", 16, 0, 0, 0, 64, 512, 4096), name="decode_64"),
        # the same batch over the FP8 cache
        dict(_case("step", "28x4", 16, 0, 0, 0, 64, 512, 4096, fp8=True), name="decode_64_fp8"),
        # prompt processing alone: four chunks on prefixes of different length
        dict(_case("step", "28x4", 16, 4, 512, 1536, 0, 0, 0), name="prefill_4x512"),
        # prefill and decode co-located: one 2048-token chunk on a long prefix
        # beside 128 decodes
        dict(_case("step", "28x4", 16, 1, 2048, 7000, 128, 128, 8192), name="mixed_2048_128"),
        # the same step over the FP8 cache
        dict(_case("step", "28x4", 16, 1, 2048, 7000, 128, 128, 8192, fp8=True), name="mixed_2048_128_fp8"),
        # co-location with eight kv heads and 32-token blocks
        dict(_case("step", "32x8", 32, 1, 1024, 3000, 64, 100, 5000), name="mixed_32x8"),
        # speculative verification: 32 sequences of four tokens each
        dict(_case("step", "28x4", 16, 0, 0, 0, 32, 700, 5000, tokens=4), name="verify_32x4"),
        # latent attention, the largest step: one 1024-token prompt and 256 decodes
        dict(_case("step", "latent", 64, 1, 1024, 0, 256, 1024, 16384), name="latent_mixed"),
        # the same prompt without absorption: expansion and 192/128-wide attention
        dict(_case("expand", "latent", 64, 1, 1024, 0, 0, 0, 0), name="latent_expand"),
        # decode from a process that may not allocate
        dict(_case("noalloc", "32x8", 16, 0, 0, 0, 16, 200, 6000), name="noalloc_16"),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["decode", "decode", "prefill", "mixed", "mixed", "verify", "latent", "latent", "expand", "noalloc"])
    heads = rng.choice(["4x2", "28x4", "28x4", "32x8"])
    fp8 = heads == "28x4" and rng.random() < 0.4
    bs = 16 if fp8 else rng.choice([16, 32, 64])
    replan = rng.random() < 0.2
    lens = rng.randrange(1 << 20)
    lo = spread(20, 1000)
    if kind == "decode":
        return _case("step", heads, bs, 0, 0, 0, spread(1, 160), lo, lo + spread(50, 8000), fp8=fp8, replan=replan, lens=lens)
    if kind == "prefill":
        n = rng.randint(1, 5)
        return _case("step", heads, bs, n, spread(20, 2400 // n), spread(1, 8000), 0, 0, 0, fp8=fp8, replan=replan, lens=lens)
    if kind == "mixed":
        n = rng.randint(1, 3)
        return _case("step", heads, bs, n, spread(20, 2400 // n), spread(1, 8000), spread(1, 160), lo, lo + spread(50, 7000),
                     fp8=fp8, replan=replan, lens=lens)
    if kind == "verify":
        return _case("step", heads, bs, 0, 0, 0, spread(1, 64), lo, lo + spread(50, 6000), tokens=rng.randint(2, 8), fp8=fp8,
                     replan=replan, lens=lens)
    if kind == "latent":
        n = rng.randint(0, 1)
        return _case("step", "latent", rng.choice([16, 32, 64]), n, spread(16, 900), spread(1, 500),
                     spread(1, 128), lo, lo + spread(100, 14000), replan=replan, lens=lens)
    if kind == "expand":
        return _case("expand", "latent", rng.choice([16, 64]), 1, spread(50, 1000), spread(1, 1000), 0, 0, 0, lens=lens)
    n, hi = spread(1, 64), spread(100, 6000)
    return _case("noalloc", heads, bs, 0, 0, 0, n, 20, min(20 + hi, 900 // n * NOALLOC_SPLIT), lens=lens)


# ------------------------------------------------------------------ inputs

def _lengths(case):
    """(query_len, context_len, phase) of the case's sequences."""
    rng = np.random.default_rng([17, case["lens"]])
    q, ctx, ph = [], [], []
    for i in range(case["chunks"]):
        # prefixes spread evenly up to the longest, chunks full
        n = case["chunks"]
        pre = case["prefix"] * i // (n - 1) if n > 1 else case["prefix"]
        q.append(max(1, case["chunk"]))
        ctx.append(q[-1] + pre)
        ph.append(0)
    lo, hi = case["ctx_lo"], case["ctx_hi"]
    for c in (np.exp(rng.uniform(math.log(lo), math.log(hi), case["decodes"])) if case["chunks"] and case["path"] == "step"
              and case["heads"] != "latent" else rng.uniform(lo, hi, case["decodes"])) if case["decodes"] else []:
        q.append(case["tokens"])
        ctx.append(max(case["tokens"], int(c)))
        ph.append(1)
    return np.array(q, np.int32), np.array(ctx, np.int32), np.array(ph, np.uint8)


def _inputs(case, seed):
    """Everything a user's program has before the call, as CUDA tensors and
    host metadata: cache pools in bf16, new rows, queries, the block table."""
    hq, hkv, dq, dv, latent = HEADS[case["heads"]]
    bs = case["bs"]
    q_len, ctx, phase = _lengths(case)
    T = int(q_len.sum())
    nblk = (ctx.astype(np.int64) + bs - 1) // bs
    num_blocks = int(math.ceil(1.25 * int(nblk.sum())))
    rng = np.random.default_rng([29, seed])
    perm = rng.permutation(num_blocks).astype(np.int32)
    bt = rng.integers(0, num_blocks, size=(len(ctx), int(nblk.max()) + 1)).astype(np.int32)
    off, slots = 0, []
    for s in range(len(ctx)):
        bt[s, :nblk[s]] = perm[off:off + nblk[s]]
        off += int(nblk[s])
        pos = np.arange(int(ctx[s] - q_len[s]), int(ctx[s]), dtype=np.int64)
        slots.append(bt[s, pos // bs].astype(np.int64) * bs + pos % bs)
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(*shape, std=1.0):
        return (torch.randn(shape, device="cuda", dtype=torch.float32, generator=g) * std).to(torch.bfloat16)

    x = {"q_len": q_len, "ctx": ctx, "phase": phase, "bt": bt, "num_blocks": num_blocks, "T": T,
         "slots": torch.from_numpy(np.concatenate(slots)).cuda()}
    if latent:
        x["k"] = normal(num_blocks, bs, dq)
        x["k_new"], x["v"], x["v_new"] = normal(T, dq), None, None
    else:
        x["k"], x["v"] = normal(num_blocks, bs, hkv, dq), normal(num_blocks, bs, hkv, dv)
        x["k_new"], x["v_new"] = normal(T, hkv, dq), normal(T, hkv, dv)
    if case["path"] == "expand":
        x["q"] = normal(T, hq, 192, std=2.0)
        x["w_uk"], x["w_uv"] = normal(hq, 512, 128, std=512 ** -0.5), normal(hq, 512, 128, std=512 ** -0.5)
        # rows of the expanded cache: every sequence's positions in order, from
        # a 16-row block boundary, padding rows with slot -1
        rows, ebt, first = [], np.zeros((len(ctx), int((ctx.max() + 15) // 16)), np.int32), 0
        for s in range(len(ctx)):
            pos = np.arange(int(ctx[s]), dtype=np.int64)
            n16 = (int(ctx[s]) + 15) // 16
            rows += [bt[s, pos // bs].astype(np.int64) * bs + pos % bs, np.full(16 * n16 - len(pos), -1, np.int64)]
            ebt[s, :n16] = np.arange(first, first + n16)
            first += n16
        x["rows"], x["ebt"], x["eblocks"] = torch.from_numpy(np.concatenate(rows)).cuda(), ebt, first
    else:
        x["q"] = normal(T, hq, dq, std=2.0)
    return x


def _prefix_slots(x, bs):
    out = []
    for s in range(len(x["ctx"])):
        pos = np.arange(int(x["ctx"][s] - x["q_len"][s]), dtype=np.int64)
        out.append(x["bt"][s, pos // bs].astype(np.int64) * bs + pos % bs)
    return torch.from_numpy(np.concatenate(out)).cuda()


def prepare(case, seed):
    hq, hkv, dq, dv, latent = HEADS[case["heads"]]
    x = _inputs(case, seed)
    x["case"] = case
    x["desc"] = fnpu.make_desc(hq, hkv, dq, dv, case["bs"], x["num_blocks"], latent, 0.0, case["fp8"])
    if case["fp8"]:
        # the cache as a serving process has it: filled by the library's append
        sl = _prefix_slots(x, case["bs"])
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        pools = [torch.randint(0, 256, (x["num_blocks"] * FP8_BLOCK,), dtype=torch.uint8, device="cuda", generator=g)
                 for _ in range(2)]
        if sl.numel():
            fnpu.kv_append(x["desc"], x["k"].view(-1, hkv, dq)[sl].contiguous(), x["v"].view(-1, hkv, dv)[sl].contiguous(), sl,
                           pools[0], pools[1])
        x["k"], x["v"] = pools
    T = x["T"]
    if case["path"] == "expand":
        n = int(x["rows"].numel())
        x["edesc"] = fnpu.make_desc(hq, hq, 192, 128, 16, x["eblocks"])
        x["ws"] = torch.empty((n, 512), dtype=torch.bfloat16, device="cuda")
        x["ek"] = torch.empty((x["eblocks"] * 16, hq, 192), dtype=torch.bfloat16, device="cuda")
        x["ev"] = torch.empty((x["eblocks"] * 16, hq, 128), dtype=torch.bfloat16, device="cuda")
        x["out"] = torch.empty((T, hq, 128), dtype=torch.bfloat16, device="cuda")
        x["plan"] = fnpu.mixed_attn_plan(x["edesc"], x["q_len"], x["ctx"], x["phase"], x["ebt"])
    else:
        x["out"] = torch.empty((T, hq, dv), dtype=torch.bfloat16, device="cuda")
        if case["path"] == "noalloc":
            x["ctx_dev"], x["bt_dev"] = torch.from_numpy(x["ctx"]).cuda(), torch.from_numpy(x["bt"]).cuda()
            x["max_ctx"] = int(x["ctx"].max())
        else:
            x["plan"] = fnpu.mixed_attn_plan(x["desc"], x["q_len"], x["ctx"], x["phase"], x["bt"])
    x["lse"] = torch.empty((T, hq), dtype=torch.float32, device="cuda")
    # what a pass returns: results and the updated cache (its bits)
    pools = [None if t is None else t if t.dtype == torch.uint8 else t.view(torch.int16) for t in (x["k"], x["v"])]
    x["result"] = {"out": x["out"], "lse": x["lse"], "k_cache": pools[0], "v_cache": pools[1]}
    if case["path"] == "expand":
        x["result"].update(ek=x["ek"], ev=x["ev"])
    return x


def run(x):
    case = x["case"]
    if case["path"] == "step":
        if case["replan"]:
            fnpu.mixed_attn_replan(x["plan"], x["q_len"], x["ctx"], x["phase"], x["bt"])
        fnpu.mixed_step(x["plan"], x["k_new"], x["v_new"], x["slots"], x["q"], x["k"], x["v"], x["out"], x["lse"])
    else:
        fnpu.kv_append(x["desc"], x["k_new"], x["v_new"], x["slots"], x["k"], x["v"])
        if case["path"] == "noalloc":
            fnpu.decode_attn_noalloc(x["desc"], x["ctx_dev"], x["bt_dev"], x["max_ctx"], x["q"], x["k"], x["v"], x["out"], x["lse"])
        else:
            fnpu.mla_expand(x["desc"], x["k"], x["rows"], x["w_uk"], x["w_uv"], x["ws"], x["ek"], x["ev"])
            fnpu.mixed_attn_run(x["plan"], x["q"], x["ek"], x["ev"], x["out"], x["lse"])
    return x["result"]


# -------------------------------------------------------------------- work

def work(case):
    hq, hkv, dq, dv, latent = HEADS[case["heads"]]
    q, ctx, _ = (a.astype(np.int64) for a in _lengths(case))
    T, pre = int(q.sum()), ctx - q
    pairs = int((q * pre + q * (q + 1) // 2).sum())
    row = 2 * (dq if latent else hkv * (dq + dv))                      # a bf16 cache row of all heads
    stored = hkv * (dq + dv + 8) if case["fp8"] else row
    # prefix rows read, new rows read and stored, slots, block table
    b = int(pre.sum()) * stored + T * (row + stored + 8) + 4 * int(((ctx + case["bs"] - 1) // case["bs"]).sum())
    if case["path"] == "expand":
        # weights and queries read, expanded keys and values and the output written
        n = int(ctx.sum())
        b += 2 * 2 * hq * 512 * 128 + n * hq * (192 + 128) * 2 + T * hq * (192 * 2 + 128 * 2 + 4)
        return {"bytes": b, "flops": 2 * n * hq * 512 * 256 + 2 * hq * pairs * (192 + 128)}
    return {"bytes": b + T * hq * (2 * dq + 2 * dv + 4), "flops": 2 * hq * pairs * (dq + dv)}


def tolerance(case):
    # Outputs are bf16 and the probabilities of the second product bf16 or f16:
    # against 64 bits the outputs are 1.7e-3 to 2.3e-3 off in the 2-norm (the
    # rounding of the output alone is 1.7e-3), and 3.6e-3 where the expanded
    # keys and values are rounded to bf16 on the way. Four times that, and ten
    # standard deviations of it for a single value. Cache contents are whole.
    return {"rel": 1.4e-2, "max": 1e-1} if case["path"] == "expand" else {"rel": 9e-3, "max": 6e-2}


# ------------------------------------------------- the same in 64 bits

def _attend64(q, k, v, scale):
    """Causal attention of the last len(q) positions: q [n, hq, dq], k [c, hkv,
    dq], v [c, hkv, dv], all float64; returns [n, hq, dv], [n, hq]."""
    n, hq, dq = q.shape
    c, hkv, dv = v.shape
    G = hq // hkv
    out = torch.empty((n, hq, dv), dtype=torch.float64, device=q.device)
    lse = torch.empty((n, hq), dtype=torch.float64, device=q.device)
    hidden = torch.arange(c, device=q.device)[None, :] > torch.arange(c - n, c, device=q.device)[:, None]
    step = max(1, (1 << 28) // max(1, c * G))  # rows of one kv head at a time: 2 GB of scores
    for h in range(hkv):
        for i in range(0, n, step):
            qi = q[i:i + step, h * G:(h + 1) * G]
            s = (qi.reshape(-1, dq) @ k[:, h].T).view(qi.shape[0], G, c) * scale
            s.masked_fill_(hidden[i:i + step, None, :], -math.inf)
            m = s.amax(-1, keepdim=True)
            p = torch.exp(s - m)
            z = p.sum(-1, keepdim=True)
            out[i:i + step, h * G:(h + 1) * G] = ((p / z).view(-1, c) @ v[:, h]).view(qi.shape[0], G, dv)
            lse[i:i + step, h * G:(h + 1) * G] = (m + torch.log(z))[..., 0]
    return out, lse


def _fp8(rows):
    """Stored value of bf16 rows in the FP8 cache: e4m3 codes of row / scale,
    scale = amax / 448 in fp32."""
    f = rows.float()
    a = f.abs().amax(-1, keepdim=True)
    # (a tensor divisor: division by a Python number multiplies by its reciprocal)
    scale = torch.where(a > 0, a / torch.full_like(a, 448.0), torch.ones_like(a))
    return (f / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).double() * scale.double()


def exact(case, seed):
    hq, hkv, dq, dv, latent = HEADS[case["heads"]]
    bs = case["bs"]
    x = _inputs(case, seed)
    k = x["k"].view(-1, hkv, dq)
    k[x["slots"]] = x["k_new"].view(-1, hkv, dq)
    if not latent:
        v = x["v"].view(-1, hkv, dv)
        v[x["slots"]] = x["v_new"].view(-1, hkv, dv)
    stored = _fp8 if case["fp8"] else (lambda rows: rows.double())
    outs, lses, at, ek, ev = [], [], 0, [], []
    for s in range(len(x["ctx"])):
        n, c = int(x["q_len"][s]), int(x["ctx"][s])
        pos = np.arange(c, dtype=np.int64)
        sl = torch.from_numpy(x["bt"][s, pos // bs].astype(np.int64) * bs + pos % bs).cuda()
        q = x["q"][at:at + n].double()
        at += n
        ks = stored(k[sl])
        if case["path"] == "expand":
            cpart = ks[:, 0, :512]
            kk = torch.cat([torch.einsum("nc,hcd->nhd", cpart, x["w_uk"].double()), ks[:, :, 512:].expand(-1, hq, -1)], 2)
            vv = torch.einsum("nc,hcd->nhd", cpart, x["w_uv"].double())
            pad = 16 * ((c + 15) // 16) - c
            ek += [kk, kk.new_zeros(pad, hq, 192)]
            ev += [vv, vv.new_zeros(pad, hq, 128)]
            o, l = _attend64(q, kk, vv, 192 ** -0.5)
        else:
            o, l = _attend64(q, ks, ks[:, :, :dv] if latent else stored(v[sl]), dq ** -0.5)
        outs.append(o)
        lses.append(l)
    r = {"out": torch.cat(outs), "lse": torch.cat(lses), "k_cache": None, "v_cache": None}
    if case["path"] == "expand":
        r.update(ek=torch.cat(ek), ev=torch.cat(ev))
    return r
