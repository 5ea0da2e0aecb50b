"""What is timed: the calls that a serving engine makes per attention layer of a prefill step.

A case is one batch shape with the plan, workspace and list buffers such an engine keeps from layer to layer, and `op`
says which calls it makes:

  sparse  fp2_select_blocks + fp2_sparse_prefill (the path itself);
  chunk   the same for one chunk of a chunked prefill, the pooled means of the cached prefix taken over from the
          previous chunk's workspace first (fp2_pool_carry);
  dense   fp2_dense_prefill (what an engine falls back to where it does not want pruning);
  index   fp2_select_blocks + fp2_export_csr (the index stage for a consumer with an attention kernel of its own).

Inputs are drawn on the GPU after the recipe of paper_2608_19758_b200/inputs.py: noise plus a locality signal, an
attention sink and a few vertical keys per KV head, pages shuffled over one pool.  `kept` is the share of the candidate
blocks that the threshold keeps on such inputs, as measured; only work() reads it.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2608_19758_b200 import binding

D, B = 128, 128


def _case(op, dtype, seqs, lo, hi, prefix, hq, hkv, page, alpha, kept, lens=0):
    return dict(op=op, dtype=dtype, seqs=seqs, lo=lo, hi=hi, prefix=prefix, hq=hq, hkv=hkv, page=page, alpha=alpha,
                kept=kept, lens=lens)


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)
    return [
        # one short prompt of a small model on unpaged (one page per block) memory: latency and launches
        named("short_prompt_2k", "sparse", "bf16", 1, 2048, 2048, 0.0, 4, 1, 128, 0.1, 0.67),
        # many short prompts at once, none of a round length, group size 7
        named("short_batch_g7", "sparse", "bf16", 24, 60, 1500, 0.0, 28, 4, 16, 0.1, 0.93, lens=1),
        # one prompt of middling length at the density reported for such lengths
        named("prompt_8k_fp8", "sparse", "fp8", 1, 8191, 8191, 0.0, 28, 4, 64, 1e-3, 0.29),
        named("prompt_32k", "sparse", "bf16", 1, 32768, 32768, 0.0, 32, 8, 64, 1e-3, 0.15),
        # the long prompts the path is made for, at the 95 % sparsity reported for that length
        named("prompt_128k", "sparse", "bf16", 1, 131072, 131072, 0.0, 32, 8, 64, 4.6e-3, 0.047),
        named("prompt_128k_fp8", "sparse", "fp8", 1, 131072, 131072, 0.0, 28, 4, 64, 6.3e-3, 0.041),
        # a continuous batch: ragged lengths, up to three quarters of a sequence already in the cache, default threshold
        named("batch_256k", "sparse", "bf16", 16, 1024, 65536, 0.75, 32, 8, 16, 0.1, 0.045, lens=2),
        named("batch_256k_fp8", "sparse", "fp8", 16, 1024, 65536, 0.75, 32, 8, 16, 0.1, 0.045, lens=2),
        # the last 8192 tokens of a chunked prefill of a long prompt
        named("chunk_8k_of_128k", "chunk", "bf16", 1, 131072, 131072, 0.9375, 32, 8, 64, 4.6e-3, 0.042),
        # no pruning
        named("dense_32k", "dense", "bf16", 1, 32768, 32768, 0.0, 32, 8, 64, 0.0, 1.0),
        named("dense_16k_fp8", "dense", "fp8", 1, 16384, 16384, 0.0, 28, 4, 64, 0.0, 1.0),
        # block lists handed to somebody else's kernel
        named("index_64k", "index", "bf16", 1, 65536, 65536, 0.0, 32, 8, 64, 0.01, 0.06),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("sparse", "sparse", "sparse", "sparse", "chunk", "dense", "index"))
    dtype = rng.choice(("bf16", "bf16", "fp8"))
    hq, hkv = rng.choice(((4, 1), (8, 2), (28, 4), (32, 8), (32, 8), (32, 4), (16, 16)))
    page = rng.choice((16, 16, 32, 64, 64, 128))
    # heads x tokens (squared for the dense path) stay below those of the largest listed cases
    most = 32768 if op == "dense" else 131072
    seqs = 1 if op == "chunk" else rng.choice((1, 1, 1, _log_uniform(rng, 2, 32)))
    alpha = 0.0 if op == "dense" else rng.choice((0.1, 0.1, 0.05, 0.02, 0.01, 4.6e-3))
    if op == "index":
        seqs = 1   # long enough that more than the always-kept blocks are at stake
    if seqs == 1:
        n = _log_uniform(rng, {"chunk": 4096, "index": 8192}.get(op, 300), most)
        if rng.random() < 0.3:
            n = max(256, n // 256 * 256)
        lo = hi = n
    else:
        hi = _log_uniform(rng, 512, 16384 if op == "dense" else 32768)
        lo = max(16, hi // rng.choice((4, 16, 64)))
        seqs = max(2, min(seqs, (most if op == "dense" else 2 * most) // hi))
    prefix = rng.uniform(0.5, 0.95) if op == "chunk" else rng.choice((0.0, 0.0, round(rng.uniform(0.1, 0.75), 3)))
    c = _case(op, dtype, seqs, lo, hi, round(prefix, 4), hq, hkv, page, alpha, 1.0, lens=rng.randrange(1 << 30))
    if op != "dense":
        # sink, window and diagonal blocks are always kept; of the others about this share
        other = 0.6 * (0.1 / alpha) ** 0.45 * 10.0 / max(20.0, hi / B)
        c["kept"] = round(min(1.0, 7.0 * B / (hi / 2 + 3.5 * B) + min(0.6, 0.05 * other)), 4)
    return c


def lengths(case):
    """[(KV tokens, of these cached before the call)] of the batch: part of its shape, the same for every seed."""
    if case["seqs"] == 1:
        n = case["hi"]
        pre = int(n * case["prefix"])
        return [(n, pre)]
    rng = random.Random(case["lens"])
    out = []
    for _ in range(case["seqs"]):
        n = _log_uniform(rng, case["lo"], case["hi"])
        out.append((n, int(n * rng.uniform(0.0, case["prefix"]))))
    return out


def _quantize(x):
    """Per-head e4m3 (dim 1 = heads): bits and scales."""
    scale = (x.abs().amax(dim=(0, 2)) / 448.0).clamp_min(1e-12)
    bits = (x / scale[None, :, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
    return bits, scale.float()


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(0x5EED + 7919 * int(seed))
    hq, hkv, p = case["hq"], case["hkv"], case["page"]
    g = hq // hkv
    seqs = lengths(case)
    fp8 = case["dtype"] == "fp8"

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device=dev)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device=dev)

    need = [-(-n // p) for n, _ in seqs]
    pool = sum(need) + max(1, sum(need) // 10 if len(seqs) > 1 else 0)
    ids = torch.randperm(pool, generator=gen, device=dev).to(torch.int32)
    table = torch.full((len(seqs), max(need)), -1, dtype=torch.int32, device=dev)
    keep = torch.float32 if fp8 else torch.bfloat16
    total_q = sum(n - pre for n, pre in seqs)
    q = torch.empty(total_q, hq, D, dtype=keep, device=dev)
    k = torch.zeros(pool * p, hkv, D, dtype=keep, device=dev)
    v = torch.zeros(pool * p, hkv, D, dtype=keep, device=dev)
    cu, first_page = [0], 0
    for b, (n, pre) in enumerate(seqs):
        table[b, :need[b]] = ids[first_page:first_page + need[b]]
        first_page += need[b]
        tok = torch.arange(n, device=dev)
        slot = table[b][tok // p].long() * p + tok % p
        period = torch.exp(rand(hkv, 8) * math.log(16.0) + math.log(256.0))
        phase = rand(hkv, 8, D) * (2.0 * math.pi)
        w = randn(hkv, D)
        w = w / w.norm(dim=1, keepdim=True) * math.sqrt(D)
        vert = (rand(hkv, 16) * n).long()
        for h in range(hkv):
            ang = tok[:, None] * (2.0 * math.pi / period[h])
            u = 1.5 / math.sqrt(8.0) * (ang.cos() @ phase[h].cos() - ang.sin() @ phase[h].sin())
            kh = randn(n, D) + u
            kh[:4] += 4.0 * w[h]
            kh[vert[h].unique()] += 3.0 * w[h]
            k[slot, h] = kh.to(keep)
            v[slot, h] = randn(n, D).to(keep)
            q[cu[-1]:cu[-1] + n - pre, h * g:(h + 1) * g] = (randn(n - pre, g, D) + u[pre:, None] + 0.5 * w[h]).to(keep)
        cu.append(cu[-1] + n - pre)
    qs = ks = vs = None
    if fp8:
        (q, qs), (k, ks), (v, vs) = _quantize(q), _quantize(k), _quantize(v)
    k, v = k.view(pool, p, hkv, D), v.view(pool, p, hkv, D)

    def plan_for(seqs, cu):
        return binding.Plan(dict(num_seqs=len(seqs), total_q=cu[-1], num_q_heads=hq, num_kv_heads=hkv, head_dim=D,
                                 block_size=B, tile_rows=128, page_size=p, num_pages=pool,
                                 max_pages_per_seq=table.shape[1], sink_tokens=256, window_tokens=512,
                                 use_correction=1, alpha=case["alpha"], softmax_scale=0.0, dtype=1 if fp8 else 0),
                            cu, [n for n, _ in seqs])

    plan = plan_for(seqs, cu)
    s = dict(op=case["op"], plan=plan, q=q, k=k, v=v, table=table, qs=qs, ks=ks, vs=vs,
             cu=torch.tensor(cu, dtype=torch.int32, device=dev),
             lk=torch.tensor([n for n, _ in seqs], dtype=torch.int32, device=dev),
             ws=plan.new_workspace(), lists=plan.new_lists(),
             out=torch.empty(total_q, hq, D, dtype=torch.bfloat16, device=dev),
             lse=torch.empty(hq, total_q, dtype=torch.float32, device=dev))
    if case["op"] == "chunk":
        # the chunk before this one: its pooled means are in its workspace
        (n, pre), = seqs
        new = min(n - pre, pre)
        s["prev"] = plan_for([(pre, pre - new)], [0, new])
        s["prev_ws"] = s["prev"].new_workspace()
        binding.fp2_pool_blocks(s["prev"], k, v, table, torch.tensor([pre], dtype=torch.int32, device=dev), ks, vs,
                                s["prev_ws"])
    if case["op"] == "index":
        s["csr_cu"] = torch.zeros(plan.num_segments + 1, dtype=torch.int32, device=dev)
        s["csr_idx"] = torch.zeros(plan.idx_capacity * 2, dtype=torch.int32, device=dev)
    return s


def run(s):
    plan, op = s["plan"], s["op"]
    off, cnt, idx = s["lists"]
    if op == "dense":
        binding.fp2_dense_prefill(plan, s["q"], s["k"], s["v"], s["table"], s["cu"], s["lk"], s["qs"], s["ks"], s["vs"],
                                  s["out"], s["lse"], s["ws"])
        return s["out"], s["lse"]
    if op == "chunk":
        binding.fp2_pool_carry(plan, s["ws"], s["prev"], s["prev_ws"], [0])
    binding.fp2_select_blocks(plan, s["q"], s["k"], s["v"], s["table"], s["cu"], s["lk"], s["qs"], s["ks"], s["vs"],
                              off, cnt, idx, s["ws"])
    if op == "index":
        binding.fp2_export_csr(plan, cnt, idx, 64, s["csr_cu"], s["csr_idx"], s["ws"])
        return off, cnt, idx, s["csr_cu"], s["csr_idx"]
    binding.fp2_sparse_prefill(plan, s["q"], s["k"], s["v"], s["table"], s["cu"], s["lk"], off, cnt, idx, s["qs"],
                               s["ks"], s["vs"], s["out"], s["lse"], s["ws"])
    return off, cnt, idx, s["out"], s["lse"]


def work(case):
    """Bytes: queries, keys and values in, outputs and lists out, once each.  FLOPs: the pooled scores of every candidate
    block, exact attention over the kept ones (for the dense path: over the visible keys)."""
    g = case["hq"] // case["hkv"]
    e = 1 if case["dtype"] == "fp8" else 2
    nbytes = flops = 0.0
    for n, pre in lengths(case):
        lq = n - pre
        rows = lq * case["hq"]
        nbytes += rows * D * e + 2.0 * n * case["hkv"] * D * e
        if case["op"] != "index":
            nbytes += rows * (2 * D + 4)
        visible = lq * pre + lq * (lq + 1) / 2.0
        if case["op"] == "dense":
            flops += 4.0 * D * visible * case["hq"]
            continue
        flops += 2.0 * D * visible / B * case["hq"]
        pairs = visible * g / (B * 128.0) * case["hkv"]
        nbytes += 4.0 * case["kept"] * pairs * (3 if case["op"] == "index" else 1)
        if case["op"] != "index":
            flops += 4.0 * D * visible * case["hq"] * case["kept"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Outputs are BF16 and the probabilities 16-bit: against attention in 64 bits the path shows 1.8e-3, at most 0.011 in
    # a value, and with its sums cut into parts up to 0.011 in a value.  A block whose energy is within rounding of the
    # threshold may fall either way, which moves entries of one list.
    if case["op"] == "index":
        return {"rel": 0.0, "differ": 1e-4}
    return {"rel": 7e-3, "max": 0.045, "differ": 1e-4}
