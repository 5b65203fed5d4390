"""The work this library is used for, as a list of timed cases.

An engine that serves a block-wise diffusion model keeps one paged KV pool and one LoSA cache per attention
layer (`LosaLayer`), ingests a prompt once (page summaries, or quantisation to FP8 pages), and then denoises
block after block: a dense first step, a handful of sparse steps, and the append of the finished block.  A
case names one of those pieces at one size:

  op = "steps"   two consecutive sparse denoising steps of every layer (`losa_denoise_step`): the inner loop.
                 The inputs alternate, so every step has the same number of freshly changed tokens.
       "first"   the first step of a block of every layer: every token active, the whole prefix attended
       "block"   a whole block: first step, `steps` - 1 sparse steps, append of the block to the cache (the
                 lengths are put back first, as when a block is generated again)
       "ingest"  what a new prompt costs before its first step: the page summaries of a cache whose pages are
                 in place, or (kv = "fp8") its quantisation to FP8 pages
  api = "step"   the whole-step call; "stages": the six calls of the interface one by one

Sizes are those of the benchmark's configurations (`workloads.config`), made odd where real prompts are; the
synthetic inputs are `workloads.DeviceWorkload`'s: keys clustered by page, few tokens of a block changing.
"""
from __future__ import annotations

import math

import torch

from paper_2604_12056_b200 import binding as B
from paper_2604_12056_b200 import workloads as wl
from paper_2604_12056_b200.layer import LosaLayer

QWEN = {"q_heads": 32, "kv_heads": 8, "dim": 128}


def _case(name, op, lens, *, page=32, block=32, topk=64, active=3, dtype="bf16", kv="native", selector="exact",
          state="f32", layers=1, steps=8, api="step", heavy=0.0, **heads):
    c = {"name": name, "op": op, "lens": lens, "page": page, "block": block, "topk": topk, "active": active,
         "dtype": dtype, "kv": kv, "selector": selector, "state": state, "layers": layers, "steps": steps,
         "api": api, "heavy": heavy}
    c.update(heads or QWEN)
    return c


def listed():
    return [
        # the smallest use: one fp32 layer with a 1K prefix, a whole 4-step block through the six calls;
        # launches and the host path are all of it
        _case("tiny_f32_block", "block", "1024", page=16, block=16, topk=8, active=4, dtype="f32", steps=4,
              api="stages", q_heads=4, kv_heads=1, dim=64),
        # fp32 at a model's head shape: a whole block of two short ragged prompts (fp32 checks of a model)
        _case("f32_block", "block", "4096,2875", topk=32, dtype="f32"),
        # one interactive sequence with a short prompt, four layers: latency of the sparse step
        _case("one_seq_8k_steps", "steps", "8192", topk=32, layers=4),
        # one sequence, long prompt, short block, small budget, five changed tokens
        _case("one_seq_64k_steps", "steps", "65521", block=16, topk=16, active=5, layers=2),
        # a serving batch of ragged odd prompts, a quarter of the block changing, one list per KV head
        _case("ragged_batch_pooled_steps", "steps", "16381,24571,32768,32003", active=8, selector="pooled", layers=2),
        # very long context, pages and block of 64, heavy-hitter pages
        _case("long_128k_steps", "steps", "131072", page=64, block=64, active=5, layers=2, heavy=0.05),
        # ... and the first step of its block: 256 query rows per KV head over the whole prefix
        _case("long_128k_first", "first", "131072", page=64, block=64, active=5, heavy=0.05),
        # the benchmark's serving batch: eight 32K prompts, the sparse step at the mean number of changed tokens
        _case("batch8_32k_steps", "steps", "32768,32768,32768,32768,32768,32768,32768,32768", layers=2),
        # ... and its dense first step
        _case("batch8_32k_first", "first", "32768,32768,32768,32768,32768,32768,32768,32768"),
        # the same batch on an FP8 cache, a whole block (odd lengths: the append re-quantises partial pages)
        _case("batch8_fp8_block", "block", "32768,32741,32768,31999,32768,32768,30013,32768", kv="fp8"),
        # ingest of a batch of prompts: page summaries of a bf16 cache
        _case("ingest_bf16", "ingest", "32768,32749,16381,8192"),
        # ... and quantisation of the same batch to FP8 pages
        _case("ingest_fp8", "ingest", "32768,32749,16381,8192", kv="fp8"),
    ]


def draw(rng):
    """One more case of the same ranges: 1 to 8 sequences of 1K to 128K tokens (262,144 together, 131,072 for
    a whole block; fp32: 6,144), odd lengths
    among them, every page size, block size, head shape, selector, cache and state format."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    op = rng.choice(["steps", "steps", "steps", "first", "block", "ingest"])
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    batch = rng.choice([1, 1, 2, 3, 4, 8])
    most = (6144 if dtype == "f32" else 131072 if op == "block" else 262144) // batch
    longest = log_int(1024, min(most, 131072))
    lens = [longest] + [max(64, int(longest * rng.uniform(0.4, 1.0))) for _ in range(batch - 1)]
    hq, hkv, d = rng.choice([(32, 8, 128), (32, 8, 128), (32, 8, 128), (32, 4, 128), (16, 8, 128), (16, 4, 64)])
    block = rng.choice([16, 32, 32, 64, 24, 13])
    while block * hq // hkv > 256:
        block //= 2
    return {
        "op": op, "lens": ",".join(str(v) for v in lens), "page": rng.choice([16, 32, 32, 64]), "block": block,
        "topk": log_int(8, 128), "active": max(1, min(block // 2, log_int(1, 16))), "dtype": dtype,
        "kv": "fp8" if dtype == "bf16" and rng.random() < 0.35 else "native",
        "selector": "pooled" if rng.random() < 0.3 else "exact",
        "state": "bf16" if dtype == "bf16" and rng.random() < 0.2 else "f32", "layers": 1, "steps": 4,
        "api": "stages" if rng.random() < 0.2 else "step", "heavy": 0.0, "q_heads": hq, "kv_heads": hkv, "dim": d,
    }


def _lens(case):
    return tuple(int(v) for v in case["lens"].split(","))


def _config(case):
    return wl.Config("case", 9, case["q_heads"], case["kv_heads"], case["dim"], case["page"], _lens(case), case["block"],
                     case["steps"], case["topk"], case["active"], case["dtype"], True, heavy_frac=case["heavy"],
                     rho=0.5 if case["heavy"] else 0.7)


def prepare(case, seed):
    cfg, op = _config(case), case["op"]
    layers = []
    for i in range(case["layers"]):
        w = wl.DeviceWorkload(cfg, replica=seed, layer=i)
        layer = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, pooled=case["selector"] == "pooled",
                          fp8_kv=case["kv"] == "fp8", state_bf16=case["state"] == "bf16")
        n = 0 if op == "ingest" else (2 if op == "steps" else (cfg.steps if op == "block" else 1))
        inputs = []
        for t in range(n):
            inputs.append(w.start_block() if t == 0 else w.next_step())
        layers.append((layer, inputs))
    if op == "steps":                      # the block is under way: its first step is behind it
        for layer, inputs in layers:
            _step(case, layer, inputs[0])
            inputs.append(inputs.pop(0))
    return {"case": case, "layers": layers, "kv_len": [layer.kv_len.clone() for layer, _ in layers],
            "m": torch.full((cfg.batch,), case["active"], dtype=torch.int32, device="cuda")}


def _step(case, layer, x, m=None):
    m = x.m_per_seq if m is None else m
    if case["api"] == "stages":
        layer.run_step(x.q, x.k_blk, x.v_blk, m)
    else:
        layer.run_step_fused(x.q, x.k_blk, x.v_blk, m)


def run(state):
    case, op = state["case"], state["case"]["op"]
    out = []
    for i, (layer, _) in enumerate(state["layers"]):
        if op == "ingest":
            if layer.fp8_kv:
                B.losa_quantize_kv_pages(layer.ctx, layer.kv_native, layer.kv)
                out.append((layer.k_codes, layer.v_codes, layer.k_scale, layer.v_scale, layer.kmin, layer.kmax))
            else:
                B.losa_build_page_summaries(layer.ctx, layer.kv)
                out.append((layer.kmin, layer.kmax))
        elif op == "first":
            layer.step.zero_()
        elif op == "block":
            layer.kv_len.copy_(state["kv_len"][i])
    if op == "ingest":
        return out
    for t in range(len(state["layers"][0][1])):                # in model order: step by step, layer by layer
        for layer, inputs in state["layers"]:
            _step(case, layer, inputs[t], state["m"])
    for layer, inputs in state["layers"]:
        if op == "block":
            layer.finalize_block(inputs[-1].k_blk, inputs[-1].v_blk)
            out += [layer.kv_len, layer.kmin, layer.kmax]
        out.append((layer.out, layer.lse_out, layer.o_p, layer.lse_p, layer.q_prev, layer.active_idx, layer.n_active,
                    layer.union_pages, layer.union_count))
    return out


# ---------------------------------------------------------------- the same results in 64 bits, plain torch
def exact(case, seed):
    """What `run` returns on its first pass over these inputs, in float64 from the definitions.  Index lists, lengths,
    and values that are only copied or picked (page summaries, codes) have no such value: None."""
    if case["op"] == "ingest":
        return None
    cfg, op = _config(case), case["op"]
    out = []
    for i in range(case["layers"]):
        w = wl.DeviceWorkload(cfg, replica=seed, layer=i)
        xs = [w.start_block()] + [w.next_step() for _ in range({"steps": 1, "first": 0}.get(op, cfg.steps - 1))]
        shape = tuple(xs[0].q.shape)
        st = {"o": torch.zeros(shape, dtype=torch.float64, device="cuda"), "merged": None,
              "l": torch.zeros(shape[:3], dtype=torch.float64, device="cuda"), "q": None}
        caches = [_exact_cache(case, w, s) for s in range(cfg.batch)]
        for x in xs + (xs[:1] if op == "steps" else []):
            _exact_step(case, cfg, caches, x, st)
        if op == "block":
            out += [None, None, None]
        out.append((*st["merged"], st["o"], st["l"], st["q"], None, None, None, None))
    return out


def _exact_cache(case, w, s):
    """Keys and values [P, g, H_kv, d] of a prefix (zero past its end), the valid tokens, and each page's min / max keys."""
    L, g = int(w.kv_len[s]), case["page"]
    P = -(-L // g)
    phys = w.page_table[s, :P].long()
    valid = (torch.arange(P * g, device="cuda") < L).view(P, g)
    kv = [t[phys].double().transpose(1, 2).masked_fill(~valid[:, :, None, None], 0.0) for t in (w.k_pages, w.v_pages)]
    if case["kv"] == "fp8":            # E4M3 codes under one power-of-two scale per (page, KV head)
        for j, t in enumerate(kv):
            amax = t.abs().amax((1, 3), keepdim=True)
            scale = 2.0 ** torch.ceil(torch.log2(amax.clamp_min(1e-30) / 448.0)).clamp(-6, 7)
            kv[j] = (t / scale).clamp(-448, 448).to(torch.float8_e4m3fn).double() * scale
    no = ~valid[:, :, None, None]
    return kv[0], kv[1], valid, kv[0].masked_fill(no, math.inf).amin(1), kv[0].masked_fill(no, -math.inf).amax(1)


def _exact_attend(q, k, v, scale):
    """Softmax attention of q [.., n, d] over k, v [t, d]: output and log of the exponentials' sum."""
    sc = q @ k.T * scale
    lse = torch.logsumexp(sc, -1)
    return torch.exp(sc - lse[..., None]) @ v, lse


def _exact_step(case, cfg, caches, x, st):
    G, B = cfg.group, cfg.block_size
    q, kb, vb = x.q.double(), x.k_blk.double(), x.v_blk.double()
    out, lse = torch.empty_like(q), torch.empty_like(st["l"])
    for s, (k, v, valid, kmin, kmax) in enumerate(caches):
        P = k.shape[0]
        if st["q"] is None:
            act = torch.arange(B, device="cuda")
        else:
            delta = (q[s] - st["q"][s]).square().mean((1, 2))
            act = torch.argsort(delta, descending=True, stable=True)[:case["active"]].sort().values
        for h in range(cfg.n_kv_heads):
            heads = slice(h * G, (h + 1) * G)
            qa = q[s, act, heads]
            pages = torch.arange(P, device="cuda")
            if st["q"] is not None:
                u = qa.clamp_min(0) @ kmax[:, h].T + qa.clamp_max(0) @ kmin[:, h].T
                if case["selector"] == "pooled":
                    u = u.amax(1)
                top = torch.argsort(u, dim=-1, descending=True, stable=True)[..., :min(case["topk"], P)]
                pages = torch.unique(top)
            t = valid[pages]
            o, l = _exact_attend(qa, k[pages, :, h][t], v[pages, :, h][t], cfg.sm_scale)
            st["o"][s, act, heads], st["l"][s, act, heads] = o, l
            ob, lb = _exact_attend(q[s, :, heads], kb[s, :, h], vb[s, :, h], cfg.sm_scale)
            lse[s, :, heads] = torch.logaddexp(lb, st["l"][s, :, heads])
            wp = torch.exp(st["l"][s, :, heads] - lse[s, :, heads])[..., None]
            out[s, :, heads] = wp * st["o"][s, :, heads] + torch.exp(lb - lse[s, :, heads])[..., None] * ob
    st["q"], st["merged"] = q, (out, lse)


# Share of the independent draws that a block's selections are worth: the queries of a block share a
# direction, so the distinct pages of n lists of k pages out of P are P (1 - (1 - k/P)^(f n)) with f
# as measured on these inputs (per-head lists, lists pooled over a KV head's heads, heavy-hitter keys).
_OVERLAP = {"exact": 0.5, "pooled": 0.8, "heavy": 0.1}


def work(case):
    lens, g, blk, d, hq, hkv = _lens(case), case["page"], case["block"], case["dim"], case["q_heads"], case["kv_heads"]
    es = 4 if case["dtype"] == "f32" else 2
    kv_es = 1 if case["kv"] == "fp8" else es
    G, n, tokens = hq // hkv, len(lens), sum(lens)
    rows = n * blk * hq * d                                     # elements of q
    summaries = sum(-(-L // g) for L in lens) * hkv * 2 * d * es

    if case["op"] == "ingest":
        b = tokens * hkv * d * (2 * es + 2 * kv_es if case["kv"] == "fp8" else es) + summaries
        return {"bytes": b * case["layers"], "flops": 2 * tokens * hkv * d * case["layers"]}

    o_es = 2 if case["state"] == "bf16" else 4
    block_io = rows * es * (3 + 2 / G)                          # q, block K and V, the output, q kept for the next step
    block_flops = 4.0 * rows * blk

    def first():
        return tokens * hkv * d * 2 * kv_es + block_io + rows * o_es, 4.0 * blk * hq * d * tokens + block_flops

    def sparse():
        b, f = summaries + block_io + rows * (es + o_es), block_flops
        m = min(case["active"], blk)
        for L in lens:
            P = -(-L // g)
            k = min(case["topk"], P)
            lists = m * (1 if case["selector"] == "pooled" else G)
            eff = max(1.0, lists * _OVERLAP["heavy" if case["heavy"] else case["selector"]])
            pages = P * (1.0 - (1.0 - k / P) ** eff)
            b += pages * hkv * min(g, L) * d * 2 * kv_es
            f += 4.0 * m * hq * d * pages * g + 4.0 * m * hq * d * P
        return b, f

    if case["op"] == "first":
        b, f = first()
    elif case["op"] == "steps":
        b, f = sparse()
        b, f = 2 * b, 2 * f
    else:
        b, f = first()
        sb, sf = sparse()
        b += (case["steps"] - 1) * sb + 4 * n * blk * hkv * d * es
        f += (case["steps"] - 1) * sf
    return {"bytes": b * case["layers"], "flops": f * case["layers"]}


def tolerance(case):
    """About four times the largest difference from the same path evaluated in 64 bits on the same lists: fp32 2-norm
    7.8e-7, single values 7.5e-6; bf16 2.4e-3 and 1.4e-2.  Index outputs are exact."""
    if case["op"] == "ingest":
        return "exact"                                          # minima, maxima, codes and scales
    if case["dtype"] == "f32":
        return {"rel": 4e-6, "max": 4e-5, "differ": 0.0}        # fp32 sums
    # P is rounded to 8 significant bits before its product with V, the output (and, where chosen, the state) to bf16
    return {"rel": 1e-2, "max": 0.06, "differ": 0.0}
