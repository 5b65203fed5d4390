"""Selection where only close candidates take exact scores (many lists of 48 pages and more, pooled ones of 60 and more), against the
oracle's lists: pages that tie exactly or differ in one bit of one key, pages that crowd, lists shorter than the budget, more
candidates than a CTA has threads, bounds kept in registers and read again, prefixes that tie as a whole."""
import numpy as np
import pytest

from helpers import OracleLayer
from paper_2604_12056_b200 import workloads as wl
from test_gpu_parity import compare

pytestmark = pytest.mark.gpu

HEADS = dict(n_q_heads=32, n_kv_heads=4, head_dim=64, page_size=16)      # 4 sequences x 32 heads: 128 lists


@pytest.mark.parametrize("pooled", [False, True])
@pytest.mark.parametrize("same", ["few", "pairs", "crowd", "all"])
@pytest.mark.parametrize("kw", [
    dict(kv_lens=(16 * 100, 16 * 60 + 3, 16 * 48, 16 * 49), topk=48),            # 49 pages: every candidate but one is listed
    dict(kv_lens=(16 * 300, 16 * 129 + 1, 700, 0), topk=127),                    # 128 candidates and more: sorted as a whole
    dict(kv_lens=(16 * 1024, 16 * 1025 + 7, 16 * 64, 16 * 33), topk=64, m_active=1),
    dict(kv_lens=(32 * 90, 32 * 130 + 5, 32 * 70, 31), topk=50, page_size=32, head_dim=128, n_q_heads=32, n_kv_heads=8),
    dict(kv_lens=(32 * 600, 32 * 130 + 5, 32 * 70, 32 * 61), topk=60, page_size=32, head_dim=128, n_q_heads=32, n_kv_heads=8),
    dict(kv_lens=(16 * 700, 16 * 500, 16 * 401, 16 * 1100), topk=400, m_active=1),       # up to 512 candidates
])
def test_lists_where_only_close_candidates_take_exact_scores(kw, same, pooled):
    import torch
    from paper_2604_12056_b200.layer import LosaLayer, to_device, to_host
    cfg = wl.config("c2", **{**HEADS, **dict(block_size=4, steps=2, m_active=2), **kw})
    w = wl.Workload(cfg)
    g = cfg.page_size
    for s in range(cfg.batch):                       # (logical pages 2i, 2i + 1; not the last, which may be partial)
        for i in range((int(w.kv_len[s]) // g - 1) // 2):
            a, b = w.page_table[s, 2 * i], w.page_table[s, 2 * i + 1]
            if same == "pairs" or (same == "few" and i % 5 == 0):
                w.k_pages[b] = w.k_pages[a]
                if i % 3 == 0:
                    w.k_pages[b, :, i % g, i % cfg.head_dim] ^= 1        # the last bit of one key element per head
            elif same == "crowd" and i < 20:             # 40 pages of one score: the other way, unless few pages are candidates
                w.k_pages[a] = w.k_pages[b] = w.k_pages[w.page_table[s, 0]]
            elif same == "all":
                w.k_pages[a] = w.k_pages[b] = w.k_pages[w.page_table[s, 0]]
    layers = [LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, pooled=pooled) for _ in range(2)]
    ora = OracleLayer(w, pooled=pooled)
    for t, inp in enumerate(w.block_steps()):
        x = [to_device(v) for v in (inp.q, inp.k_blk, inp.v_blk, inp.m_per_seq)]
        layers[0].run_step_fused(*x)
        layers[1].run_step(*x, want_scores=True)
        torch.cuda.synchronize()
        ref = ora.run_step(inp)
        for layer, what in zip(layers, ("whole step", "six calls")):
            assert layer.ctx.poll_status() == 0
            snap = layer.snapshot()
            if what == "whole step":
                snap["delta"] = ref["delta"]         # (not an output of this call)
            compare(snap, ref, cfg, f"{what} {t}")
        if t == 0:
            continue
        scores = to_host(layers[1].topk_scores)       # in descending order, the whole-step lists being those of the six calls
        for s in range(cfg.batch):
            n = min(cfg.topk, -(-int(w.kv_len[s]) // g))
            for a in range(int(ref["na"][s])):
                row = scores[s, ref["act"][s, a], :, :n]
                assert (np.diff(row, axis=-1) <= 0).all()
