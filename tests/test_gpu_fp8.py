"""FP8 (E4M3) K/V pages on the GPU against the oracle (needs a B200): the quantiser bit for bit
(codes, scales, tails, summaries of the dequantised keys), then whole denoising blocks on the FP8
cache - index outputs exact, attention within the bf16 tolerances of the definition evaluated on the
dequantised cache - including block finalisation, which re-quantises the touched pages."""
import numpy as np
import pytest

from helpers import OracleFp8Layer
from paper_2604_12056_b200 import workloads as wl
from test_gpu_parity import compare

pytestmark = pytest.mark.gpu


def assert_cache_equal(g, o, cfg):
    from paper_2604_12056_b200.layer import to_host
    kv_len = to_host(g.kv_len)
    assert (kv_len == o.kv_len).all()
    P = [(int(L) + cfg.page_size - 1) // cfg.page_size for L in kv_len]
    pt = to_host(g.page_table)
    used = np.concatenate([pt[s, :P[s]] for s in range(cfg.batch)]) if sum(P) else np.zeros(0, np.int64)
    for name in ("k_codes", "v_codes", "k_scale", "v_scale"):
        assert (to_host(getattr(g, name))[used] == getattr(o, name)[used]).all(), name
    assert (to_host(g.kmin)[used] == wl.elem_to_f32(o.kmin)[used]).all()
    assert (to_host(g.kmax)[used] == wl.elem_to_f32(o.kmax)[used]).all()


def run_fp8_blocks(cfg, n_blocks=1, fused=False, m=None):
    from paper_2604_12056_b200.layer import LosaLayer, to_device
    w = wl.Workload(cfg)                          # the unused tail of a partial last page holds NaN: the quantiser must not read it
    g = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    o = OracleFp8Layer(w)
    assert g.ctx.poll_status() == 0
    assert_cache_equal(g, o, cfg)
    for b in range(n_blocks):
        steps = w.block_steps(m)
        for t, inp in enumerate(steps):
            last = t == len(steps) - 1 and n_blocks > 1
            args = (to_device(inp.q), to_device(inp.k_blk), to_device(inp.v_blk), to_device(inp.m_per_seq))
            (g.run_step_fused if fused else g.run_step)(*args)
            snap = g.snapshot()
            assert g.ctx.poll_status() == 0
            ref = o.run_step(inp, finalize=last)
            if fused:
                snap["delta"] = ref["delta"]
            compare(snap, ref, cfg, f"fp8 {cfg.name} block {b} step {t}")
            if last:
                g.finalize_block(args[1], args[2])
                assert g.ctx.poll_status() == 0
                assert_cache_equal(g, o, cfg)
                assert (g.snapshot()["step"] == 0).all()
    return g, o


@pytest.mark.parametrize("fused", [False, True])
def test_fp8_cache_whole_block(fused):
    run_fp8_blocks(wl.config("c2", kv_lens=(2048, 1500), steps=4), fused=fused)


@pytest.mark.parametrize("g,d,hq,hkv", [(16, 64, 4, 1), (32, 128, 8, 2), (64, 128, 8, 8), (16, 128, 16, 1), (64, 64, 6, 2)])
def test_fp8_cache_ragged_batches_and_page_sizes(g, d, hq, hkv):
    cfg = wl.config("c2", n_q_heads=hq, n_kv_heads=hkv, head_dim=d, page_size=g, kv_lens=(21 * g + 5, 0, 1, 9 * g, 128 + g),
                    block_size=12, steps=3, topk=5, m_active=3)
    run_fp8_blocks(cfg)


def test_fp8_cache_appends_blocks_and_requantises_touched_pages():
    # block of 24 tokens on pages of 16 / 32: every append ends inside a page, so the next one re-quantises it
    for g in (16, 32):
        cfg = wl.config("c5", page_size=g, kv_lens=(200, 90, 64), n_blocks=3, steps=2, topk=4, block_size=24)
        run_fp8_blocks(cfg, n_blocks=3, fused=True)


@pytest.mark.parametrize("g,d", [(16, 64), (32, 64), (64, 64), (16, 128), (32, 128), (64, 128)])
def test_fp8_pages_zero_codes_and_a_block_off_its_alignment(g, d):
    """Every (page size, d) of the page kernels: columns that round to zero codes of both signs, pages of one token,
    odd heads (warps past the last page), and a block whose rows are not 16-byte aligned when it is appended."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer, to_device
    cfg = wl.config("c5", page_size=g, head_dim=d, n_q_heads=6, n_kv_heads=3, kv_lens=(3 * g + 1, 2 * g, 5), steps=1, topk=2,
                    block_size=min(g + 3, 61), n_blocks=2)
    w = wl.Workload(cfg)
    k = wl.bf16_bits_to_f32(w.k_pages)
    k[..., 3::5] = np.sign(k[..., 3::5]) * 1e-6
    w.k_pages[...] = wl.f32_to_bf16_bits(k)
    gl = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    o = OracleFp8Layer(w)
    assert_cache_equal(gl, o, cfg)
    inp = w.block_steps()[0]
    gl.run_step(to_device(inp.q), to_device(inp.k_blk), to_device(inp.v_blk), to_device(inp.m_per_seq))
    o.run_step(inp, finalize=True)
    off = []
    for a in (inp.k_blk, inp.v_blk):
        buf = torch.empty(a.size + 1, dtype=torch.bfloat16, device="cuda")
        buf[1:] = to_device(a).flatten()
        off.append(buf[1:].view(a.shape))
    gl.finalize_block(*off)
    assert gl.ctx.poll_status() == 0
    assert_cache_equal(gl, o, cfg)


def listed_prefix(layer, cfg, s, h):
    """Keys and values [n, d] of the pages listed for sequence s and KV head h as stage 4 must see them: code times
    scale, in float64."""
    import torch
    pages = layer.union_pages[s, h, :int(layer.union_count[s, h])].long()
    valid = (pages[:, None] * cfg.page_size + torch.arange(cfg.page_size, device="cuda")) < layer.kv_len[s]
    phys = layer.page_table[s, pages].long()
    return [(codes[phys, h].view(torch.float8_e4m3fn).double() * scale[phys, h].double()[:, None, None])[valid]
            for codes, scale in ((layer.k_codes, layer.k_scale), (layer.v_codes, layer.v_scale))]


def assert_rows_exact_to_p(layer, cfg, q, s, what, p_bits=11):
    """o_p and lse_p of the last step's active rows against float64 over the listed pages, column by column.  P is
    rounded to fp16 relative to the row's largest weight: half a unit of its p_bits = 11 bits, below 2^-14 half a unit
    of 2^-24, so that a column is off by at most 2^-11 sum p |v| + 2^-25 p_max sum |v|; as much again for the sums
    in fp32 and 2^x."""
    import torch
    G = cfg.n_q_heads // cfg.n_kv_heads
    act = layer.active_idx[s, :int(layer.n_active[s])].long()
    for h in range(cfg.n_kv_heads):
        k, v = listed_prefix(layer, cfg, s, h)
        for i in range(h * G, (h + 1) * G):
            sc = q[s, act, i].double() @ k.T * cfg.sm_scale
            p = torch.softmax(sc, -1)
            bound = 2.0 ** (1 - p_bits) * (p @ v.abs()) + 2.0 ** -24 * p.amax(-1, keepdim=True) * v.abs().sum(0)
            err = (layer.o_p[s, act, i].double() - p @ v).abs()
            assert (err <= bound).all(), f"{what}: sequence {s} head {i}, worst {(err / bound).max():.3g} of the bound"
            assert (layer.lse_p[s, act, i].double() - torch.logsumexp(sc, -1)).abs().max() <= 1e-3, what


@pytest.mark.parametrize("g,d", [(16, 64), (32, 64), (64, 64), (16, 128), (32, 128), (64, 128)])
def test_fp8_pages_of_very_different_scales(g, d):
    """Neighbouring pages whose key and value scales differ (2^-6 .. 2^2 and 2^-6 .. 2^5), a KV head of small value
    scales only, more pages than the staging rings hold, groups that end inside a run of 32 columns."""
    from paper_2604_12056_b200.layer import LosaLayer, to_device
    cfg = wl.config("c2", page_size=g, head_dim=d, n_q_heads=8, n_kv_heads=2, kv_lens=(61 * g - 3, 7 * g), steps=2, topk=3,
                    block_size=16, m_active=3)
    w = wl.Workload(cfg)
    rng = np.random.default_rng(5)
    for pool, factors in ((w.k_pages, (0.25, 1.0, 4.0)), (w.v_pages, (0.03, 1.0, 30.0, 1000.0))):
        f = rng.choice(factors, size=pool.shape[:2]).astype(np.float32)
        if pool is w.v_pages:
            f[:, 1] = factors[0]
        pool[...] = wl.f32_to_bf16_bits(wl.bf16_bits_to_f32(pool) * f[:, :, None, None])
    gl = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    o = OracleFp8Layer(w)
    assert_cache_equal(gl, o, cfg)
    assert len(np.unique(o.k_scale)) > 2 and len(np.unique(o.v_scale)) > 3
    for t, inp in enumerate(w.block_steps()):
        q = to_device(inp.q)
        gl.run_step(q, to_device(inp.k_blk), to_device(inp.v_blk), to_device(inp.m_per_seq))
        snap, ref = gl.snapshot(), o.run_step(inp)
        assert gl.ctx.poll_status() == 0
        for key in ("act", "na", "topk", "up", "uc"):
            assert (snap[key] == ref[key]).all(), key
        for s in range(cfg.batch):                            # the lists are the oracle's: rows against float64 over them
            assert_rows_exact_to_p(gl, cfg, q, s, f"step {t}")
        assert (np.abs(snap["lse_p"] - ref["lse_p"]) <= 1e-3).all()


def hot_token_layer(g, d, at, channel, above, n_tokens, N=1, Hkv=2, G=2):
    """Prompts whose values are those of ordinary low-scale pages (N(0.5, 1)), except for one page of zeros with one
    token of a single large channel; that token's score lies `above` (log2 units) over all others, which are about
    equal.  Returns the layer after its dense step, the config, the queries and sequence 0's expected output."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    Bk = 4
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tokens,) * N, block_size=Bk, steps=1,
                    topk=1, m_active=1)
    P = N * cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7 * g + d + at)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    u = rnd(d)
    u /= u.norm()
    kp = 0.05 * rnd(P, Hkv, g, d)
    kp -= (kp @ u)[..., None] * u                           # orthogonal to the queries' direction
    vp = 0.5 + rnd(P, Hkv, g, d)
    page, tok = torch.arange(N, device="cuda") * cfg.max_pages_per_seq + at // g, at % g
    vp[page] = 0.0
    vp[page, :, tok, 0] = channel
    kp[page, :, tok] = u * (above * float(np.log(2.0)) / (4.0 * cfg.sm_scale))
    q = (4.0 * u + 0.02 * rnd(N, Bk, Hkv * G, d)).bfloat16()
    kb, vb = (rnd(N, Bk, Hkv, d).bfloat16() for _ in range(2))
    table = torch.arange(P, dtype=torch.int32, device="cuda").view(N, -1).contiguous()
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.full((N,), n_tokens, dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    out = torch.empty(q.shape[1:], dtype=torch.float64, device="cuda")
    for i in range(Hkv * G):
        k, v = listed_prefix(layer, cfg, 0, i // G)
        k, v = (torch.cat([a, b[0, :, i // G].double()]) for a, b in ((k, kb), (v, vb)))
        out[:, i] = torch.softmax(q[0, :, i].double() @ k.T * cfg.sm_scale, -1) @ v
    return layer, cfg, q, out


@pytest.mark.parametrize("g,d", [(16, 64), (32, 64), (64, 64), (16, 128), (32, 128), (64, 128)])
@pytest.mark.parametrize("above,channel,at", [(13.0, 30000.0, 3), (14.0, 16000.0, 100), (13.0, 57000.0, 700), (6.0, 400.0, 3), (10.0, 600.0, 3)])
def test_fp8_weights_beside_a_page_of_large_scale(g, d, above, channel, at):
    """The value scale of a page must not cost the weights of pages with smaller scales their bits: the columns that
    only low-scale pages fill are as good as with weights that carry no scale."""
    layer, cfg, q, out = hot_token_layer(g, d, at, channel, above, 1000)
    assert float(layer.v_scale.max()) >= 64 * float(layer.v_scale.min())
    assert_rows_exact_to_p(layer, cfg, q, 0, f"page {g} d {d}")
    assert ((layer.out[0].double() - out).abs() <= 2e-2 + 1e-2 * out.abs()).all()


def test_fp8_output_beside_a_page_of_large_scale_in_a_batch():
    """Eight prompts of 32,000 tokens: a share holds some 440 pages, and the hot token's page is in the first of each
    prompt's.  The low-scale tokens of that share are a sixth of the output's other columns."""
    layer, cfg, q, out = hot_token_layer(16, 128, 3, 30000.0, 13.0, 32000, N=8, Hkv=8, G=1)
    err = (layer.out[0].double() - out).abs()
    assert (err <= 2e-2 + 1e-2 * out.abs()).all(), f"worst {err[..., 1:].max():.3g}"
    assert_rows_exact_to_p(layer, cfg, q, 0, "batch")


@pytest.mark.parametrize("g,d", [(16, 64), (32, 128), (64, 128)])
def test_fp8_scales_of_any_value(g, d):
    """A caller's own scales, not powers of two and below 2^-6 too: every page's code times its scale.  The multiplier, its
    product with a code and P are each rounded to 11 bits: three times 2^-11, so 2^-9 takes their place in the bound."""
    import torch
    from paper_2604_12056_b200 import binding as B
    layer, cfg, q, _ = hot_token_layer(g, d, 3, 400.0, 1.0, 1000)
    for scale, factors in ((layer.k_scale, (1.0, 0.81, 1.3)), (layer.v_scale, (1.0, 1.37, 0.0137, 91.0))):
        scale *= torch.tensor(factors, device="cuda")[torch.arange(len(scale), device="cuda") % len(factors)][:, None]
    B.losa_sparse_prefix_attn(layer.ctx, q, layer.kv, layer.active_idx, layer.n_active, layer.union_pages, layer.union_count, layer.state)
    assert layer.ctx.poll_status() == 0
    assert_rows_exact_to_p(layer, cfg, q, 0, f"page {g} d {d}", p_bits=9)


@pytest.mark.parametrize("g,d", [(16, 64), (16, 128), (32, 64), (32, 128), (64, 64), (64, 128)])
def test_fp8_runs_of_one_page_prompts_in_one_share(g, d):
    """One long prompt beside 40 of a single page, lengths 1 .. g and scales of every size: a CTA's share of the list
    then holds some twenty groups of one page, as many as the staging rings have slots."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    # a one-page segment is charged 11 items: 148 shares of at least 26 of them
    N, Hkv, Bk = 41, 8, 4
    P = 26 * 11 * 148 // Hkv
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + d)
    lens = [P * g] + [1 + int(x) for x in torch.randint(0, g, (N - 1,), generator=gen, device="cuda")]
    cfg = wl.config("c2", n_q_heads=Hkv, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=tuple(lens), block_size=Bk, steps=1,
                    topk=1, m_active=1)
    n_phys = P + N - 1
    f = torch.exp2(torch.randint(-2, 9, (2, n_phys, Hkv, 1, 1), generator=gen, device="cuda"))
    kp = (torch.randn(n_phys, Hkv, g, d, generator=gen, device="cuda") * f[0].clamp_max(4.0)).bfloat16()
    vp = (torch.randn(n_phys, Hkv, g, d, generator=gen, device="cuda") * f[1].clamp_max(64.0)).bfloat16()
    order = torch.randperm(n_phys, generator=gen, device="cuda").to(torch.int32)
    table = torch.zeros(N, cfg.max_pages_per_seq, dtype=torch.int32, device="cuda")
    table[0, :P] = order[:P]
    table[1:, 0] = order[P:]
    q = torch.randn(N, Bk, Hkv, d, generator=gen, device="cuda").bfloat16()
    kb, vb = (torch.randn(N, Bk, Hkv, d, generator=gen, device="cuda").bfloat16() for _ in range(2))
    layer = LosaLayer(cfg, kp, vp, table, torch.tensor(lens, dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    for s in range(1, N):
        assert_rows_exact_to_p(layer, cfg, q, s, f"page {g} d {d}, {lens[s]} tokens")


def test_fp8_cache_dense_mode_and_two_row_groups():
    cfg = wl.config("c4", kv_lens=(64 * 40 + 17,), steps=2, topk=8, m_active=40, heavy_frac=0.0)
    run_fp8_blocks(cfg)


def test_fp8_cache_needs_scales_and_a_bf16_context():
    import ctypes as C
    from paper_2604_12056_b200 import binding as B
    from paper_2604_12056_b200.layer import LosaLayer
    cfg = wl.config("c2", kv_lens=(256,), block_size=8, steps=2, topk=2, m_active=1)
    w = wl.Workload(cfg)
    g = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    bad = B.make_kv(g.k_codes, g.v_codes, g.kmin, g.kmax, g.page_table, g.kv_len, g.k_scale, g.v_scale)
    bad.v_scale = 0
    with pytest.raises(B.LosaError) as e:
        B.losa_sparse_prefix_attn(g.ctx, g.q_prev, bad, g.active_idx, g.n_active, g.union_pages, g.union_count, g.state)
    assert e.value.code == B.LOSA_ERR_INVALID_ARG
    with pytest.raises(B.LosaError) as e:
        B.losa_quantize_kv_pages(g.ctx, g.kv, g.kv)              # source must be a native cache
    assert e.value.code == B.LOSA_ERR_INVALID_ARG


def test_fp8_cache_full_size_c5_layer():
    """One layer of the benchmark's default workload on an FP8 cache: dense first step on sampled
    tokens, the LoSA step in full (the oracle works on the dequantised cache)."""
    import torch
    from oracle import oracle as orc
    from paper_2604_12056_b200.layer import LosaLayer
    from test_gpu_parity import assert_close, assert_lse_close
    cfg = wl.config("c5", n_blocks=1)
    dw = wl.DeviceWorkload(cfg, replica=0, layer=5)
    g = LosaLayer(cfg, dw.k_pages, dw.v_pages, dw.page_table, dw.kv_len, fp8_kv=True)
    o = OracleFp8Layer(dw.host_copy())
    assert_cache_equal(g, o, cfg)
    d0, d1 = dw.start_block(), dw.next_step()
    g.run_step_fused(d0.q, d0.k_blk, d0.v_blk, d0.m_per_seq)
    torch.cuda.synchronize()
    s0 = g.snapshot()
    assert g.ctx.poll_status() == 0
    h0, h1 = d0.host_copy(), d1.host_copy()
    N, B = cfg.batch, cfg.block_size
    sample = np.array([4, 27], np.int32)
    act_s = np.full((N, B), -1, np.int32)
    act_s[:, :2] = sample
    up = np.full((N, cfg.n_kv_heads, cfg.max_pages_per_seq), -1, np.int32)
    up[:, :, :1024] = np.arange(1024, dtype=np.int32)
    uc = np.full((N, cfg.n_kv_heads), 1024, np.int32)
    o.o_p[:] = s0["o_p"]
    o.lse_p[:] = s0["lse_p"]
    orc.sparse_prefix_attn(o.sh, h0.q, o.kv, act_s, np.full(N, 2, np.int32), up, uc, o.o_p, o.lse_p)
    assert_close(s0["o_p"][:, sample], o.o_p[:, sample], cfg.dtype, "fp8 c5 dense step, sampled o_p")
    assert_lse_close(s0["lse_p"][:, sample], o.lse_p[:, sample], "fp8 c5 dense step, sampled lse_p")
    o.q_prev[:] = h0.q
    o.step[:] = 1
    g.run_step_fused(d1.q, d1.k_blk, d1.v_blk, d1.m_per_seq)
    torch.cuda.synchronize()
    s1 = g.snapshot()
    assert g.ctx.poll_status() == 0
    ref = o.run_step(h1)
    s1["delta"] = ref["delta"]
    compare(s1, ref, cfg, "fp8 c5 layer, LoSA step")


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("g,d", [(16, 64), (32, 128), (64, 128)])
def test_reference_maximum_that_passes_between_groups_and_segments(g, d, fp8):
    """Shares of several groups of 128 tokens that cross segments at odd group counts; the largest score of a group
    rises, falls or jumps from group to group, by less and by more than the 2^8 that moves the reference maximum,
    differently for every query row; 36 and 128 query rows (warps without rows)."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv, G, groups = 24, 4, 4, 13
    for Bk in (9, 32):
        n_tok = groups * 128 - 37
        cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tok,) * N, block_size=Bk, steps=1,
                        topk=1, m_active=1)
        P, mp = N * cfg.max_pages_per_seq, cfg.max_pages_per_seq
        gen = torch.Generator(device="cuda")
        gen.manual_seed(11 * g + d + Bk)
        rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
        u = torch.nn.functional.normalize(rnd(2, d), dim=-1)
        kp, vp = 0.1 * rnd(P, Hkv, g, d), rnd(P, Hkv, g, d)
        grp = (torch.arange(mp, device="cuda") * g // 128).float().repeat(N)            # group of a sequence's page
        level = torch.stack([5.0 * grp, 5.0 * (groups - grp), 40.0 * torch.rand(P, generator=gen, device="cuda"), 12.0 * (grp % 2)])   # log2 units
        level = level[torch.arange(P, device="cuda") // mp % 4, torch.arange(P, device="cuda")]           # one kind per sequence
        kp[:, :, 5] += (level * float(np.log(2.0)) / (3.0 * cfg.sm_scale))[:, None, None] * u[0]
        q = 3.0 * u[0] * torch.rand(N, Bk, Hkv * G, 1, generator=gen, device="cuda") + 0.5 * rnd(N, Bk, Hkv * G, d)
        kb, vb = (rnd(N, Bk, Hkv, d).bfloat16() for _ in range(2))
        q = q.bfloat16()
        table = torch.arange(P, dtype=torch.int32, device="cuda").view(N, -1).contiguous()
        layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.full((N,), n_tok, dtype=torch.int32, device="cuda"), fp8_kv=fp8)
        layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
        assert layer.ctx.poll_status() == 0
        for s in range(N):
            if fp8:
                assert_rows_exact_to_p(layer, cfg, q, s, f"{Bk} tokens")
                continue
            for h in range(Hkv):
                k, v = (t[table[s].long(), h].reshape(-1, d)[:n_tok].double() for t in (layer.k_pages, layer.v_pages))
                heads = slice(h * G, (h + 1) * G)
                sc = q[s, :, heads].double() @ k.T * cfg.sm_scale
                p = torch.softmax(sc, -1)
                # P is rounded to 8 significant bits: half a unit of 2^-8 of every weight, as much again for the rest
                assert ((layer.o_p[s, :, heads].double() - p @ v).abs() <= 2.0 ** -8 * (p @ v.abs())).all(), (s, h, Bk)
                assert (layer.lse_p[s, :, heads].double() - torch.logsumexp(sc, -1)).abs().max() <= 1e-4


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("g,d", [(16, 128), (32, 64), (64, 128)])
def test_shares_of_several_short_pieces_with_and_without_rows(g, d, fp8):
    """Some four pieces per CTA of 1 to 7 groups of 128 tokens, 8 to 128 query rows each, in an order in which most softmax
    warps have rows in one piece and none in the next: a piece's output must be read before the next one's first product,
    by warps that handled the last group and by those that did not.  Against float64, and the same bits every time."""
    import torch
    from paper_2604_12056_b200 import binding as B
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv, G, Bk = 64, 8, 8, 16
    n_tok = 7 * 128 - 3
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tok,) * N, block_size=Bk, steps=1,
                    topk=1, m_active=1)
    mp, n_pages = cfg.max_pages_per_seq, 7 * 128 // g
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3 * g + d)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda").bfloat16()
    table = torch.arange(N * mp, dtype=torch.int32, device="cuda").view(N, mp)
    layer = LosaLayer(cfg, rnd(N * mp, Hkv, g, d), rnd(N * mp, Hkv, g, d), table, torch.full((N,), n_tok, dtype=torch.int32, device="cuda"), fp8_kv=fp8)
    q = rnd(N, Bk, Hkv * G, d)
    layer.n_active.copy_(torch.tensor([16, 1, 5, 9, 13, 2, 12, 4], dtype=torch.int32).repeat(N // 8))
    layer.active_idx.fill_(-1)
    layer.union_pages.fill_(-1)
    for s in range(N):
        na = int(layer.n_active[s])
        layer.active_idx[s, :na] = torch.arange(Bk - na, Bk, dtype=torch.int32)
        for h in range(Hkv):
            n = min(n_pages, int(torch.randint(1, 8, (1,), generator=gen, device="cuda")) * (128 // g) - (s + h) % 3 * (g < 64))
            layer.union_pages[s, h, :n] = torch.randperm(n_pages, generator=gen, device="cuda")[:n].sort().values.int()
            layer.union_count[s, h] = n
    first = None
    for _ in range(10):
        layer.o_p.zero_()
        B.losa_sparse_prefix_attn(layer.ctx, q, layer.kv, layer.active_idx, layer.n_active, layer.union_pages, layer.union_count, layer.state)
        assert layer.ctx.poll_status() == 0
        first = (layer.o_p.clone(), layer.lse_p.clone()) if first is None else first
        assert torch.equal(layer.o_p, first[0]) and torch.equal(layer.lse_p, first[1])
    for s in range(N):
        if fp8:
            assert_rows_exact_to_p(layer, cfg, q, s, "fp8")
            continue
        act = layer.active_idx[s, :int(layer.n_active[s])].long()
        for h in range(Hkv):
            pages = layer.union_pages[s, h, :int(layer.union_count[s, h])].long()
            valid = (pages[:, None] * g + torch.arange(g, device="cuda")) < n_tok
            k, v = (t[table[s, pages].long(), h][valid].double() for t in (layer.k_pages, layer.v_pages))
            for i in range(h * G, (h + 1) * G):
                sc = q[s, act, i].double() @ k.T * cfg.sm_scale
                p = torch.softmax(sc, -1)
                # P is rounded to 8 significant bits: half a unit of 2^-8 of every weight, as much again for the rest
                assert ((layer.o_p[s, act, i].double() - p @ v).abs() <= 2.0 ** -8 * (p @ v.abs())).all(), (s, i)
                assert (layer.lse_p[s, act, i].double() - torch.logsumexp(sc, -1)).abs().max() <= 1e-4


@pytest.mark.parametrize("g,d", [(16, 64), (32, 64), (16, 128), (64, 128)])
@pytest.mark.parametrize("power", [-100, -20, 0, 10])
def test_fp8_queries_of_any_magnitude(g, d, power):
    """The queries enter the first product as three E5M2 terms under a scale of the row: rows of every magnitude, elements
    2^-20 .. 1 of a row's largest, a row of zeros, a row of one element; against float64 on the dequantised keys."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    Hkv, G, Bk, n_tok = 2, 4, 8, 3 * 128 + 5
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tok,), block_size=Bk, steps=1, topk=1,
                    m_active=1)
    P = cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + d + power)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    kp, vp = rnd(P, Hkv, g, d) * 2.0 ** max(-6, min(8, -power)), rnd(P, Hkv, g, d)      # (scores of ordinary size where keys can leave them)
    q = rnd(1, Bk, Hkv * G, d) * torch.exp2(torch.randint(-20, 1, (1, Bk, Hkv * G, d), generator=gen, device="cuda").float())
    q[0, 1] = 0.0
    q[0, 2] *= torch.arange(d, device="cuda") == 7
    q[0, 3] = rnd(Hkv * G, d)
    q = (q * 2.0 ** power).bfloat16()
    kb, vb = (rnd(1, Bk, Hkv, d).bfloat16() for _ in range(2))
    table = torch.arange(P, dtype=torch.int32, device="cuda")[None].contiguous()
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.tensor([n_tok], dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(1, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    for h in range(Hkv):
        k, v = listed_prefix(layer, cfg, 0, h)
        for i in range(h * G, (h + 1) * G):
            qd = q[0, :, i].double()
            sc = qd @ k.T * cfg.sm_scale
            # an element is exact down to 2^-24 of its row's largest, which no element here is below: what remains are the
            # fp32 sums, 2^-21 of the sum of magnitudes
            off = cfg.sm_scale * 2.0 ** -21 * (qd.abs() @ k.abs().T).amax(-1)
            lse = torch.logsumexp(sc, -1)
            assert ((layer.lse_p[0, :, i].double() - lse).abs() <= off + 1e-5 + 2.0 ** -22 * lse.abs()).all(), (h, i)
            p = torch.softmax(sc, -1)
            bound = (2.0 ** -10 + 2 * off[:, None]) * (p @ v.abs()) + 2.0 ** -24 * p.amax(-1, keepdim=True) * v.abs().sum(0)
            assert ((layer.o_p[0, :, i].double() - p @ v).abs() <= bound).all(), (h, i)


@pytest.mark.parametrize("g,d", [(16, 128), (64, 64)])
@pytest.mark.parametrize("top,below", [(2, 8), (2, 14), (8, 10), (8, 16), (8, 22), (15, 12), (15, 22)])
def test_fp8_query_elements_far_below_a_large_one_keep_their_bits(g, d, top, below):
    """One element of 2^top per row meets keys of zero, the others are 2^-below of it and make the scores: all eight bits of
    them count.  Against float64 on the dequantised keys; no error but that of fp32 sums."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    Hkv, G, Bk, n_tok = 2, 4, 8, 3 * 128 + 5
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tok,), block_size=Bk, steps=1, topk=1,
                    m_active=1)
    P = cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + d + top + below)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    kp, vp = rnd(P, Hkv, g, d) * 2.0 ** min(13, max(-4, below - top)), rnd(P, Hkv, g, d)       # (keys as large as FP8 pages hold them)
    kp[..., 3] = 0.0
    q = rnd(1, Bk, Hkv * G, d)
    q = q.sign() * (0.5 + q.abs()).clamp_max(3.9) * 2.0 ** (top - below - 1)             # 2^-24 of the largest or more
    q[..., 3] = 1.5 * 2.0 ** top
    q = q.bfloat16()
    kb, vb = (rnd(1, Bk, Hkv, d).bfloat16() for _ in range(2))
    table = torch.arange(P, dtype=torch.int32, device="cuda")[None].contiguous()
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.tensor([n_tok], dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(1, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    for h in range(Hkv):
        k, v = listed_prefix(layer, cfg, 0, h)
        for i in range(h * G, (h + 1) * G):
            qd = q[0, :, i].double()
            sc = qd @ k.T * cfg.sm_scale
            off = cfg.sm_scale * 2.0 ** -21 * (qd.abs() @ k.abs().T).amax(-1)       # fp32 sums
            lse = torch.logsumexp(sc, -1)
            assert ((layer.lse_p[0, :, i].double() - lse).abs() <= off + 1e-5 + 2.0 ** -22 * lse.abs()).all(), (h, i)
            p = torch.softmax(sc, -1)
            bound = (2.0 ** -10 + 2 * off[:, None]) * (p @ v.abs()) + 2.0 ** -24 * p.amax(-1, keepdim=True) * v.abs().sum(0)
            assert ((layer.o_p[0, :, i].double() - p @ v).abs() <= bound).all(), (h, i)


def test_fp8_query_with_an_infinity_or_nan_spoils_its_row_only():
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    cfg = wl.config("c2", n_q_heads=4, n_kv_heads=1, kv_lens=(200,), block_size=4, steps=1, topk=1, m_active=1)
    w = wl.DeviceWorkload(cfg)
    x = w.start_block()
    layer = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    q = x.q.clone()
    q[0, 1, 0, 5] = float("inf")
    q[0, 2, 3, 9] = float("nan")
    layer.run_step(q, x.k_blk, x.v_blk, x.m_per_seq)
    assert layer.ctx.poll_status() == 0
    bad = torch.zeros(4, 4, dtype=torch.bool, device="cuda")
    bad[1, 0] = bad[2, 3] = True
    assert torch.isnan(layer.o_p[0, 1, 0]).all() and torch.isfinite(layer.o_p[0][~bad]).all()
    clean = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    clean.run_step(x.q, x.k_blk, x.v_blk, x.m_per_seq)
    assert (layer.o_p[0][~bad] == clean.o_p[0][~bad]).all()
