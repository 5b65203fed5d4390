"""Stage 4 on FP8 pages with few query rows (tokens on the tensor cores' lanes, values as an operand): rows about the limit
of 16, value scales about the spread up to which that path is taken, groups of pages that end inside a
product's 32 tokens, rising and falling scores, tails that hold NaN; against float64 over the listed pages."""
import numpy as np
import pytest

from paper_2604_12056_b200 import workloads as wl
from test_gpu_fp8 import assert_rows_exact_to_p, listed_prefix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,d", [(16, 128), (32, 128), (64, 128), (32, 64)])       # (d = 64: the other path)
@pytest.mark.parametrize("m,G", [(1, 1), (5, 3), (4, 4), (17, 1)])               # 1, 15, 16 and 17 rows (17: the other path)
@pytest.mark.parametrize("powers", [(0,), (0, 1, 2), (0, 3), (1, 7), (1, 11), (1, 12), (-9, -8)])    # of the pages' values (a scale is 2^-6 at least)
def test_few_rows_against_float64(g, d, m, G, powers):
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv = 4, 8
    lens = (19000 // g * g + 5, 128 * 149, 20000 // (2 * g) * 2 * g + g, g - 1)   # shares of eight groups and more, which end anywhere
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=lens, block_size=m, steps=1, topk=1,
                    m_active=1)
    mp = cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + d + 7 * m + G + len(powers))
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    u = torch.nn.functional.normalize(rnd(d), dim=-1)
    kp, vp = 0.3 * rnd(N * mp, Hkv, g, d), rnd(N * mp, Hkv, g, d).clamp(-3.4, 3.4)
    # the largest score of a page rises by up to 60 binary places over a prefix (0), falls (1) or jumps (2)
    at = torch.arange(mp, device="cuda").float() / mp
    level = torch.stack([60.0 * at, 60.0 * (1.0 - at), 60.0 * torch.rand(mp, generator=gen, device="cuda"), 0.0 * at]).reshape(-1)
    kp[:, :, 3] += (level * float(np.log(2.0)) / (3.0 * cfg.sm_scale))[:, None, None] * u
    vp[:, :, 0, 0] = 3.5                                    # (every page's largest value: its scale is known)
    vp *= torch.exp2(torch.tensor(powers, device="cuda")[torch.arange(N * mp, device="cuda") % len(powers)].float())[:, None, None, None]
    q = (3.0 * u * torch.rand(N, m, Hkv * G, 1, generator=gen, device="cuda") + 0.5 * rnd(N, m, Hkv * G, d)).bfloat16()
    kb, vb = (rnd(N, m, Hkv, d).bfloat16() for _ in range(2))
    table = torch.randperm(N * mp, generator=gen, device="cuda").int().view(N, mp)
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.tensor(lens, dtype=torch.int32, device="cuda"), fp8_kv=True)
    if powers == (-9, -8):                                  # a caller's own scales, below what the quantiser gives, no powers of two
        layer.v_scale *= 0.013
    for s, n in enumerate(lens):
        if n % g:
            for codes in (layer.k_codes, layer.v_codes):
                codes[table[s, n // g].long(), :, n % g:] = 0x7f
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    for s in range(N):
        assert_rows_exact_to_p(layer, cfg, q, s, f"{m * G} rows")


@pytest.mark.parametrize("odd", [0.0, -1.0, float("inf")])
def test_value_scales_that_are_no_positive_numbers_take_the_other_path(odd):
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    cfg = wl.config("c2", n_q_heads=32, n_kv_heads=8, kv_lens=(80000,), block_size=4, steps=1, topk=1, m_active=1)
    w = wl.DeviceWorkload(cfg)
    x = w.start_block()
    layer = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True)
    layer.v_scale[w.page_table[0, 5].long()] = odd
    layer.run_step(x.q, x.k_blk, x.v_blk, x.m_per_seq)
    assert layer.ctx.poll_status() == 0
    if np.isfinite(odd):
        assert_rows_exact_to_p(layer, cfg, x.q, 0, str(odd))
    else:
        assert not torch.isfinite(layer.o_p).all()


@pytest.mark.parametrize("g", [16, 32, 64])
@pytest.mark.parametrize("powers", [(1, 12), (0, 1)])                         # the other path (scales 2^11 apart), this one
def test_few_rows_in_shares_of_short_pieces(g, powers):
    """Shares of some 30 groups, but pieces of one to ten: a piece ends before the last set of softmax warps has had a group,
    and the share's first one while that set may still be in its walk without a group, whichever path the others are on.
    Against float64, and the same bits every time."""
    import torch
    from paper_2604_12056_b200 import binding as B
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv, G, Bk, d = 64, 16, 4, 4, 128
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + len(powers) + powers[1])
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    lens = tuple(128 * (1 + 3 * s % 10) - (s % 3) * 7 for s in range(N - 1)) + (128 * 10,)
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=lens, block_size=Bk, steps=1, topk=1,
                    m_active=1)
    mp = cfg.max_pages_per_seq
    kp, vp = 0.3 * rnd(N * mp, Hkv, g, d), rnd(N * mp, Hkv, g, d).clamp(-3.4, 3.4)
    vp[:, :, 0, 0] = 3.5                                    # (every page's largest value: its scale is known)
    vp *= torch.exp2(torch.tensor(powers, device="cuda")[torch.arange(N * mp, device="cuda") % 2].float())[:, None, None, None]
    q = rnd(N, Bk, Hkv * G, d).bfloat16()
    kb, vb = (rnd(N, Bk, Hkv, d).bfloat16() for _ in range(2))
    table = torch.arange(N * mp, dtype=torch.int32, device="cuda").view(N, mp)
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.tensor(lens, dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    first = layer.o_p.clone(), layer.lse_p.clone()
    for s in range(N):
        assert_rows_exact_to_p(layer, cfg, q, s, f"scales {powers}")
    for _ in range(20):
        layer.o_p.zero_()
        B.losa_sparse_prefix_attn(layer.ctx, q, layer.kv, layer.active_idx, layer.n_active, layer.union_pages, layer.union_count, layer.state)
        assert layer.ctx.poll_status() == 0
        assert torch.equal(layer.o_p, first[0]) and torch.equal(layer.lse_p, first[1])


def hot_token_per_prompt(g, m, G, powers, above, faint=0):
    """Prompts whose first page holds one token with a score `above` (log2 units) over all others, which are about equal, and in whose
    column 5 only the tokens of page `faint` have values: the column is theirs alone, beside a weight of one.  Long enough for
    twice the shares of eight groups that are this path's least, whatever the number of SMs."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv, d = 2, 8, 128
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_tok = n_sms * 4096 * 2 // (N * Hkv) // g * g + 5
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=(n_tok,) * N, block_size=m, steps=1, topk=1,
                    m_active=1)
    mp = cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + m + G + int(above))
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    u = torch.nn.functional.normalize(rnd(d), dim=-1)
    kp = 0.05 * rnd(N * mp, Hkv, g, d)
    kp -= (kp @ u)[..., None] * u                           # orthogonal to the queries' direction
    vp = rnd(N * mp, Hkv, g, d).clamp(-3.4, 3.4)
    vp[..., 5] = 0.0
    vp[:, :, 0, 0] = 3.5                                    # (every page's largest value: its scale is known)
    vp[faint::mp, :, :, 5] = 1.0 + rnd(N, Hkv, g).abs().clamp_max(2.0)
    vp[0::mp, :, 3, 5] = 0.0
    kp[0::mp, :, 3] = u * (above * float(np.log(2.0)) / (4.0 * cfg.sm_scale))
    vp *= torch.exp2(torch.tensor(powers, device="cuda")[torch.arange(N * mp, device="cuda") % len(powers)].float())[:, None, None, None]
    q = (4.0 * u + 0.02 * rnd(N, m, Hkv * G, d)).bfloat16()
    kb, vb = (rnd(N, m, Hkv, d).bfloat16() for _ in range(2))
    table = torch.arange(N * mp, dtype=torch.int32, device="cuda").view(N, mp)
    layer = LosaLayer(cfg, kp.bfloat16(), vp.bfloat16(), table, torch.full((N,), n_tok, dtype=torch.int32, device="cuda"), fp8_kv=True)
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    return layer, cfg, q


@pytest.mark.parametrize("g", [16, 32, 64])
@pytest.mark.parametrize("m,G", [(1, 1), (4, 4)])
@pytest.mark.parametrize("above", [12, 18, 21, 24])
def test_small_weights_beside_a_large_one_keep_their_bits(g, m, G, above):
    """The reference lies 2^11 below a row's largest weight and P' is an fp16 value: weights keep all eleven bits down to 2^-25
    of it.  So a column that only weights of about 2^-above fill is off by half a unit of each, 2^-11 sum p |v|, and as much
    again for the sums in fp32 and 2^x; nothing is lost on the grid of 2^-24 that fp16 ends with."""
    import torch
    layer, cfg, q = hot_token_per_prompt(g, m, G, (0,), above)
    for s in range(cfg.batch):
        for h in range(cfg.n_kv_heads):
            k, v = listed_prefix(layer, cfg, s, h)
            heads = slice(h * G, (h + 1) * G)
            p = torch.softmax(q[s, :, heads].double() @ k.T * cfg.sm_scale, -1)
            want = p @ v[:, 5]                              # (no value of the column is negative)
            assert (want < 2.0 ** (10 - above)).all() and (want > 2.0 ** (-2 - above)).all()
            assert ((layer.o_p[s, :, heads, 5].double() - want).abs() <= 2.0 ** -10 * want).all(), (s, h)


@pytest.mark.parametrize("g", [16, 32, 64])
@pytest.mark.parametrize("powers,above", [((7, 1), 12), ((7, 1), 18), ((4, 1), 21), ((11, 1), 14)])
def test_small_weights_on_pages_of_small_scale_keep_their_bits(g, powers, above):
    """As above, the large weight on a page whose values are 2^(p0 - p1) as large: a weight's P' carries its page's scale, so it
    keeps eleven bits down to 2^(p0 - p1 - 25) of the row's largest."""
    import torch
    layer, cfg, q = hot_token_per_prompt(g, 4, 4, powers, above, faint=1)
    for s in range(cfg.batch):
        for h in range(cfg.n_kv_heads):
            k, v = listed_prefix(layer, cfg, s, h)
            heads = slice(4 * h, 4 * h + 4)
            p = torch.softmax(q[s, :, heads].double() @ k.T * cfg.sm_scale, -1)
            want = p @ v[:, 5]
            assert ((layer.o_p[s, :, heads, 5].double() - want).abs() <= 2.0 ** -10 * want).all(), (s, h)


@pytest.mark.parametrize("g", [16, 32, 64])
@pytest.mark.parametrize("m,G,powers,few", [(1, 1, (0,), True), (4, 4, (1, 7), True), (16, 1, (11, 1), True), (17, 1, (1,), False),
                                            (4, 4, (1, 12), False), (1, 1, (7, 11, 7), True), (1, 1, (7, 12, 7), False)])
def test_which_path_a_share_takes(g, m, G, powers, few):
    """A weight of 2^-34 of its row's largest is 2^-23 under this path's reference, a value fp16 has, and 2^-27 under the other
    path's, less than half of its smallest: the column tells which one the share took."""
    layer, cfg, _ = hot_token_per_prompt(g, m, G, powers, 34)
    assert ((layer.o_p[..., 5] != 0) == few).all()


@pytest.mark.parametrize("g", [16, 32, 64])
@pytest.mark.parametrize("powers", [(1,), (1, 12)])                           # this path, the other one
@pytest.mark.parametrize("where", ["key scale", "key code", "query"])
def test_values_that_are_no_numbers_stay_in_the_cached_state(g, powers, where):
    """A listed page whose key scale or one of whose key codes is NaN leaves NaN in o_p of all rows of its KV head, and a query
    with an infinity in o_p of its row; no others."""
    import torch
    from paper_2604_12056_b200 import binding as B
    G, m, page = 4, 4, 901
    layer, cfg, q = hot_token_per_prompt(g, m, G, powers, 12)
    bad = torch.zeros(cfg.batch, m, cfg.n_q_heads, dtype=torch.bool, device="cuda")
    phys = int(layer.page_table[1, page])
    if where == "query":
        q[1, 2, 9, 7] = float("inf")
        bad[1, 2, 9] = True
    else:
        bad[1, :, 2 * G:3 * G] = True
        if where == "key scale":
            layer.k_scale[phys, 2] = float("nan")
        else:
            layer.k_codes[phys, 2, 5, 77] = 0x7f
    B.losa_sparse_prefix_attn(layer.ctx, q, layer.kv, layer.active_idx, layer.n_active, layer.union_pages, layer.union_count, layer.state)
    assert layer.ctx.poll_status() == 0
    assert torch.isnan(layer.o_p[bad]).all() and torch.isfinite(layer.o_p[~bad]).all()
    assert not torch.isfinite(layer.lse_p[bad]).any() and torch.isfinite(layer.lse_p[~bad]).all()


def assert_this_path(layer, cfg, rows):
    """What launch and kernel decide by: the table's length, the rows, the pages listed."""
    import torch
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert layer.union_count.numel() * cfg.max_pages_per_seq * cfg.page_size >= n_sms * 32 * 128
    assert rows <= 16 and int(layer.union_count.sum()) >= n_sms * 128 // cfg.page_size


@pytest.mark.parametrize("state_bf16", [False, True])
@pytest.mark.parametrize("pooled", [False, True])
def test_few_rows_of_whole_steps(pooled, state_bf16):
    """Short prompts in a table for long ones: sparse steps through the whole-step call, both selectors and state formats,
    against the six calls' bits and float64 over the listed pages; the first step, with all rows, beside them."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    N, m, lens = 4, 3, (2500, 3000, 1801, 2200)
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    cfg = wl.config("c2", kv_lens=(n_sms * 32 * 128 // (N * 8) + 64,) * N, block_size=16, steps=4, topk=24, m_active=m)
    w = wl.DeviceWorkload(cfg)
    layers = [LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True, pooled=pooled, state_bf16=state_bf16) for _ in range(2)]
    exact = LosaLayer(cfg, w.k_pages, w.v_pages, w.page_table, w.kv_len, fp8_kv=True, pooled=pooled)
    for layer in layers + [exact]:
        layer.kv_len.copy_(torch.tensor(lens, dtype=torch.int32))
    for t in range(4):
        x = w.start_block() if t == 0 else w.next_step()
        args = (x.q, x.k_blk, x.v_blk, torch.full((N,), m, dtype=torch.int32, device="cuda"))
        layers[0].run_step_fused(*args)
        layers[1].run_step(*args)
        exact.run_step_fused(*args)
        assert all(layer.ctx.poll_status() == 0 for layer in layers + [exact])
        if t > 0:
            assert_this_path(layers[0], cfg, m * 4)
        for name in ("active_idx", "n_active", "union_count", "o_p", "lse_p"):
            assert torch.equal(getattr(layers[0], name), getattr(layers[1], name)), (t, name)
        assert torch.equal(layers[0].o_p.bfloat16(), exact.o_p.bfloat16())
        for s in range(N):
            assert_rows_exact_to_p(exact, cfg, x.q, s, f"step {t}")


@pytest.mark.parametrize("g", [16, 32, 64])
def test_few_rows_of_one_page_prompts(g):
    """Some thousand segments of one or two pages, partial ones among them: every group is a piece of its own."""
    import torch
    from paper_2604_12056_b200.layer import LosaLayer
    N, Hkv, G, Bk, d = 64, 16, 4, 4, 128
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    lens = tuple((1 + (s % 2) * (g < 32)) * g - s % 5 for s in range(N - 1)) + (n_sms * 32 * 128 // (N * Hkv) + g,)
    cfg = wl.config("c2", n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=d, page_size=g, kv_lens=lens, block_size=Bk, steps=1, topk=1,
                    m_active=1)
    mp = cfg.max_pages_per_seq
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda").bfloat16()
    table = torch.arange(N * mp, dtype=torch.int32, device="cuda").view(N, mp)
    layer = LosaLayer(cfg, rnd(N * mp, Hkv, g, d), rnd(N * mp, Hkv, g, d), table, torch.tensor(lens, dtype=torch.int32, device="cuda"), fp8_kv=True)
    q, kb, vb = rnd(N, Bk, Hkv * G, d), rnd(N, Bk, Hkv, d), rnd(N, Bk, Hkv, d)
    layer.run_step(q, kb, vb, torch.ones(N, dtype=torch.int32, device="cuda"))
    assert layer.ctx.poll_status() == 0
    assert_this_path(layer, cfg, Bk * G)
    for s in range(N):
        assert_rows_exact_to_p(layer, cfg, q, s, f"prompt {s}")


def test_few_rows_expired_wait_is_reported_and_the_context_stays_usable():
    """With the bound of its waits set to a few cycles every CTA gives up at the first one that is not satisfied at once, on this path
    before or behind the choice of it: the call reports it and ends, and the next one, with the default bound, is right."""
    import torch
    from paper_2604_12056_b200 import binding as B
    layer, cfg, q = hot_token_per_prompt(32, 4, 4, (1,), 12)
    want = layer.o_p.clone(), layer.lse_p.clone()
    call = lambda: B.losa_sparse_prefix_attn(layer.ctx, q, layer.kv, layer.active_idx, layer.n_active, layer.union_pages, layer.union_count, layer.state)
    layer.ctx.set_wait_limit(1)
    call()
    assert layer.ctx.poll_status() == B.LOSA_ERR_TIMEOUT
    layer.ctx.set_wait_limit(0)
    layer.o_p.zero_()
    call()
    assert layer.ctx.poll_status() == 0
    assert torch.equal(layer.o_p, want[0]) and torch.equal(layer.lse_p, want[1])
