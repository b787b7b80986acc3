"""GPU parity of kernel variants that a rule on sizes chooses between, at the sizes where each can go wrong: one tile
and less, tile edges and remainders, the smallest and largest of a variant's range."""
import numpy as np
import pytest
import torch

from oracle import hero_oracle as O
from workloads import synthetic as S
from tests.util import make_pair, rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu


def H():
    import paper_2508_17588_b200 as h
    return h


# One output rounding to bf16 (2^-9 relative at most, 2^-9 / sqrt(3) rms) on top of an fp32 accumulation whose error
# is two orders below it: 2^-9 bounds the relative 2-norm with room to spare.
GEMM_TOL = 2.0 ** -9


@pytest.mark.parametrize("M,N,K", [
    # 148 SMs: CTA pairs on 256 x 256, 224, 192 and 128 tiles; last row tile one row, last column tile 8 columns
    (3841, 2056, 72), (8774, 776, 136), (3073, 3912, 8), (3510, 3080, 520), (2305, 1160, 520), (4097, 3080, 264),
    (681, 3536, 8), (1394, 1024, 1024), (1281, 1160, 1544),
    # one tile per CTA: 128 and 64 columns, K whole or over clusters of two and four CTAs (uneven K runs among them)
    (544, 1968, 8), (640, 3080, 136), (7, 1464, 8), (1, 8, 72), (33, 8, 592), (129, 1096, 520), (257, 520, 1544),
    (136, 2904, 760), (23, 16, 1768), (129, 200, 4104), (300, 776, 3080), (371, 768, 3072), (100, 40, 2056)])
def test_gemm_tile_variants(M, N, K):
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    a = S.round_bf16(rng.standard_normal((M, K)).astype(np.float32))
    w = S.round_bf16((rng.standard_normal((N, K)) / np.sqrt(K)).astype(np.float32))
    bias = S.round_bf16(rng.standard_normal(N).astype(np.float32))
    guard = torch.full((M + 1, N), 7.0, device="cuda", dtype=torch.bfloat16)
    H().hero_gemm_bf16(to_dev(a, "bf16"), to_dev(w, "bf16"), to_dev(bias, "bf16"), guard[:M], 0)
    H().hero_isolated_status()
    want = a.astype(np.float64) @ w.astype(np.float64).T + bias.astype(np.float64)
    assert rel_l2(to_host(guard[:M]), want) <= GEMM_TOL
    assert bool((guard[M] == 7.0).all())


@pytest.mark.parametrize("dtype,B,N,D,n_sel,with_add", [
    # 1 .. 16 packets a lane with the last ones partly or not at all there, few rows and several per warp; wider rows
    # than the warp kernel takes
    ("bf16", 2, 40, 8, 40, True), ("bf16", 1, 9, 264, 9, False), ("bf16", 2, 2700, 1152, 2650, True),
    ("bf16", 3, 2000, 2056, 1900, False), ("bf16", 2, 40, 2816, 17, True), ("bf16", 1, 5000, 4088, 4900, False),
    ("bf16", 1, 20, 4104, 20, True), ("fp32", 2, 3000, 132, 2900, True), ("fp32", 1, 50, 2048, 33, False),
    ("fp32", 1, 5000, 1540, 5000, True), ("fp32", 1, 20, 2052, 20, False), ("bf16", 2, 9, 12288, 5, True),
    ("fp32", 1, 9, 12288, 9, False),
    # one row a warp up to four (rows of two packets a lane and less) and three (five and six) blocks an SM, one more; warps without a row
    ("bf16", 1, 4800, 64, 4736, True), ("bf16", 1, 4800, 64, 4737, True), ("fp32", 2, 1800, 640, 1776, True),
    ("fp32", 2, 1800, 640, 1777, True), ("bf16", 3, 50, 1032, 13, True)])
def test_gather_ln_variants(dtype, B, N, D, n_sel, with_add):
    g = torch.Generator(device="cuda").manual_seed(D + n_sel)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = (torch.randn(B, N, D, device="cuda", generator=g) * 2 + 0.5).to(dt)
    add = (torch.randn(B, N, D, device="cuda", generator=g) * 0.3).to(dt) if with_add else None
    idx = torch.randperm(N, device="cuda", generator=g)[:n_sel].sort().values
    mod = torch.randn(B, 4 * D, device="cuda", generator=g) * 0.5
    out = torch.full((B, n_sel, D), float("nan"), device="cuda", dtype=dt)
    H().hero_gather_ln_modulate(x, add, idx.int(), mod[:, :D], mod[:, D:2 * D], out)
    rows = x[:, idx].double() + (0 if add is None else add[:, idx].double())
    mean = rows.mean(-1, keepdim=True)
    var = (rows - mean).square().mean(-1, keepdim=True)
    want = (rows - mean) / (var + 1e-5).sqrt() * (1 + mod[:, None, D:2 * D].double()) + mod[:, None, :D].double()
    # one rounding to the output type (2^-8 relative at most in bf16) over fp32 statistics of D terms (sqrt(4104) 2^-24)
    tol = 2.0 ** -8 if dtype == "bf16" else 2e-5
    assert float((out.double() - want).abs().max()) <= tol * float(want.abs().max())


# fp32 dot products of up to K = 1540 terms and 1045 keys, summed in fp32: the error of such a sum grows with the root
# of its length, sqrt(1540) * 2^-24 = 2.3e-6, and a block chains a handful of them.
FP32_TOL = 2e-5


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def row_counts(cfgd):
    """Rows per item of a full pass and of a refresh in quota mode 0."""
    return S.n_rows(cfgd), (S.n_rows(cfgd) - cfgd["n_text"]) * cfgd["ratio_num"] // cfgd["ratio_den"]


@pytest.mark.parametrize("over,splits", [
    # attention: head dimensions, one query tile and less, keys whole or split over clusters of 2, 4 and 8 (full, refresh)
    (dict(hidden=128, head_dim=32, n_heads=4, grid_h=5, grid_w=6, n_text=1, batch=1), (1, 1)),       # 31 rows: half a key tile
    (dict(hidden=128, head_dim=64, n_heads=2, grid_h=8, grid_w=8, n_text=1, batch=2), (1, 1)),       # 65 keys: one in tile two
    (dict(hidden=128, head_dim=128, n_heads=1, grid_h=19, grid_w=23, n_text=5, batch=1), (8, 8)),    # 7 tiles over eight
    (dict(hidden=512, head_dim=128, n_heads=4, grid_h=13, grid_w=31, n_text=5, batch=1), (2, 4)),
    (dict(hidden=64, head_dim=64, n_heads=1, grid_h=33, grid_w=31, n_text=22, batch=1), (4, 8)),
    (dict(hidden=384, head_dim=32, n_heads=12, grid_h=11, grid_w=31, n_text=5, batch=1), (2, 4)),
    # widths that are no multiple of a GEMM tile
    (dict(hidden=384, head_dim=32, n_heads=12, ffn_dim=1540, grid_h=19, grid_w=23, n_text=5, batch=2, has_gate=1), (2, 8)),
    (dict(hidden=192, head_dim=64, n_heads=3, ffn_dim=52, grid_h=31, grid_w=33, n_text=0, batch=2), (2, 8)),
], ids=["half_tile", "65_keys", "hd128_eight", "hd128_two_four", "hd64_four_eight", "hd32_two_four", "wide", "narrow_ffn"])
def test_fp32_block_variants(over, splits):
    cfgd = dict(S.CONFIGS["tiny"], n_blocks=1, n_shallow=1, frames=1, seed=41, **over)
    n = S.n_rows(cfgd)
    assert splits == tuple(H().hero_plan_fp32_attention(cfgd["batch"], rows, n, cfgd["n_heads"], cfgd["head_dim"], sms())
                           for rows in row_counts(cfgd))
    orc, hero, _ = make_pair(cfgd)
    x_host = S.tokens(cfgd)
    for s in range(4):                                     # two full passes, two refreshes
        temb = S.temb(cfgd, s)
        want = orc.step(s, x_host, temb)
        x = to_dev(x_host, "fp32")
        hero.hero_step(s, x, to_dev(temb, "fp32"))
        assert rel_l2(to_host(x) - x_host, want - x_host) <= FP32_TOL, s
    hero.close()


@pytest.mark.parametrize("B,frames,grid_h,grid_w,n_text,heads,ratio_den,key_offset", [
    # one block per query group; one query row; one and two query tiles in the last group
    (2, 1, 9, 11, 2, 1, 4, 0), (3, 1, 16, 24, 1, 2, 384, 0), (2, 5, 18, 31, 120, 16, 4, 0),
    # clusters of two, three and four, runs of unequal length, one key in the last tile
    (1, 1, 33, 45, 77, 12, 4, 0), (1, 10, 20, 25, 0, 1, 10, 100), (2, 1, 31, 43, 12, 9, 3, 0), (2, 1, 20, 25, 76, 12, 2, 100),
    # groups cut over all blocks: one whole round and 27 groups, two whole rounds and four groups (37 parts each, one row in
    # the last), with and without rows that the fixed scaling cannot hold (a constant added to all scores of a row)
    (1, 8, 25, 31, 0, 7, 8, 0), (1, 8, 25, 31, 0, 7, 8, 100), (1, 8, 24, 32, 1, 12, 16, 100)])
def test_attention_modes(B, frames, grid_h, grid_w, n_text, heads, ratio_den, key_offset):
    """One block whose attention branch is the attention itself (identity projection, no modulation)."""
    D, N = heads * 64, frames * grid_h * grid_w + n_text
    cfg = dict(n_blocks=1, n_shallow=1, hidden=D, n_heads=heads, head_dim=64, ffn_dim=32, temb_dim=8, batch=B, frames=frames,
               grid_h=grid_h, grid_w=grid_w, n_text=n_text, patch_h=2, patch_w=2, ratio_num=1, ratio_den=ratio_den,
               quota_mode=0, warmup_full_steps=1, full_interval=0, dtype="bf16", has_gate=0, seed=5)
    g = torch.Generator(device="cuda").manual_seed(N + heads)
    mk = lambda *s, std=1.0: (torch.randn(*s, device="cuda", generator=g) * std).bfloat16()
    zero = lambda *s: torch.zeros(*s, device="cuda", dtype=torch.bfloat16)
    w = dict(w_mod=zero(4 * D, 8), b_mod=zero(4 * D), w_qkv=mk(3 * D, D, std=1.5 / D ** 0.5), b_qkv=mk(3 * D, std=0.1),
             w_o=torch.eye(D, device="cuda", dtype=torch.bfloat16), b_o=zero(D), w_1=zero(32, D), b_1=zero(32),
             w_2=zero(D, 32), b_2=zero(D))
    u = torch.randn(heads, 64, device="cuda", generator=g)
    w["b_qkv"][D:2 * D] += (key_offset * u / u.norm(dim=1, keepdim=True)).view(-1).bfloat16()
    hero = H().Hero(cfg, [w])
    temb, idx = mk(B, 8), torch.empty(N, dtype=torch.int32, device="cuda")
    scale = 0.125 * 1.4426950408889634
    for cached in (False, True, True):
        x = mk(B, N, D)
        rows = torch.arange(N, device="cuda")
        xd = x.double()
        if cached:
            n = hero.hero_select_tokens(0, idx)
            rows = idx[:n].long()
            hero.hero_refresh_block(0, x, temb, idx, n)
        else:
            hero.hero_refresh_block(0, x, temb)
        hero.hero_check_status()
        k, v, got = (hero.hero_state_get(0, name).cuda().view(B, N, D) for name in ("k", "v", "g_attn"))
        r = xd[:, rows]
        a = ((r - r.mean(-1, keepdim=True)) / (r.var(-1, unbiased=False, keepdim=True) + 1e-5).sqrt()).bfloat16().double()
        q = ((a @ w["w_qkv"][:D].double().T + w["b_qkv"][:D].double()) * scale).bfloat16()
        want = torch.empty(B, len(rows), D, device="cuda", dtype=torch.double)
        for b in range(B):
            for h in range(heads):
                c = slice(h * 64, h * 64 + 64)
                p = torch.softmax(q[b, :, c].double() @ k[b, :, c].double().T * 0.6931471805599453, -1)
                want[b, :, c] = p @ v[b, :, c].double()
        err = (got[:, rows].double() - want).norm(dim=-1) / want.norm(dim=-1)
        # per row: output rounding 2^-9, weights rounded to 2^-9 each, q 2^-9 (scores of a few units, so the weights move
        # by a few times that); the sum of three bounds with a factor of two for the scores
        assert float(err.max()) <= 2.0 ** -6, (cached, int(err.argmax()))
        assert float((got[:, rows].double() - want).norm() / want.norm()) <= 2.0 ** -7
    hero.close()


@pytest.mark.parametrize("blocks,frames,grid_h,grid_w,patch_h,patch_w,over", [
    # a band (grid rows of one row of patches) of one turn of a warp, of one token more, of a block's 1024 tokens and more
    (1, 2, 9, 16, 2, 3, {}), (2, 2, 9, 11, 3, 4, dict(track_mode=1)), (1, 1, 16, 64, 16, 4, {}), (1, 1, 5, 205, 5, 3, {}),
    (1, 1, 3, 2100, 2, 2, dict(quota_mode=1, ratio_num=1, ratio_den=3)),
    # patches as large as the grid and larger, one row, one column
    (1, 2, 33, 37, 40, 50, dict(ratio_num=1, ratio_den=7)), (1, 1, 1, 1500, 1, 7, dict(quota_mode=1)), (1, 3, 70, 1, 70, 1, {}),
    # more tokens than threads fit the chip, in many bands and in few
    (10, 4, 128, 80, 2, 2, {}), (8, 1, 9, 4300, 3, 3, {})])
def test_selection_variants(blocks, frames, grid_h, grid_w, patch_h, patch_w, over):
    """Lists and ages of all blocks, bit for bit, through calls on one block and through steps (every block at once)."""
    cfgd = dict(dict(S.CONFIGS["tiny"], hidden=64, n_heads=1, head_dim=64, ffn_dim=4, temb_dim=4, n_blocks=blocks,
                     n_shallow=blocks, batch=1, n_text=3, frames=frames, grid_h=grid_h, grid_w=grid_w, patch_h=patch_h,
                     patch_w=patch_w, full_interval=0, warmup_full_steps=1, seed=77), **over)
    cfg = O.Config.from_dict(cfgd)
    w = {k: np.zeros(s, np.float32) for k, s in S.weight_shapes(cfgd).items()}
    hero = H().Hero(cfgd, [H().device_weights(w, "fp32")] * blocks)
    n_rows = 3 + frames * grid_h * grid_w
    for l in range(blocks):                                # (caches as after a full pass)
        for name in ("k", "v", "g_attn", "g_ffn"):
            hero.hero_state_set(l, name, torch.zeros(1, n_rows, 64))
    hero.hero_state_set(0, "steps", torch.tensor([1, 0, 0], dtype=torch.int32))
    ages = [np.zeros(cfg.n_video, np.uint16) for _ in range(blocks)]
    x, temb = torch.zeros(1, n_rows, 64, device="cuda"), torch.zeros(1, 4, device="cuda")
    for call in range(3):
        if call == 2:
            hero.hero_step(1, x, temb)
        for l in range(blocks):
            rows, ages[l] = O.select_tokens(cfg, ages[l], l, call)
            if call < 2:
                idx = torch.full((cfg.n_video,), -1, dtype=torch.int32, device="cuda")
                n = hero.hero_select_tokens(l, idx)
                got = idx.cpu().numpy()
                assert n == len(rows) and np.array_equal(got[:n], rows) and (got[n:] == -1).all()
            assert np.array_equal(hero.hero_state_get(l, "ages").numpy(), ages[l]), (call, l)
    hero.hero_check_status()
    hero.close()


def cut_block(heads=7, **over):
    """A block whose attention cuts its last query groups over all blocks of the grid: 25 groups of 6200 rows a head."""
    cfg = dict(n_blocks=1, n_shallow=1, hidden=heads * 64, n_heads=heads, head_dim=64, ffn_dim=32, temb_dim=8, batch=1, frames=8,
               grid_h=25, grid_w=31, n_text=0, patch_h=2, patch_w=2, ratio_num=1, ratio_den=8, quota_mode=0,
               warmup_full_steps=1, full_interval=0, dtype="bf16", has_gate=0, seed=5, **over)
    hero = H().Hero(cfg, [H().device_weights(S.block_weights(cfg, 0), "bf16")])
    return hero, to_dev(S.tokens(cfg), "bf16"), to_dev(S.temb(cfg, 0), "bf16")


def test_rows_of_cut_groups_are_written_once_when_most_others_are_out_of_range():
    """Ten whole rounds and twenty cut groups, nearly all rows out of the fixed scaling's range: more than a thread block
    keeps a list of.  Slices of 32 rows that are in range stay in the cut groups what they are when all rows are, bit for
    bit, and the whole output repeats itself."""
    B, heads, N = 2, 30, 16 * 25 * 31
    D = heads * 64
    cfg = dict(n_blocks=1, n_shallow=1, hidden=D, n_heads=heads, head_dim=64, ffn_dim=32, temb_dim=8, batch=B, frames=16,
               grid_h=25, grid_w=31, n_text=0, patch_h=2, patch_w=2, ratio_num=1, ratio_den=2, quota_mode=0,
               warmup_full_steps=1, full_interval=0, dtype="bf16", has_gate=0, seed=5)
    g = torch.Generator(device="cuda").manual_seed(11)
    mk = lambda *s, std=1.0: (torch.randn(*s, device="cuda", generator=g) * std).bfloat16()
    zero = lambda *s: torch.zeros(*s, device="cuda", dtype=torch.bfloat16)
    u = torch.randn(heads, 64, device="cuda", generator=g)
    offset = (2000 * u / u.norm(dim=1, keepdim=True)).view(-1)              # a constant of hundreds on all scores of a row
    # keys and values of the refreshed rows do not depend on x: the two runs below see the same
    w = dict(w_mod=zero(4 * D, 8), b_mod=zero(4 * D), w_qkv=zero(3 * D, D), b_qkv=mk(3 * D, std=0.1),
             w_o=torch.eye(D, device="cuda", dtype=torch.bfloat16), b_o=zero(D), w_1=zero(32, D), b_1=zero(32),
             w_2=zero(D, 32), b_2=zero(D))
    w["w_qkv"][:D] = mk(D, D, std=1.5 / D ** 0.5)
    w["b_qkv"][D:2 * D] = offset.bfloat16()
    hero, temb = H().Hero(cfg, [w]), mk(B, 8)
    hero.hero_state_set(0, "k", (torch.randn(B, N, D, device="cuda", generator=g) + offset).bfloat16())
    hero.hero_state_set(0, "v", mk(B, N, D))
    for name in ("g_attn", "g_ffn"):
        hero.hero_state_set(0, name, zero(B, N, D))
    rows = torch.arange(0, N, 2, device="cuda")
    n = len(rows)
    x = mk(B, N, D)
    calm = (torch.arange(n, device="cuda") // 32 % 4 == 1)                  # their queries are the bias alone
    x[:, rows[calm]] = 0

    def attention(x):
        hero.hero_refresh_block(0, x.clone(), temb, rows.int(), n)
        return hero.hero_state_get(0, "g_attn").cuda()[:, rows]

    got = attention(x)
    for _ in range(3):
        assert torch.equal(attention(x), got)
    all_calm = attention(zero(B, N, D))
    hero.hero_check_status()
    q_groups = (n + 255) // 256
    assert B * heads * q_groups == 10 * 148 + 20
    cut = calm & (torch.arange(n, device="cuda") >= (q_groups - 20) * 256)  # of the last head of the last item
    assert torch.equal(got[-1, cut][:, -64:], all_calm[-1, cut][:, -64:])
    k, v = (hero.hero_state_get(0, name).cuda().view(B, N, D) for name in ("k", "v"))
    r = x[:, rows].double()
    a = ((r - r.mean(-1, keepdim=True)) / (r.var(-1, unbiased=False, keepdim=True) + 1e-5).sqrt()).bfloat16().double()
    q = ((a @ w["w_qkv"][:D].double().T + w["b_qkv"][:D].double()) * 0.125 * 1.4426950408889634).bfloat16()
    for b, h in ((0, 0), (0, heads - 1), (1, 3), (1, heads - 1)):
        c = slice(h * 64, h * 64 + 64)
        p = torch.softmax(q[b, :, c].double() @ k[b, :, c].double().T * 0.6931471805599453, -1)
        want = p @ v[b, :, c].double()
        # (a few units of score between the keys on top of the constant: as in test_attention_modes)
        err = (got[b, :, c].double() - want).norm(dim=-1) / want.norm(dim=-1)
        assert float(err.max()) <= 2.0 ** -6 and float((got[b, :, c].double() - want).norm() / want.norm()) <= 2.0 ** -7
    hero.close()


def test_only_a_context_that_may_cut_groups_pays_for_it():
    """The cut attention's workspace (20 MB) is allocated where the largest pass can take it, and nowhere else."""
    def device_bytes(**over):
        cfg = dict(dict(n_blocks=1, n_shallow=1, hidden=448, n_heads=7, head_dim=64, ffn_dim=32, temb_dim=8, batch=1, frames=8,
                        grid_h=25, grid_w=31, n_text=0, patch_h=2, patch_w=2, ratio_num=1, ratio_den=8, quota_mode=0,
                        warmup_full_steps=1, full_interval=0, dtype="bf16", has_gate=0, seed=5), **over)
        w = {k: torch.zeros(s, device="cuda", dtype=torch.bfloat16) for k, s in S.weight_shapes(cfg).items()}
        hero = H().Hero(cfg, [w])
        total = hero.hero_device_bytes()
        hero.close()
        n = S.n_rows(cfg)
        # K, V, two branches, three workspaces and the staged x; FFN rows; lists and counters
        return total - 2 * cfg["batch"] * n * (8 * cfg["hidden"] + cfg["ffn_dim"])
    assert device_bytes() > 15 << 20                                       # 175 groups on 148 SMs, 65 key tiles
    for over in (dict(hidden=320, n_heads=5), dict(frames=7), dict(hidden=64, n_heads=1, frames=1)):
        assert device_bytes(**over) < 1 << 20, over                        # 125 groups; 57 tiles; neither


@pytest.mark.parametrize("then", ["nothing", "reset", "check"])
def test_a_launch_that_gave_up_does_not_reach_into_later_ones(then):
    """What a cut attention keeps between thread blocks is left as by blocks that gave up half way: the next full pass is
    what it is without that, whether or not the caller resets the context or asks for its status first."""
    hero, x0, temb = cut_block()
    hero.hero_refresh_block(0, x0.clone(), temb)
    want = hero.hero_state_get(0, "g_attn")
    hero.hero_check_status()
    for _ in range(2):
        hero.hero_refresh_block(0, -2 * x0.flip(1), temb)              # (leaves parts of other values behind)
        hero.hero_selftest_wait_timeout(50)
        if then == "reset":
            hero.hero_reset()
        if then == "check":
            with pytest.raises(H().HeroError):
                hero.hero_check_status()
        for _ in range(2):
            hero.hero_refresh_block(0, x0.clone(), temb)
            assert torch.equal(hero.hero_state_get(0, "g_attn"), want)
    if then != "check":
        with pytest.raises(H().HeroError):
            hero.hero_check_status()
    hero.hero_check_status()
    hero.close()


@pytest.mark.parametrize("B,n_q,N,heads", [(2, 300, 1000, 3), (1, 129, 97, 1), (1, 513, 2113, 2)])
def test_what_a_thread_block_falls_back_to_is_the_exported_path(B, n_q, N, heads):
    """Rows that the fixed scaling cannot hold (scores rise by far more than 2^100 behind the first 96 keys) come out of
    the attention and of the running maximum alone the same, bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(N)
    mk = lambda *s: torch.randn(*s, device="cuda", generator=g)
    u = torch.nn.functional.normalize(mk(heads, 64), dim=1).view(-1)
    q = (mk(B, n_q, heads * 64) + 40 * u).bfloat16()
    j = torch.arange(N, device="cuda")[:, None]
    k = (mk(B, N, heads * 64) + (j >= 96) * (40 + 20 * j / N) * u).bfloat16()
    v, out, safe = mk(B, N, heads * 64).bfloat16(), torch.empty_like(q), torch.empty_like(q)
    scores = q[:, :, :64].double() @ k[:, :, :64].double().mT * 0.18
    assert float((scores[:, :, -1] - scores[:, :, :96].amax(-1)).amin()) > 100
    H().hero_attention_bf16(q, k, v, out, heads)
    H().hero_attention_bf16_safe(q, k, v, safe, heads)
    H().hero_isolated_status()
    assert torch.equal(out, safe)


@pytest.mark.parametrize("dtype,over", [
    # the pass from block to block: one packet a lane and less, several with the last one partly there, the widest it serves
    # and one beyond; lists of different length from block to block, one list for all, lists that are empty for some blocks
    # of a step and one row for others, a collapsed deep stack
    ("fp32", dict(hidden=64, head_dim=32, n_heads=2, ffn_dim=64, batch=3, n_text=3)),
    ("fp32", dict(hidden=768, head_dim=64, n_heads=12, ffn_dim=64, share_selection=1)),
    ("fp32", dict(hidden=832, head_dim=64, n_heads=13, ffn_dim=64)),
    ("fp32", dict(hidden=64, head_dim=32, n_heads=2, ffn_dim=64, ratio_num=1, ratio_den=90)),
    ("bf16", dict(hidden=64, head_dim=64, n_heads=1, ffn_dim=64)),
    ("bf16", dict(hidden=64, head_dim=64, n_heads=1, ffn_dim=64, n_text=0, ratio_num=1, ratio_den=90)),
    ("bf16", dict(hidden=448, head_dim=64, n_heads=7, ffn_dim=64, deep_collapse=1)),
    ("bf16", dict(hidden=1536, head_dim=64, n_heads=24, ffn_dim=64, batch=1)),
    ("bf16", dict(hidden=1600, head_dim=64, n_heads=25, ffn_dim=64, batch=1)),
    # rows of eight items that a warp has one of at most (448, at three blocks an SM), and one row more: a loop; the last packets
    # of a row partly there; two blocks an SM, where the limit is 296
    ("bf16", dict(hidden=64, head_dim=64, n_heads=1, ffn_dim=64, batch=8, grid_h=21, grid_w=21, n_text=7, n_blocks=3, n_shallow=2)),
    ("bf16", dict(hidden=64, head_dim=64, n_heads=1, ffn_dim=64, batch=8, grid_h=21, grid_w=21, n_text=8, n_blocks=3, n_shallow=2)),
    ("bf16", dict(hidden=448, head_dim=64, n_heads=7, ffn_dim=64, batch=8, grid_h=21, grid_w=21, n_text=8, n_blocks=3, n_shallow=2,
                  ratio_num=1, ratio_den=50)),
    ("fp32", dict(hidden=320, head_dim=64, n_heads=5, ffn_dim=64, batch=8, grid_h=21, grid_w=22, n_text=0, n_blocks=3, n_shallow=2)),
    ("fp32", dict(hidden=448, head_dim=64, n_heads=7, ffn_dim=64, batch=8, grid_h=17, grid_w=17, n_text=8, n_blocks=2, n_shallow=2)),
    # into the deep stack: one refreshed block in front of as many deep ones as a launch holds, and of more
    ("fp32", dict(hidden=64, head_dim=32, n_heads=2, ffn_dim=64, n_blocks=33, n_shallow=1)),
    ("fp32", dict(hidden=64, head_dim=32, n_heads=2, ffn_dim=64, n_blocks=36, n_shallow=2))],
    ids=["fp32_64", "fp32_768_shared", "fp32_832", "fp32_64_sparse", "bf16_64", "bf16_64_sparse", "bf16_448_collapse",
         "bf16_1536", "bf16_1600", "bf16_64_at_one_row", "bf16_64_loop", "bf16_448_loop_sparse", "fp32_320_loop", "fp32_448_loop",
         "deep_32", "deep_34"])
def test_pass_from_block_to_block(dtype, over):
    cfgd = dict(S.CONFIGS["tiny"], frames=1, seed=43, temb_dim=64, dtype=dtype, full_interval=3,
                **{**dict(grid_h=9, grid_w=7, batch=2, n_blocks=5, n_shallow=3, ratio_num=3, ratio_den=10), **over})
    K, sparse = cfgd["n_shallow"], cfgd["ratio_den"] == 90
    orc, hero, _ = make_pair(cfgd)
    for l in range(K):                                     # the blocks' call counters apart, so that their lists differ in length
        orc.blocks[l].calls = 7 - l if sparse else 2 * l
        hero.hero_state_set(l, "calls", torch.tensor([orc.blocks[l].calls], dtype=torch.int32))
    x_host = S.tokens(cfgd)
    lengths = []
    for s in range(7):                                     # full, full, two cached, full, two cached
        temb = S.temb(cfgd, s)
        lists = [O.select_tokens(orc.cfg, b.ages, l, b.calls)[0] for l, b in enumerate(orc.blocks[:K])]
        want = orc.step(s, x_host, temb)
        x = to_dev(x_host, dtype)
        hero.hero_step(s, x, to_dev(temb, dtype))
        # fp32 as above; bf16: x is rounded once per block (independent errors of 2^-9 of x at most, whatever the size of the
        # update), on top of the blocks' own tolerance of 2e-2 of the update
        update = np.linalg.norm(want - x_host)
        bound = FP32_TOL * update if dtype == "fp32" else 5 ** 0.5 * 2.0 ** -9 * np.linalg.norm(want) + 2e-2 * update
        assert np.linalg.norm(to_host(x) - want) <= bound, s
        if orc.is_full_step(s):
            continue
        # What the step refreshed, by itself, within a block's tolerance: keys and values left as they were are 0.14 of their
        # size away and more in all these cases (the embedding and the blocks in front have changed).
        lengths.append([len(r) for r in lists])
        for l, rows in enumerate(lists):
            rows = lists[0] if cfgd.get("share_selection") else rows
            b = orc.blocks[l]
            if len(rows):
                for name, full in (("k", b.k_cache), ("v", b.v_cache), ("g_attn", b.g[0]), ("g_ffn", b.g[1])):
                    got = to_host(hero.hero_state_get(l, name))[:, rows]
                    assert rel_l2(got, full[:, rows]) <= (FP32_TOL if dtype == "fp32" else 2e-2), (s, l, name)
    if K > 1 and not cfgd.get("share_selection"):
        assert any(len(set(n)) > 1 for n in lengths), lengths
    if sparse:
        assert {0, 1} == {n for step in lengths for n in step}
    hero.close()


@pytest.mark.parametrize("dtype,over", [
    ("bf16", dict(hidden=1536, head_dim=64, n_heads=24, grid_h=36, grid_w=32, n_text=32)),     # a warp per row, one each
    ("fp32", dict(hidden=512, head_dim=64, n_heads=8, grid_h=36, grid_w=48, n_text=48)),       # the same
    ("bf16", dict(hidden=1536, head_dim=64, n_heads=24, grid_h=36, grid_w=33, n_text=0))],     # one row more
    ids=["bf16", "fp32", "bf16_several_rows"])
def test_pass_from_block_to_block_behind_an_upload(dtype, over):
    """A cached step from pinned buffers whose first block is done long before x is on the device: 7 MB travel for 0.14 ms
    while a dozen rows of a thin block take a third of that.  The pass behind that block sees all of x, bit for bit."""
    cfgd = dict(S.CONFIGS["tiny"], batch=2, n_blocks=4, n_shallow=3, frames=1, seed=59, temb_dim=64, ffn_dim=64, dtype=dtype,
                full_interval=0, ratio_num=1, ratio_den=90, **over)
    weights = [H().device_weights(S.block_weights(cfgd, l), dtype) for l in range(4)]
    on_device, on_host = H().Hero(cfgd, weights), H().Hero(cfgd, weights)
    g = torch.Generator(device="cuda").manual_seed(4)
    for s in range(8):                                     # two full steps, six cached ones, other tokens every time
        x = torch.randn(2, S.n_rows(cfgd), cfgd["hidden"], device="cuda", generator=g).to(on_device.dt)
        temb = to_dev(S.temb(cfgd, s), dtype)
        h_x = x.cpu().pin_memory()
        on_device.hero_step(s, x, temb)
        on_host.hero_step_host(s, h_x, temb.cpu().pin_memory())
        assert torch.equal(h_x, x.cpu()), s
    for hero in (on_device, on_host):
        hero.hero_check_status()
        hero.close()


@pytest.mark.parametrize("B,n_q,N,heads", [(1, 300, 97, 1), (2, 77, 600, 3), (1, 371, 1562, 12), (2, 640, 6200, 30)],
                         ids=["one_tile", "cluster", "cluster_of_four", "whole"])
def test_attention_output_at_any_16_byte_boundary(B, n_q, N, heads):
    """Rows leave in 32-byte stores where the output allows it, else in 16-byte ones: the same values, nothing beside them."""
    g = torch.Generator(device="cuda").manual_seed(n_q)
    q, k, v = (torch.randn(B, n, heads * 64, device="cuda", generator=g).bfloat16() for n in (n_q, N, N))
    q = q * 0.18
    size = B * n_q * heads * 64
    outs = []
    for shift in (16, 8):                                  # elements: 32 bytes, 16 bytes
        flat = torch.full((size + 32,), 7.0, device="cuda", dtype=torch.bfloat16)
        H().hero_attention_bf16_q_scaled(q, k, v, flat[shift:shift + size].view(B, n_q, heads * 64), heads)
        H().hero_isolated_status()
        assert bool((flat[:shift] == 7.0).all()) and bool((flat[shift + size:] == 7.0).all())
        outs.append(flat[shift:shift + size].clone())
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("over,full,refresh", [
    # (tile, CTAs that share its k) of the QKV, output, up and down projections in the full pass and in the refresh
    (dict(hidden=512, n_heads=8, ffn_dim=2048, grid_h=16, grid_w=19, n_text=5, batch=2),
     ((64, 1), (64, 3), (64, 2), (64, 3)), ((32, 1), (32, 1), (32, 1), (32, 3))),
    # the last row tile eight rows in the full pass, 16 in the refresh
    (dict(hidden=256, n_heads=4, ffn_dim=1024, grid_h=13, grid_w=15, n_text=5, batch=1),
     ((32, 1), (32, 1), (32, 1), (32, 2)), ((32, 1), (32, 1), (32, 1), (32, 4))),
    # k no multiple of a chunk
    (dict(hidden=320, n_heads=5, ffn_dim=1276, grid_h=22, grid_w=26, n_text=25, batch=2, has_gate=1),
     ((64, 1), (32, 1), (64, 1), (64, 4)), ((32, 1), (32, 1), (32, 1), (32, 3))),
    (dict(hidden=384, n_heads=6, ffn_dim=1540, grid_h=8, grid_w=12, n_text=4, batch=1),
     ((32, 1), (32, 1), (32, 1), (64, 8)), ((32, 3), (32, 3), (32, 1), (32, 8))),
    # one row tile, long k; one chunk of k with four of its 128 there
    (dict(hidden=64, n_heads=1, ffn_dim=4092, grid_h=5, grid_w=6, n_text=0, batch=1),
     ((32, 1), (32, 1), (32, 1), (32, 8)), ((32, 1), (32, 1), (32, 1), (32, 8))),
    (dict(hidden=192, n_heads=3, ffn_dim=4, grid_h=7, grid_w=50, n_text=1, batch=1),
     ((32, 1), (32, 1), (32, 1), (32, 1)), ((32, 1), (32, 1), (32, 1), (32, 1)))],
    ids=["width512", "width256", "width320", "width384", "long_k", "short_k"])
def test_fp32_gemm_tiles_and_clusters(over, full, refresh):
    cfgd = dict(S.CONFIGS["tiny"], n_blocks=1, n_shallow=1, frames=1, seed=43, head_dim=64, **over)
    D, F = cfgd["hidden"], cfgd["ffn_dim"]
    for want, rows in zip((full, refresh), row_counts(cfgd)):
        assert want == tuple(H().hero_plan_fp32_gemm(cfgd["batch"] * rows, n, k, sms())
                             for n, k in ((3 * D, D), (D, D), (F, D), (D, F)))
    orc, hero, _ = make_pair(cfgd)
    x_host = S.tokens(cfgd)
    for s in range(3):                                     # two full passes, one refresh
        temb = S.temb(cfgd, s)
        want = orc.step(s, x_host, temb)
        x = to_dev(x_host, "fp32")
        hero.hero_step(s, x, to_dev(temb, "fp32"))
        assert rel_l2(to_host(x) - x_host, want - x_host) <= FP32_TOL, s
    hero.close()


@pytest.mark.parametrize("qk_norm,rope", [(1, 1), (0, 1), (1, 0)])
@pytest.mark.parametrize("over,qkv,down", [
    # tiles of 64 columns, a head each: one row tile and several; the down-projection on 64 columns over two and four CTAs
    (dict(hidden=64, n_heads=1, ffn_dim=2048, grid_h=9, grid_w=10, n_text=7, batch=1), ((64, 1), (64, 1)), ((64, 4), (64, 4))),
    (dict(hidden=448, n_heads=7, ffn_dim=1792, grid_h=17, grid_w=18, n_text=1, batch=2), ((64, 1), (64, 1)), ((64, 2), (64, 4))),
    # tiles of 128 columns in the full pass
    (dict(hidden=512, n_heads=8, ffn_dim=512, grid_h=25, grid_w=20, n_text=0, batch=2), ((128, 1), (64, 1)), ((64, 1), (64, 4)))],
    ids=["one_head", "7_heads", "wide"])
def test_qk_treatment_by_tile_width(over, qkv, down, qk_norm, rope):
    cfgd = dict(S.CONFIGS["tiny"], n_blocks=1, n_shallow=1, frames=1, seed=47, head_dim=64, temb_dim=64, dtype="bf16", rope=rope,
                qk_norm=qk_norm, **over)
    D, F = cfgd["hidden"], cfgd["ffn_dim"]
    rows = [cfgd["batch"] * n for n in row_counts(cfgd)]
    assert qkv == tuple(H().hero_plan_bf16_gemm(m, 3 * D, D, True, sms()) for m in rows)
    assert down == tuple(H().hero_plan_bf16_gemm(m, D, F, False, sms()) for m in rows)
    # scores of a few units, so that the attention says what became of q
    w = S.block_weights(cfgd, 0)
    if qk_norm:
        for name in ("qn_w", "kn_w"):
            w[name] = S.round_bf16(1.5 * w[name])
    else:
        w["w_qkv"][:2 * D] = S.round_bf16(w["w_qkv"][:2 * D] * np.float32(75 / D ** 0.5))
    orc, hero, _ = make_pair(cfgd, [w])
    x_host = S.tokens(cfgd)
    for s in range(3):                                     # two full passes, one refresh
        temb = S.temb(cfgd, s)
        want = orc.step(s, x_host, temb)
        x = to_dev(x_host, "bf16")
        hero.hero_step(s, x, to_dev(temb, "bf16"))
        hero.hero_check_status()
        b = orc.blocks[0]
        blind = b.v_cache.mean(1) @ w["w_o"].astype(np.float64).T + w["b_o"]        # attention that does not look at q
        assert rel_l2(np.broadcast_to(blind[:, None], b.g[0].shape), b.g[0]) > 0.3
        # keys and values are one projection of a LayerNormed row away from x: two roundings to bf16 of the inputs of a
        # K-term sum and one of its result, the latter through the rotation; far below the 2e-2 that a whole block may be off
        for name, ref, tol in (("k", b.k_cache, 1e-2), ("v", b.v_cache, 1e-2), ("g_attn", b.g[0], 2e-2), ("g_ffn", b.g[1], 2e-2)):
            got = to_host(hero.hero_state_get(0, name))
            assert rel_l2(got, ref) <= tol, (s, name)
            ref[...] = got
        update = np.linalg.norm(want - x_host)
        assert np.linalg.norm(to_host(x) - want) <= 2.0 ** -9 * np.linalg.norm(want) + 2e-2 * update, s
    hero.close()
