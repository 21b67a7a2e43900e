"""Attention at the ends of what it accepts."""
import numpy as np
import pytest
import torch

from paper_2510_13161_b200 import inputs as I
from tests.helpers import make_mirror, oracle_attention
from tests.test_gpu_attn import compare, run_gpu
from tests.test_gpu_attn_fp8 import run_and_compare, small
from tests.test_gpu_attn_tiles import config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,kappa,gamma", [(2 * 353, 5, 10), (2 * 353, 4, 13), (2 * 149, 9, 14)])       # 153, 159 and 156 row tiles of whole nodes
def test_more_row_tiles_than_sms(hq, kappa, gamma):
    cfg = config(hq, 2, 64, kappa, gamma, 20, 40, batch=1)
    x = I.gen_verify_inputs(cfg, 3, "cuda", with_lm_head=False)
    out, lse = run_gpu(make_mirror(cfg), x)
    compare(out, lse, oracle_attention(x), range(cfg.layers))


def test_very_many_units():
    """2^24 units of one token each: a token that sees only itself gets its own value back."""
    L, B, H, d = 128, 1024, 128, 64
    cfg = I.VerifyConfig("t", 1024, H, H, d, L, B, 0, 0, 1, 1, 64, "greedy", 0.02, 1.0)
    m = make_mirror(cfg)
    new = lambda: torch.zeros((L, B, 1, H, d), dtype=torch.bfloat16, device="cuda")       # noqa: E731
    pool = torch.zeros((L, 1, H, 16, d), dtype=torch.bfloat16, device="cuda")
    q, k, v, out = new(), new(), new().normal_(0, 1), new()
    kv = m.kv(pool, pool, torch.zeros((B, 1), dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda"))
    tree = m.tree(torch.zeros((B, 1), dtype=torch.int32, device="cuda"), 1, 1, parent=[-1])
    m.mirror_attn_verify(kv, tree, q, k, v, out=out)
    assert m.device_status() == (0, 0)
    assert torch.equal(out, v)


@pytest.mark.parametrize("hq", [4, 32])                     # one row tile per head, and two
@pytest.mark.parametrize("grow", [13.0, 30.0, 50.0])        # nats by which the last page's scores exceed those of the first tile
def test_large_values_behind_scores_that_grow(hq, grow):
    """Values of 1e25 under weights that grow along the keys: sums of weights times values stay in fp32's range."""
    cfg = config(hq, 2, 128, 2, 4, 600, 600, batch=1)
    x = I.gen_verify_inputs(cfg, 9, "cuda", with_lm_head=False, shuffle_pages=False)
    x.q.fill_(1.0)
    x.k_pool.zero_(); x.k_new.zero_()
    page = int(x.page_table[0, 36])
    x.k_pool[0, page] = grow / 128.0 * np.sqrt(128.0)
    x.v_pool.mul_(1e25); x.v_new.mul_(1e25)
    out, lse = run_gpu(make_mirror(cfg), x)
    o_ref, lse_ref = oracle_attention(x)[0]
    assert torch.isfinite(out.float()).all()
    # bf16 weights (equal ones here: 2^-9 of their sum at most) and bf16 outputs
    assert np.abs(out[0].float().cpu().numpy() - o_ref).max() <= 1e-2 * np.abs(o_ref).max()
    assert np.abs(lse[0].cpu().numpy() - lse_ref).max() <= 2e-3


@pytest.mark.parametrize("hq,hkv,d,prefix", [
    (8, 1, 128, 40000),       # 148 parts, one row tile
    (8, 1, 64, 20000),        # 79 parts
    (32, 1, 128, 40000),      # 74 parts, four row tiles
    (20, 4, 128, 33000),      # four units of 37 parts
    (4, 4, 128, 17000),       # four units of 37 parts, few rows
])
def test_units_that_many_groups_share(hq, hkv, d, prefix):
    """More parts per unit than the merge has room for at a time: it takes them in batches."""
    cfg = config(hq, hkv, d, 3, 4, prefix, prefix, batch=1)
    x = I.gen_verify_inputs(cfg, 13, "cuda", with_lm_head=False)
    m = make_mirror(cfg)
    out, lse = run_gpu(m, x)
    compare(out, lse, oracle_attention(x), range(cfg.layers))
    for _ in range(20):
        again, lse2 = run_gpu(m, x)
        assert torch.equal(again, out) and torch.equal(lse2, lse)


@pytest.mark.parametrize("hq,hkv", [(8, 1), (32, 1), (20, 4)])
def test_units_that_many_groups_share_over_an_8_bit_cache(hq, hkv):
    run_and_compare(small(n_q_heads=hq, n_kv_heads=hkv, prefix_lo=33000, prefix_hi=33000, batch=1, layers=1), 14)


@pytest.mark.parametrize("hq,hkv,d,kappa,gamma,layers,batch,lo,hi", [
    (64, 8, 128, 8, 7, 8, 1, 1000, 1000),        # 64 units for 74 groups: one each, nothing to merge
    (64, 8, 128, 8, 7, 4, 2, 1000, 1000),        # the same, with the merge launched in vain
    (64, 8, 128, 8, 15, 2, 1, 1000, 1000),       # 16 units for 37 groups: two each
    (16, 2, 64, 4, 8, 1, 1, 900, 900),           # 2 units for 148 groups: as many as the units have tiles for
    (64, 8, 128, 8, 7, 4, 2, 990, 1130),         # units of two lengths: an even split
    (64, 8, 128, 8, 7, 2, 1, 9000, 9000),        # long units: an even split
    (16, 1, 128, 3, 4, 1, 1, 0, 0),              # one unit
])
def test_fewer_units_than_groups(hq, hkv, d, kappa, gamma, layers, batch, lo, hi):
    cfg = config(hq, hkv, d, kappa, gamma, lo, hi, batch=batch, layers=layers)
    x = I.gen_verify_inputs(cfg, 15, "cuda", with_lm_head=False)
    out, lse = run_gpu(make_mirror(cfg), x)
    which = sorted({0, layers - 1})
    ref = oracle_attention(x, which)
    compare(out, lse, ref, which)
    x.page_table = torch.cat([x.page_table, x.page_table.new_full((batch, 2000), -1)], 1).contiguous()      # room for longer contexts
    out, lse = run_gpu(make_mirror(cfg), x)
    compare(out, lse, ref, which)


@pytest.mark.parametrize("kw", [dict(kappa=8, gamma=7, layers=4, batch=2), dict(kappa=8, gamma=15, layers=2, batch=1), dict(kappa=4, gamma=4, layers=1, batch=1)])
def test_fewer_units_than_groups_over_an_8_bit_cache(kw):
    run_and_compare(small(n_q_heads=64, n_kv_heads=8, hidden=8192, prefix_lo=1000, prefix_hi=1000, **kw), 16)
