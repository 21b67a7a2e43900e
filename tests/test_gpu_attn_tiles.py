"""GPU parity of the attention kernel at the edges of its row and key tiles: one, two, three and more tiles of 128 rows per
KV head (streams on alternate key tiles, sharing key tiles, or of two heads), groups of query heads that do not divide a
tile, prefixes around multiples of 16 and 128, and rows whose scores outgrow the offset that their first tile set."""
import numpy as np
import pytest
import torch

from paper_2510_13161_b200 import inputs as I
from tests.helpers import make_mirror
from tests.test_gpu_attn import compare, oracle_attention, run_gpu

pytestmark = pytest.mark.gpu


def config(hq, hkv, d, kappa, gamma, lo, hi, batch=2, layers=1):
    return I.VerifyConfig("t", 1024, hq, hkv, d, layers, batch, lo, hi, kappa, gamma, 64, "greedy", 0.02, 1.0)


@pytest.mark.parametrize("hq,hkv,d,kappa,gamma", [
    (8, 2, 128, 1, 1),        # 8 rows: one tile
    (8, 2, 128, 31, 1),       # 128 rows: one full tile
    (8, 2, 64, 4, 8),         # 132 rows: two tiles
    (16, 2, 128, 4, 8),       # 264 rows: three tiles, two heads
    (24, 3, 128, 8, 5),       # 328 rows: three tiles, an odd number of heads
    (16, 2, 64, 8, 8),        # 520 rows: five tiles
    (5, 1, 128, 8, 7),        # G = 5: tiles of whole nodes
    (71, 1, 64, 2, 2),        # G = 71: a share of the heads per tile
    (160, 1, 128, 1, 2),      # G = 160: more heads than a tile has rows
])
@pytest.mark.parametrize("hi", [700, 2500])          # units dealt out whole, and cut
def test_row_tiles(hq, hkv, d, kappa, gamma, hi):
    cfg = config(hq, hkv, d, kappa, gamma, 100, hi)
    x = I.gen_verify_inputs(cfg, 3, "cuda", with_lm_head=False)
    out, lse = run_gpu(make_mirror(cfg), x)
    compare(out, lse, oracle_attention(x), range(cfg.layers))


@pytest.mark.parametrize("prefix", [0, 1, 15, 16, 17, 111, 112, 113, 127, 128, 129, 255, 1024 - 9])
@pytest.mark.parametrize("hq", [4, 32])
def test_key_tiles(prefix, hq):
    cfg = config(hq, 2, 128, 2, 4, prefix, prefix, batch=1)
    x = I.gen_verify_inputs(cfg, prefix, "cuda", with_lm_head=False)
    out, lse = run_gpu(make_mirror(cfg), x)
    compare(out, lse, oracle_attention(x), range(cfg.layers))


@pytest.mark.parametrize("hq", [4, 32])
@pytest.mark.parametrize("at", [0, 3, 7, 12, 20])
def test_scores_that_outgrow_the_offset(at, hq):
    """Keys of one page (first or second half of a tile, first or later tile) 120 times the others' size: the row's offset has
    to move there, by far more than 2^80, or to stay and carry everything behind it."""
    cfg = config(hq, 2, 128, 2, 4, 400, 400, batch=1)
    x = I.gen_verify_inputs(cfg, 5, "cuda", with_lm_head=False, shuffle_pages=False)
    page = int(x.page_table[0, at])
    x.k_pool[0, page] *= 120.0
    out, lse = run_gpu(make_mirror(cfg), x)
    ref = oracle_attention(x)
    o_ref, lse_ref = ref[0]
    # A score of size s is off by about |s| 2^-23 after fp32 accumulation, which moves its weight by that much relatively:
    # 1000 x 2^-23 = 1.2e-4, on top of bf16 weights and outputs (2^-8 of the largest output together).
    err = np.abs(out[0].float().cpu().numpy() - o_ref).max()
    assert err <= 1e-2 * np.abs(o_ref).max() + 1e-5, err
    assert np.abs(lse[0].cpu().numpy() - lse_ref).max() <= 2e-3 + 1e-6 * np.abs(lse_ref).max()
    assert torch.isfinite(out.float()).all()
