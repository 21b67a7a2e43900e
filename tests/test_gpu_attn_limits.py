"""Attention at the ends of what it accepts."""
import pytest
import torch

from paper_2510_13161_b200 import inputs as I
from tests.helpers import make_mirror, oracle_attention
from tests.test_gpu_attn import compare, run_gpu
from tests.test_gpu_attn_tiles import config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,kappa,gamma", [(2 * 353, 5, 10), (2 * 353, 4, 13), (2 * 149, 9, 14)])       # 153, 159 and 156 row tiles of whole nodes
def test_more_row_tiles_than_sms(hq, kappa, gamma):
    cfg = config(hq, 2, 64, kappa, gamma, 20, 40, batch=1)
    x = I.gen_verify_inputs(cfg, 3, "cuda", with_lm_head=False)
    out, lse = run_gpu(make_mirror(cfg), x)
    compare(out, lse, oracle_attention(x), range(cfg.layers))
