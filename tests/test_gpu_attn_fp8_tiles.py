"""GPU parity of the 8-bit cache's attention kernel at the edges of its tiles: one, two, three and more tiles of 128 rows per
KV head, units shorter than the tiles over which the next unit's Q is staged, ragged pages in every place of a tile, and
scales of Q beyond those that the reciprocal serves."""
import pytest

from tests.test_gpu_attn_fp8 import run_and_compare, small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,kappa,gamma", [
    (2, 2, 1, 1),             # 2 rows
    (8, 2, 31, 1),            # 128 rows: one full tile
    (8, 2, 4, 8),             # 132 rows: two tiles
    (16, 2, 4, 8),            # 264 rows: three tiles, two heads per unit
    (24, 3, 8, 5),            # 328 rows: three tiles, an odd number of heads
    (71, 1, 2, 2),            # G = 71: a share of the heads per tile
])
@pytest.mark.parametrize("lo,hi,batch,layers", [(1, 90, 5, 5), (100, 2500, 2, 1)])      # many short units per CTA, and cut ones
def test_row_tiles(hq, hkv, kappa, gamma, lo, hi, batch, layers):
    run_and_compare(small(n_q_heads=hq, n_kv_heads=hkv, kappa=kappa, gamma=gamma, prefix_lo=lo, prefix_hi=hi, batch=batch, layers=layers), 7)


@pytest.mark.parametrize("prefix", [1, 15, 16, 111, 113, 127, 128, 129, 255])
@pytest.mark.parametrize("hq", [4, 32])
def test_key_tiles(prefix, hq):
    run_and_compare(small(n_q_heads=hq, prefix_lo=prefix, prefix_hi=prefix, batch=1), prefix)


@pytest.mark.parametrize("scale", [2.0 ** -70, 2.0 ** 70])
def test_unusual_query_scales(scale):
    def tweak(x):
        x.q.mul_(scale)
        if scale > 1:                                # (scores that fp32 can hold)
            x.k_pool.mul_(1 / scale)
            x.k_new.mul_(1 / scale)
    run_and_compare(small(n_q_heads=16, kappa=4, gamma=4, layers=1), 11, tweak=tweak)
