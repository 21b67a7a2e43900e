"""GPU parity of the attention kernel that mirror_target_forward uses in stacks of more than four layers (64-token key tiles): each
layer's attention output against the fp64 oracle on that layer's own queries, keys and values, so that nothing is inherited from
the layers before."""
import types

import numpy as np
import pytest
import torch

from paper_2510_13161_b200 import inputs as I
from tests.helpers import make_mirror, oracle_attention
from tests.test_gpu_layer import layer_case
from tests.test_gpu_timeout import stalled_mirror

pytestmark = pytest.mark.gpu
DEEP = 5                                    # layers: one more than the stacks of the other kernel


def setup(m, cfg, x, layers, norm_final, inter):
    dev = lambda t: t.cuda()                # noqa: E731
    kv = m.kv(dev(x.k_pool), dev(x.v_pool), dev(x.page_table), dev(x.prefix_len))
    return m.target([{k: dev(v) for k, v in w.items()} for w in layers], dev(norm_final), inter, 1.0e4, 1e-6), kv, m.tree(
        dev(x.tokens), cfg.kappa, cfg.gamma, parent=x.parent)


def check_attention(out, cfg, x, which=None):
    y = types.SimpleNamespace(cfg=cfg, parent=x.parent, q=out["q"], k_pool=x.k_pool, v_pool=x.v_pool, page_table=x.page_table,
                              prefix_len=x.prefix_len, k_new=out["k_new"], v_new=out["v_new"])
    for l, (ref, _) in oracle_attention(y, layers=which).items():
        err = np.abs(out["attn_out"][l].float().cpu().numpy() - ref).max()
        assert err <= 1e-2 * np.abs(ref).max() + 1e-5, (l, err, np.abs(ref).max())        # (bf16 weights and outputs: the gate of the attention tests)


def run(case, which=None, repeat=3):
    cfg, x, layers, norm_final, emb = layer_case(**case)
    m = make_mirror(cfg)
    target, kv, tree = setup(m, cfg, x, layers, norm_final, case["inter"])
    emb = emb.cuda()
    out = {k: v.clone() for k, v in m.mirror_target_forward(target, kv, tree, emb).items() if not k.startswith("_")}
    assert m.device_status() == (0, 0)
    check_attention(out, cfg, x, which)
    for _ in range(repeat):
        again = m.mirror_target_forward(target, kv, tree, emb)
        for k, v in out.items():
            assert torch.equal(again[k], v), k
    assert m.device_status() == (0, 0)


@pytest.mark.parametrize("Hq,Hkv,d,kappa,gamma", [
    (4, 2, 64, 3, 4),          # 26 rows per KV head
    (8, 2, 128, 31, 1),        # 128 rows
    (8, 2, 64, 4, 8),          # 132 rows: two row blocks
    (16, 2, 128, 4, 8),        # 264 rows: three
    (5, 1, 128, 8, 7),         # G = 5
])
@pytest.mark.parametrize("lo,hi,B", [(1, 300, 3), (900, 2500, 2)])        # short ragged requests, and units cut across CTAs
def test_row_blocks(Hq, Hkv, d, kappa, gamma, lo, hi, B):
    run(dict(H=256, Hq=Hq, Hkv=Hkv, d=d, inter=256, L=DEEP, B=B, lo=lo, hi=hi, kappa=kappa, gamma=gamma, seed=21))


@pytest.mark.parametrize("prefix", [0, 1, 15, 16, 17, 63, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("d", [64, 128])
def test_key_tiles(prefix, d):
    run(dict(H=256, Hq=4, Hkv=2, d=d, inter=256, L=DEEP, B=1, lo=prefix, hi=prefix, kappa=2, gamma=4, seed=22), repeat=1)


def test_general_tree():
    run(dict(H=256, Hq=4, Hkv=2, d=64, inter=256, L=DEEP, B=2, lo=40, hi=200, kappa=1, gamma=6, seed=23, parent=I.random_tree_parent(24, 5, max_depth=6)))


@pytest.mark.parametrize("Hkv,prefix", [(4, 33000), (1, 12000)])          # 37 and 148 parts per unit
def test_units_that_many_ctas_share(Hkv, prefix):
    run(dict(H=256, Hq=4 * Hkv, Hkv=Hkv, d=128, inter=256, L=DEEP, B=1, lo=prefix, hi=prefix, kappa=3, gamma=4, seed=24), which=[0, DEEP - 1], repeat=10)


def test_a_wait_that_runs_out(monkeypatch):
    case = dict(H=256, Hq=4, Hkv=2, d=64, inter=256, L=DEEP, B=2, lo=500, hi=700, kappa=3, gamma=4, seed=25)
    cfg, x, layers, norm_final, emb = layer_case(**case)
    m = stalled_mirror(cfg, monkeypatch)    # the first layer's K producer stops after one stage
    target, kv, tree = setup(m, cfg, x, layers, norm_final, case["inter"])
    m.mirror_target_forward(target, kv, tree, emb.cuda())
    code, detail = m.device_status()
    assert code == 7 and detail in (10, 20, 21, 23, 24, 30, 31, 32, 33, 34, 35, 36), (code, detail)
    out = m.mirror_target_forward(target, kv, tree, emb.cuda())
    assert m.device_status() == (0, 0)
    check_attention(out, cfg, x)
