"""The step with hidden rows of the caller's own: the LM head runs beside the attention, which leaves it SMs where both are long."""
import numpy as np
import pytest
import torch

from paper_2510_13161_b200 import binding, inputs as I
from tests.helpers import make_mirror

pytestmark = pytest.mark.gpu
FIELDS = ["n_accepted", "best_branch", "decide_row", "n_emitted", "emitted", "accepted_nodes", "reuse_slot"]
_MODES = {"greedy": binding.ACCEPT_GREEDY, "spec_sampling": binding.ACCEPT_SPEC_SAMPLING, "spec_tree": binding.ACCEPT_SPEC_TREE}


def parts(m, kv, tree, x, mode):
    """The same step as separate calls: each waits for the one before."""
    attn = m.mirror_attn_verify(kv, tree, x.q, x.k_new, x.v_new)
    lm = m.mirror_lmhead_reduce(x.hidden, x.W, want_logits=mode != "greedy")
    kw = dict(target_argmax=lm["argmax"]) if mode == "greedy" else dict(logits=lm["logits"], lse=lm["lse"], q_probs=x.q_probs, u_accept=x.u_accept, u_resample=x.u_resample)
    res = m.mirror_accept_select(tree, m.accept_in(_MODES[mode], True, **kw))
    return attn, lm, res.cpu()


# layers, batch, prefixes, kappa, gamma, query heads of 8 KV heads, mode: row tiles of either kind and number, whole and cut units,
# up to 128 rows (a weight stream, beside which the attention takes fewer groups), one row chunk, several
@pytest.mark.parametrize("L,B,lo,hi,kappa,gamma,hq,mode", [
    (12, 1, 1000, 1000, 8, 7, 40, "spec_tree"),            # three row tiles of 95: units of two heads
    (12, 1, 1000, 1000, 8, 6, 40, "greedy"),               # two
    (40, 1, 700, 700, 4, 4, 40, "greedy"),                 # one; many units, dealt out whole
    (6, 2, 300, 3000, 8, 7, 64, "spec_sampling"),          # four, ragged, cut
    (60, 3, 17, 90, 4, 4, 40, "greedy"),                   # short units
    (3, 4, 64, 900, 8, 7, 40, "spec_sampling"),            # 228 rows
    (2, 5, 64, 300, 8, 8, 64, "greedy"),                   # 325 rows: two row chunks
    (1, 1, 1, 1, 1, 1, 16, "spec_tree"),
])
def test_step_beside_equals_its_parts(L, B, lo, hi, kappa, gamma, hq, mode):
    cfg = I.VerifyConfig("b", 2048, hq, 8, 128, L, B, lo, hi, kappa, gamma, 64000, mode, explicit_hidden=True)
    x = I.gen_verify_inputs(cfg, 5, "cuda", force_hidden=True)
    m = make_mirror(cfg)
    kv, tree = m.kv(x.k_pool, x.v_pool, x.page_table, x.prefix_len), m.tree(x.tokens, kappa, gamma)
    ref_attn, lm, ref = parts(m, kv, tree, x, mode)
    acc = m.accept_in(_MODES[mode], True, q_probs=x.q_probs, u_accept=x.u_accept, u_resample=x.u_resample)
    first = None
    for _ in range(3):                                     # (the unit counter is left as it was found)
        attn, argmax = torch.full_like(x.q, float("nan")), torch.full((cfg.rows,), -1, dtype=torch.int32, device="cuda")
        got = m.mirror_verify_step(kv, tree, x.q, x.k_new, x.v_new, x.hidden, x.W, acc, attn, argmax_out=argmax).cpu()
        assert m.device_status() == (0, 0)
        assert torch.equal(argmax, lm["argmax"])           # (exact ties aside, which these inputs do not have)
        # another cut of the keys: the same bound as against the oracle (bf16 output and weights)
        assert (attn.float() - ref_attn.float()).abs().max() <= 1e-2 * ref_attn.float().abs().max() + 1e-5
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], ref[f], err_msg=f)
        if first is not None:
            assert torch.equal(attn, first)                # (the cut does not depend on timing)
        first = attn


def test_hidden_rows_that_are_the_attention_output_wait_for_it():
    cfg = I.VerifyConfig("a", 2048, 16, 8, 128, 6, 1, 900, 900, 4, 4, 64000, "greedy")
    x = I.gen_verify_inputs(cfg, 3, "cuda")
    m = make_mirror(cfg)
    kv, tree, acc = m.kv(x.k_pool, x.v_pool, x.page_table, x.prefix_len), m.tree(x.tokens, 4, 4), m.accept_in(binding.ACCEPT_GREEDY, True)
    argmax = torch.empty((2, cfg.rows), dtype=torch.int32, device="cuda")
    attn = torch.empty_like(x.q)
    m.mirror_verify_step(kv, tree, x.q, x.k_new, x.v_new, None, x.W, acc, attn, argmax_out=argmax[0])
    attn.zero_()
    m.mirror_verify_step(kv, tree, x.q, x.k_new, x.v_new, attn[-1].reshape(cfg.rows, cfg.hidden), x.W, acc, attn, argmax_out=argmax[1])
    torch.cuda.synchronize()
    assert torch.equal(argmax[0], argmax[1])


@pytest.mark.parametrize("own_rows", [True, False])
def test_weights_that_are_the_attention_output_wait_for_it(own_rows):
    """... whether the hidden rows are the caller's (LM head beside the attention) or the attention's (its weights requested early)."""
    V = 64
    cfg = I.VerifyConfig("w", 2048, 16, 8, 128, 6, 1, 900, 900, 4, 4, V, "greedy", explicit_hidden=own_rows)
    x = I.gen_verify_inputs(cfg, 3, "cuda", force_hidden=own_rows)
    m = make_mirror(cfg)
    kv, tree, acc = m.kv(x.k_pool, x.v_pool, x.page_table, x.prefix_len), m.tree(x.tokens, 4, 4), m.accept_in(binding.ACCEPT_GREEDY, True)
    ref = m.mirror_attn_verify(kv, tree, x.q, x.k_new, x.v_new)
    rows = x.hidden if own_rows else ref[-1].reshape(cfg.rows, cfg.hidden)
    want = m.mirror_lmhead_reduce(rows, ref.reshape(-1, cfg.hidden)[:V])["argmax"]
    attn, argmax = torch.empty_like(x.q), torch.empty(cfg.rows, dtype=torch.int32, device="cuda")
    for seed in range(3):
        attn.normal_()                                     # (weights read too early would be these)
        m.mirror_verify_step(kv, tree, x.q, x.k_new, x.v_new, x.hidden if own_rows else None, attn.reshape(-1, cfg.hidden)[:V], acc, attn, argmax_out=argmax)
        assert m.device_status() == (0, 0)
        assert torch.equal(attn, ref) and torch.equal(argmax, want)
