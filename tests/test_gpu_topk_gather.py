"""The merge of the Top-kappa lists: pairs that reach the row's bar are gathered and ranked by counting, rounds over the lists
take over when too many do.  Identical weight rows give identical logits, so copies decide which way a row goes."""
import pytest
import torch

from paper_2510_13161_b200 import binding
from tests.helpers import make_mirror
from tests.test_gpu_topk_fused import lm_cfg, rand_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 8, 32])
@pytest.mark.parametrize("every", [1, 3, 40, 1000])                        # all ids equal, and fewer and fewer copies
def test_equal_logits_go_to_the_lowest_ids(k, every):
    V, H, M = 40000, 256, 5
    W = rand_bf16((V, H), 0.05, 5); hid = rand_bf16((M, H), 1.0, 6)
    W[every // 2::every] = (hid[0].float() * 0.2).to(torch.bfloat16)       # the best ids of row 0, all with the same logit
    m = make_mirror(lm_cfg(V, H))
    for _ in range(2):                                                     # (the second call finds the bars cleared)
        res = m.mirror_lmhead_reduce(hid.cuda(), W.cuda(), topk=k)
        assert res["topk_id"][0].cpu().tolist() == list(range(every // 2, V, every))[:k]
        lp = res["topk_logprob"][0].cpu()
        assert (lp == lp[0]).all()


@pytest.mark.parametrize("M,V,k", [(17, 500, 4), (57, 9000, 8), (57, 16000, 8), (40, 1024, 32), (64, 2000, 1)])
def test_small_vocabularies_select_from_spilled_logits_where_there_is_room(M, V, k):
    """The same pairs and log-probabilities whichever way a call goes; a workspace sized for the candidate lists alone stays enough."""
    H = 256
    W = rand_bf16((V, H), 0.05, 7); hid = rand_bf16((M, H), 1.0, 8)
    W[V // 2] = W[3]; W[V - 1] = W[3]                                      # ties
    W, hid = W.cuda(), hid.cuda()
    roomy, tight = make_mirror(lm_cfg(V, H)), make_mirror(lm_cfg(V, H))
    t = binding.Tree(1, M, 0, 0, None, None); t.batch, t.n_nodes = 1, M
    tight._need[(binding.WS_LMHEAD_TOPK, 1, M)] = tight.workspace_bytes(t, None, binding.WS_LMHEAD)      # (the lists lie in the attention's region)
    assert roomy.workspace_bytes(t, None, binding.WS_LMHEAD_TOPK) > tight._need[(binding.WS_LMHEAD_TOPK, 1, M)]
    a, b = roomy.mirror_lmhead_reduce(hid, W, topk=k), tight.mirror_lmhead_reduce(hid, W, topk=k)
    assert roomy.device_status() == (0, 0) and tight.device_status() == (0, 0)
    for f in ("topk_id", "topk_logprob", "argmax", "lse"):
        assert torch.equal(a[f], b[f]), f
    (ids, lp), (ids2, lp2) = roomy.mirror_early_exit_tap(hid, W, k), tight.mirror_early_exit_tap(hid, W, k)
    assert torch.equal(ids, ids2) and torch.equal(lp, lp2) and torch.equal(ids, a["topk_id"])
