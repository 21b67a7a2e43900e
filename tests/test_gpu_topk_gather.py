"""The merge of the Top-kappa lists: pairs that reach the row's bar are gathered and ranked by counting, rounds over the lists
take over when too many do.  Identical weight rows give identical logits, so copies decide which way a row goes."""
import pytest
import torch

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
