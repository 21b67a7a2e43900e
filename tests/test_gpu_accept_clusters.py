"""GPU parity of the draws at the edges of the vocabulary's split: a cluster of 2, 4, 8 or 16 CTAs per request, chunks that
hold nothing, ragged ends, and uniforms at both ends of the cumulative sum."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2510_13161_b200 import binding, inputs as I
from tests.helpers import make_mirror
from tests.test_gpu_accept import FIELDS, cfg_for, spec_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["chain", "tree"])
@pytest.mark.parametrize("V,B", [(2, 3), (33, 2), (8192, 1), (8193, 2), (32768, 1), (32769, 2), (65537, 1), (65537, 5)])
def test_draws_at_the_edges_of_the_split(mode, V, B):
    kappa, gamma = 2, 2
    m = make_mirror(cfg_for(V, kappa, gamma, B))
    par = I.comb_parent(kappa, gamma)
    logits, qp, tok, ua, ur = spec_case(B, kappa, gamma, V, V + B)
    logits.view(B, -1, V)[0, :, : V // 2] = -1e4               # half of the chunks without mass
    lse = torch.logsumexp(logits.double(), -1).float()
    for u in (0.0, float(np.nextafter(np.float32(1), np.float32(0)))):
        ur[:] = u
        ref = (O.accept_spec if mode == "chain" else O.accept_tree)(
            tok.numpy(), logits.numpy(), lse.numpy(), qp.numpy(), ua.numpy(), ur.numpy(), par, gamma, True, 1.0)
        acc = m.accept_in(1 if mode == "chain" else binding.ACCEPT_SPEC_TREE, True, logits=logits.cuda(), lse=lse.cuda(),
                          q_probs=qp.cuda(), u_accept=ua.cuda(), u_resample=ur.cuda())
        tree = m.tree(tok.cuda(), kappa, gamma)
        for scratch in ((False, True) if mode == "tree" else (False,)):
            got = m.mirror_accept_select(tree, acc, tree_scratch=scratch).cpu()
            assert m.device_status() == (0, 0)
            for b in range(B):
                # (as in test_gpu_accept: fp64 sums in another order may differ on a knife edge only)
                same = all(np.array_equal(got[f][b], ref[f][b]) for f in FIELDS if f != "reuse_slot")
                assert same or ref["margin"][b] < 1e-9, (b, u, ref["margin"][b], {f: (got[f][b], ref[f][b]) for f in FIELDS})
