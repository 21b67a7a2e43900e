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


@pytest.mark.parametrize("V,B", [(70001, 1), (70001, 4), (40000, 9)])       # 16 and 8 CTAs per request
def test_walk_that_rejects_accepts_and_rejects_again(V, B):
    """A sibling is rejected (the residual goes to scratch memory), the next one passes the test against that residual, and its
    child is rejected: the child's residual must not land where a slower CTA of the cluster still reads the sibling's test."""
    kappa, gamma = 3, 3
    m = make_mirror(cfg_for(V, kappa, gamma, B))
    par = I.comb_parent(kappa, gamma)
    logits, qp, tok, ua, ur = spec_case(B, kappa, gamma, V, 3 * V + B)
    first = lambda k: 1 + k * gamma                             # noqa: E731  (root's k-th child)
    for b in range(B):
        for c, u in ((first(0), 1.0), (first(1), 0.0), (first(1) + 1, 1.0)):
            ua[b, c] = u
            if u == 1.0:                                        # q far above p at the token: rejected
                qp[b, c - 1] *= 0.5
                qp[b, c - 1, tok[b, c]] += 0.5
    lse = torch.logsumexp(logits.double(), -1).float()
    ref = O.accept_tree(tok.numpy(), logits.numpy(), lse.numpy(), qp.numpy(), ua.numpy(), ur.numpy(), par, gamma, True, 1.0)
    assert (ref["n_accepted"] == 1).all() and (ref["accepted_nodes"][:, 0] == first(1)).all()
    acc = m.accept_in(binding.ACCEPT_SPEC_TREE, True, logits=logits.cuda(), lse=lse.cuda(), q_probs=qp.cuda(), u_accept=ua.cuda(),
                      u_resample=ur.cuda())
    tree = m.tree(tok.cuda(), kappa, gamma)
    first_run = None
    for _ in range(100):
        got = m.mirror_accept_select(tree, acc, tree_scratch=True).cpu()
        first_run = first_run or got
        for f in FIELDS:
            assert np.array_equal(got[f], first_run[f]), f
    assert m.device_status() == (0, 0)
    for b in range(B):
        same = all(np.array_equal(first_run[f][b], ref[f][b]) for f in FIELDS if f != "reuse_slot")
        assert same or ref["margin"][b] < 1e-9, (b, ref["margin"][b])


@pytest.mark.parametrize("scratch", [False, True])
def test_tree_rule_reports_tokens_outside_the_vocabulary_where_the_walk_meets_them(scratch):
    """A node that the walk never comes to may hold anything (a padded tree); one that it comes to is rejected and reported."""
    V, kappa, gamma, B = 9000, 3, 2, 2
    m = make_mirror(cfg_for(V, kappa, gamma, B))
    logits, qp, tok, ua, ur = spec_case(B, kappa, gamma, V, 17)
    ua[:, 1] = ua[:, 2] = 0.0                                   # the first branch is accepted to its end
    lse = torch.logsumexp(logits.double(), -1).float()
    acc = m.accept_in(binding.ACCEPT_SPEC_TREE, True, logits=logits.cuda(), lse=lse.cuda(), q_probs=qp.cuda(), u_accept=ua.cuda(),
                      u_resample=ur.cuda())
    run = lambda t: m.mirror_accept_select(m.tree(t.cuda(), kappa, gamma), acc, tree_scratch=scratch).cpu()      # noqa: E731
    ref = run(tok)
    assert m.device_status() == (0, 0) and (ref["n_accepted"] == gamma).all()
    padded = tok.clone()
    padded[:, 1 + gamma:] = -1                                  # the other branches
    got = run(padded)
    assert m.device_status() == (0, 0)
    for f in FIELDS:
        assert np.array_equal(got[f], ref[f]), f
    met = tok.clone()
    met[1, 1] = V                                               # the first test of the second request
    got = run(met)
    assert m.device_status() == (6, 101)
    assert got["n_accepted"][0] == gamma and 1 not in got["accepted_nodes"][1]


@pytest.mark.parametrize("V,B", [(1000, 2), (1025, 2), (2049, 1), (4096, 3), (4097, 1), (4097, 6), (20000, 4), (33000, 5)])
@pytest.mark.parametrize("kappa", [3, 4, 9])                    # siblings under the root: few, and enough for a thread per id
@pytest.mark.parametrize("reject", [False, True])               # every sibling rejected, or as it comes
def test_walks_over_many_siblings(V, B, kappa, reject):
    gamma = 2
    m = make_mirror(cfg_for(V, kappa, gamma, B))
    par = I.comb_parent(kappa, gamma)
    logits, qp, tok, ua, ur = spec_case(B, kappa, gamma, V, V + kappa)
    if reject:
        for b in range(B):
            for k in range(kappa):
                c = 1 + k * gamma
                ua[b, c] = 1.0
                qp[b, c - 1] *= 0.5
                qp[b, c - 1, tok[b, c]] += 0.5
    lse = torch.logsumexp(logits.double(), -1).float()
    ref = O.accept_tree(tok.numpy(), logits.numpy(), lse.numpy(), qp.numpy(), ua.numpy(), ur.numpy(), par, gamma, True, 1.0)
    acc = m.accept_in(binding.ACCEPT_SPEC_TREE, True, logits=logits.cuda(), lse=lse.cuda(), q_probs=qp.cuda(), u_accept=ua.cuda(),
                      u_resample=ur.cuda())
    tree = m.tree(tok.cuda(), kappa, gamma)
    for scratch in (False, True):
        got = m.mirror_accept_select(tree, acc, tree_scratch=scratch).cpu()
        assert m.device_status() == (0, 0)
        for b in range(B):
            same = all(np.array_equal(got[f][b], ref[f][b]) for f in FIELDS if f != "reuse_slot")
            assert same or ref["margin"][b] < 1e-9, (b, scratch, ref["margin"][b])
