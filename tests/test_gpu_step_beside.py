"""The step with hidden rows of the caller's own: the LM head runs beside the attention, which leaves it SMs where both are long."""
import ctypes as C
import time

import numpy as np
import pytest
import torch

from paper_2510_13161_b200 import binding, inputs as I
from tests.helpers import make_mirror
from tests.test_gpu_attn_fp8 import quantise

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


class KernelNode(C.Structure):
    _fields_ = [("func", C.c_void_p), ("dims", C.c_uint * 7), ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def kernels(call):
    """What a call launches, out of a captured graph: {kernel: (blocks in a cluster, blocks)}, in the order of the launches."""
    call()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    cu, raw, n, got = C.CDLL("libcuda.so.1"), C.c_void_p(g.raw_cuda_graph()), C.c_size_t(), {}
    assert cu.cuGraphGetNodes(raw, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(raw, nodes, C.byref(n)) == 0
    for node in map(C.c_void_p, nodes):
        kind, p, name, attr = C.c_int(), KernelNode(), C.c_char_p(), (C.c_uint * 16)()
        assert cu.cuGraphNodeGetType(node, C.byref(kind)) == 0
        if kind.value == 0:                                # a kernel
            assert cu.cuGraphKernelNodeGetParams_v2(node, C.byref(p)) == 0
            assert (cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)) if p.func else cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern))) == 0
            assert cu.cuGraphKernelNodeGetAttribute(node, 4, C.byref(attr)) == 0           # (4: the cluster's dimensions)
            for k in ("attn_verify_kernel", "attn_merge_kernel", "lmhead_pair_free_kernel", "lmhead_merge_kernel", "accept_"):
                if k in name.value.decode():
                    got[k] = (max(1, attr[0]), p.dims[0])
    return got


class Case:
    """One problem on a context of its own, over a bf16 or an 8-bit cache."""

    def __init__(self, L, B, lo, hi, kappa, gamma, hq, mode, hidden=2048, vocab=64000, seed=5, fp8=False, headroom=0):
        cfg = self.cfg = I.VerifyConfig("b", hidden, hq, 8, 128, L, B, lo, hi, kappa, gamma, vocab, mode, explicit_hidden=True)
        x = self.x = I.gen_verify_inputs(cfg, seed, "cuda", force_hidden=True, headroom=headroom)
        m = self.m = make_mirror(cfg)
        self.tree = m.tree(x.tokens, kappa, gamma)
        self.acc = m.accept_in(_MODES[mode], True, q_probs=x.q_probs, u_accept=x.u_accept, u_resample=x.u_resample)
        self.fp8 = fp8
        if fp8:
            self.ks, self.vs, k8, v8, self.kn, self.vn = quantise(m, x)
            self.kv, self.q_scale = m.kv_fp8(k8, v8, x.page_table, x.prefix_len), float(np.float32(float(x.q.float().abs().max())) / np.float32(448.0))
        else:
            self.kv, self.kn, self.vn = m.kv(x.k_pool, x.v_pool, x.page_table, x.prefix_len), x.k_new, x.v_new
        self.attn, self.argmax = torch.empty_like(x.q), torch.empty(cfg.rows, dtype=torch.int32, device="cuda")
        self.out = binding.AcceptResult(B, gamma, "cuda")

    def step(self):
        m, x = self.m, self.x
        if self.fp8:
            m.mirror_verify_step_fp8(self.kv, self.tree, x.q, self.kn, self.vn, self.ks, self.vs, self.q_scale, x.hidden, x.W, self.acc, self.attn,
                                     out=self.out, argmax_out=self.argmax)
        else:
            m.mirror_verify_step(self.kv, self.tree, x.q, self.kn, self.vn, x.hidden, x.W, self.acc, self.attn, out=self.out, argmax_out=self.argmax)

    def parts(self):
        m, x, mode = self.m, self.x, self.cfg.mode
        if self.fp8:
            attn = m.mirror_attn_verify_fp8(self.kv, self.tree, x.q, self.kn, self.vn, self.ks, self.vs, self.q_scale)
        else:
            attn = m.mirror_attn_verify(self.kv, self.tree, x.q, self.kn, self.vn)
        lm = m.mirror_lmhead_reduce(x.hidden, x.W, want_logits=mode != "greedy")
        kw = dict(target_argmax=lm["argmax"]) if mode == "greedy" else dict(logits=lm["logits"], lse=lm["lse"], q_probs=x.q_probs, u_accept=x.u_accept, u_resample=x.u_resample)
        return attn, lm["argmax"], m.mirror_accept_select(self.tree, m.accept_in(_MODES[mode], True, **kw))

    def check(self, ref):
        assert self.m.device_status() == (0, 0)
        assert torch.equal(self.argmax, ref[1])
        # another cut of the keys: twice the bound against the oracle, which either has to keep
        assert (self.attn.float() - ref[0].float()).abs().max() <= 2e-2 * ref[0].float().abs().max() + 1e-5
        got, want = self.out.cpu(), ref[2].cpu()
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], want[f], err_msg=f)


# What the rules of a launch behind the attention can come to, named by the kernels that it takes.  A: the attention, in pairs of
# blocks where it may leave SMs to the LM head (A2); F: the LM head beside it; R: its row merge; M: the attention's merge; D: decision.
_NAMES = {"attn_verify_kernel": "A", "lmhead_pair_free_kernel": "F", "lmhead_merge_kernel": "R", "attn_merge_kernel": "M", "accept_": "D"}


@pytest.mark.parametrize("way,case", [
    ("A2FRMD", dict(L=6, B=2, lo=300, hi=3000, kappa=8, gamma=7, hq=64, mode="spec_sampling", fp8=True)),        # 114 rows, cut, over codes
    ("A2FDM", dict(L=6, B=2, lo=300, hi=3000, kappa=8, gamma=7, hq=64, mode="greedy", fp8=True)),
    ("A2FRMD", dict(L=12, B=1, lo=1000, hi=1000, kappa=8, gamma=7, hq=40, mode="spec_tree", fp8=True)),
    ("A2FD", dict(L=60, B=3, lo=17, hi=90, kappa=4, gamma=4, hq=40, mode="greedy", fp8=True)),                   # short units
    ("A1FD", dict(L=40, B=1, lo=700, hi=700, kappa=4, gamma=4, hq=40, mode="greedy", fp8=True)),                 # whole ones
    ("A1FD", dict(L=42, B=1, lo=106, hi=106, kappa=8, gamma=6, hq=56, mode="greedy", vocab=12480, hidden=7680)), # an LM head of one wave: no SMs left to it
    ("A1FRMD", dict(L=16, B=8, lo=1000, hi=3000, kappa=8, gamma=6, hq=40, mode="spec_sampling", hidden=4096)),   # 392 rows: two row chunks, sums, spilled logits
    ("A1FRMD", dict(L=16, B=8, lo=1000, hi=3000, kappa=8, gamma=6, hq=40, mode="greedy", hidden=4096)),
    ("A2FDM", dict(L=12, B=1, lo=200, hi=200, kappa=8, gamma=7, hq=40, mode="greedy", headroom=6000)),           # a table much longer than the prefix:
    ("A2FRMD", dict(L=12, B=2, lo=30, hi=200, kappa=8, gamma=7, hq=64, mode="spec_sampling", headroom=3000)),    # the device finds less to share
    ("A1MRD", dict(L=2, B=4, lo=64, hi=9000, kappa=8, gamma=7, hq=40, mode="spec_sampling", vocab=2048)),        # hardly anything to run beside it
])
def test_the_ways_a_step_can_take(way, case):
    c = Case(**case)
    got = kernels(c.step)
    assert "".join(_NAMES[k] + (str(n[0]) if k == "attn_verify_kernel" else "") for k, n in got.items()) == way
    ref = c.parts()
    for _ in range(2):
        c.attn.fill_(float("nan")), c.argmax.fill_(-1)
        c.step()
        c.check(ref)


@pytest.mark.parametrize("mode", ["greedy", "spec_sampling"])
@pytest.mark.parametrize("fp8", [False, True])
def test_steps_in_a_row_without_waiting(mode, fp8):
    """Steps on the same buffers whose contents a kernel directly ahead changes, other calls of the context between them, and a graph of it
    all replayed back to back: each step finds its own rows and leaves its own results, as one that is waited for does."""
    case = dict(L=6, B=2, lo=300, hi=3000, kappa=8, gamma=7, hq=64, mode=mode, fp8=fp8)
    c = Case(**case)
    assert {"lmhead_pair_free_kernel", "attn_merge_kernel"} <= set(kernels(c.step))
    n, src = 4, []
    gen = torch.Generator(device="cuda").manual_seed(9)
    for _ in range(n):                                     # (other queries, rows and tree K/V for every step; codes in another order)
        kn, vn = [t[:, :, torch.randperm(t.shape[2], generator=gen, device="cuda")].contiguous() for t in (c.kn, c.vn)]
        src.append((torch.empty_like(c.x.q).normal_(generator=gen), kn, vn, torch.empty_like(c.x.hidden).normal_(generator=gen)))
    buffers = (c.x.q, c.kn, c.vn, c.x.hidden)
    results = lambda: [c.attn, c.argmax] + [getattr(c.out, f) for f in FIELDS]  # noqa: E731
    want = []
    for s in src:
        for d, t in zip(buffers, s):
            d.copy_(t)
        torch.cuda.synchronize()
        c.step()
        torch.cuda.synchronize()
        want.append([r.clone() for r in results()])
    assert not torch.equal(want[0][1], want[1][1])
    # other calls of the same context: attention alone, and the target's layers
    other_q = torch.empty_like(c.x.q).normal_(generator=gen)
    plain = make_mirror(c.cfg)
    bf = (c.x.k_pool, c.x.v_pool, c.x.page_table, c.x.prefix_len)
    layers, norm_final, emb = I.gen_layer_weights(c.cfg, 512, 2, 3, "cuda")
    def between(m, i):
        kv, tree = m.kv(*bf), m.tree(c.x.tokens, c.cfg.kappa, c.cfg.gamma)
        if i % 2:
            return [m.mirror_attn_verify(kv, tree, other_q, c.x.k_new if fp8 else src[0][1], c.x.v_new if fp8 else src[0][2])]
        t = m.target(layers, norm_final, 512)
        r = m.mirror_target_forward(t, kv, tree, emb)
        return [r["hidden"], r["attn_out"]]
    want_between = [between(plain, i) for i in range(2)]
    torch.cuda.synchronize()
    got, got_between = [[torch.zeros_like(r) for r in w] for w in want], [[] for _ in range(n)]

    def all_steps():
        for i, s in enumerate(src):
            for d, t in zip(buffers, s):
                d.copy_(t)
            c.step()
            got_between[i] = between(c.m, i)
            for d, r in zip(got[i], results()):
                d.copy_(r)

    def check():
        torch.cuda.synchronize()
        assert c.m.device_status() == (0, 0)
        for i in range(n):
            for a, b in zip(got[i], want[i]):
                assert torch.equal(a, b), i
                a.zero_()
            for a, b in zip(got_between[i], want_between[i % 2]):
                assert torch.equal(a, b), i

    all_steps()
    check()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        all_steps()
    for _ in range(3):
        g.replay()
    check()


@pytest.mark.parametrize("mode,B", [("greedy", 2), ("spec_sampling", 2), ("greedy", 6)])        # 66 rows: a state per CTA, a partial per unit; 198 rows
def test_a_wait_that_runs_out_beside_the_attention(mode, B, monkeypatch):
    """The launch is given up after one limit, and the context's unit counter is as it was."""
    case = dict(L=2, B=B, lo=100, hi=100, kappa=8, gamma=4, hq=16, mode=mode, hidden=512, vocab=200000)
    ref = Case(**case)
    assert "lmhead_pair_free_kernel" in kernels(ref.step)
    ref.step()
    monkeypatch.setenv("MIRROR_WAIT_LIMIT_CYCLES", "200000000")              # 0.1 s
    monkeypatch.setenv("MIRROR_TEST_STALL_AFTER_STAGES", "1")
    c, took, codes = Case(**case), [], []
    for call in (lambda: c.m.mirror_attn_verify(c.kv, c.tree, c.x.q, c.kn, c.vn), c.step):         # the attention's own stall; both CTAs of every pair
        torch.cuda.synchronize()
        t0 = time.monotonic()
        call()
        codes.append(c.m.device_status())
        took.append(time.monotonic() - t0)
    assert codes[0][0] == 7 and codes[1][0] == 7 and codes[1][1] in (11, 12, 13, 16, 17), codes
    assert took[1] < 1.5 * took[0], took
    for _ in range(2):
        c.attn.fill_(float("nan")), c.argmax.fill_(-1)
        c.step()
        assert c.m.device_status() == (0, 0)
        assert torch.equal(c.attn, ref.attn) and torch.equal(c.argmax, ref.argmax)
        got, want = c.out.cpu(), ref.out.cpu()
        for f in FIELDS:
            np.testing.assert_array_equal(got[f], want[f], err_msg=f)


@pytest.mark.parametrize("mode", ["greedy", "spec_sampling"])
def test_rows_per_unit_can_be_set(mode, monkeypatch):
    """MIRROR_LM_ROWS, as for an LM head of its own, where the workspace has room for that many units' partials."""
    case = dict(L=2, B=1, lo=100, hi=100, kappa=4, gamma=4, hq=16, mode=mode, hidden=512, vocab=20000)
    ref, blocks = Case(**case), {}
    ref.step()
    for rows in (0, 32, 96, 128):
        if rows:
            monkeypatch.setenv("MIRROR_LM_ROWS", str(rows))
        c = Case(**case)
        blocks[rows] = kernels(c.step)["lmhead_pair_free_kernel"][1]
        assert c.m.device_status() == (0, 0) and torch.equal(c.argmax, ref.argmax)
    # a CTA per `rows` ids; 32 would be 313 pairs of CTAs, more than there are, and more units than partials where each has its own
    assert blocks[96] == 2 * 105 and blocks[128] == 2 * 79 and blocks[32] == (296 if mode == "greedy" else blocks[0]), blocks
