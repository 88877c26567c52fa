"""head_dim 64, bf16 inputs: calls whose results are fp32 (partial forwards, merges, accumulated gradients) keep fp32
probabilities.  A split of P into two bf16 parts, good enough for bf16 results, is off by 2e-6 .. 1e-5 here."""
import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import workloads as W
from helpers import error_metrics, f32, oracle_fwd_bwd, to_dev

pytestmark = pytest.mark.gpu

# fp32 products and sums of 1,600 terms: roundings of 2^-24 of partial sums that grow to the result, 2^-24 sqrt(1600 / 3)
REL = 1.4e-6


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


@pytest.mark.parametrize("kind", [W.CHAIN, W.BLOCK])
def test_fp32_results_keep_fp32_probabilities(ba, oracle, kind):
    lens = [150, 1450]
    n = sum(lens)
    anchors = np.arange(3, n, 8, dtype=np.int32)
    p = W.Problem(W.cu_from_lengths(lens), anchors, W.uniform_branch_offsets(len(anchors), 4), kind, None, 4, 2, 64, dtype="bf16")
    t = W.make_tensors(p, seed=71, std=0.5)
    d = to_dev(p, t)
    qkv = (d["q_main"], d["q_branch"], d["k"], d["v"])
    want = oracle_fwd_bwd(oracle, p, t, backward=False)
    auto, simt = ba.Plan(p), ba.Plan(p, impl=ba.IMPL_SIMT)
    every, keys = ((0, n), (0, p.num_branches)), (0, n)
    o, lse = ba.branch_attn_fwd_partial(auto, *qkv, *every, keys, ba.PART_ALL)
    assert error_metrics(f32(o), want["o"])[1] <= REL and error_metrics(f32(lse), want["lse"])[1] <= REL
    o2, lse2 = ba.branch_attn_fwd_partial(simt, *qkv, *every, keys, ba.PART_ALL)
    assert torch.equal(o, o2) and torch.equal(lse, lse2)
    # in three steps, merged in place: rows that see nothing of a step, rows that have seen nothing before it
    acc = ba.branch_attn_fwd_partial(auto, *qkv, *every, (700, n), ba.PART_MAIN)
    for kv, parts in (((0, 100), ba.PART_MAIN), ((100, 700), ba.PART_ALL)):
        acc = ba.branch_attn_fwd_partial_merge(auto, *qkv, *every, kv, parts, *acc)
    assert error_metrics(f32(acc[0]), want["o"])[1] <= 2 * REL and error_metrics(f32(acc[1]), want["lse"])[1] <= REL
    ob, lb = ba.branch_attn_fwd(auto, *qkv)
    grads = []
    for plan in (auto, simt):
        g = [torch.zeros(s, device="cuda") for s in (d["q_main"].shape, d["q_branch"].shape, d["k"].shape, d["v"].shape)]
        ba.branch_attn_bwd(plan, *qkv, ob, lb, d["d_o"], accumulate=True, grads=g)
        grads.append(g)
    for name, a, b in zip(("dQ_main", "dQ_branch", "dK", "dV"), *grads):
        assert float(a.abs().max()) > 0 and torch.equal(a, b), name
    auto.check()


def test_tensors_on_8_byte_boundaries(ba):
    """Views that begin 8 bytes into an allocation: no tensor map can start there, the plain-FMA kernels can."""
    p = W.odd_shapes(W.TREE, head_dim=64, dtype="bf16")
    d = to_dev(p, W.make_tensors(p, seed=72, std=0.5))

    def shifted(x):
        buf = torch.zeros(x.numel() + 4, dtype=x.dtype, device="cuda")
        buf[4:] = x.flatten()
        return buf[4:].view(x.shape)

    results = []
    for move, impl in ((lambda x: x, ba.IMPL_SIMT), (shifted, ba.IMPL_AUTO)):
        plan = ba.Plan(p, impl=impl)
        qkv = [move(d[x]) for x in ("q_main", "q_branch", "k", "v")]
        o, lse = ba.branch_attn_fwd(plan, *qkv, out=move(torch.zeros_like(d["d_o"])))
        o = o.clone()                                   # (the backward's own pass over O and dO needs 16 bytes)
        grads = [move(torch.zeros_like(x)) for x in qkv]
        ba.branch_attn_bwd(plan, *qkv, o, lse, d["d_o"], grads=grads)
        plan.check()
        results.append((o, lse, *grads))
    assert results[1][2].data_ptr() % 16 == 8
    for a, b in zip(*results):
        assert torch.equal(a, b)
