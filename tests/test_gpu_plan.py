"""The plan is validated and counted on the host and built without waiting for the GPU: bad metadata of every
kind is refused at once, and a plan built on one stream can be used from another straight away."""
import copy

import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import workloads as W
from helpers import f32, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


def bad(p, **changes):
    q = copy.copy(p)
    for k, v in changes.items():
        setattr(q, k, np.asarray(v, np.int32))
    return q


def test_bad_metadata_is_refused(ba):
    p = W.odd_shapes(W.TREE)
    cu, an, of, pa = (np.array(x) for x in (p.cu_seqlens, p.anchor_idx, p.branch_offsets, p.parent))

    def at(x, i, v):
        y = x.copy()
        y[i] = v
        return y

    n = p.n_main
    cases = [dict(cu_seqlens=at(cu, 0, 1)), dict(cu_seqlens=at(cu, 1, cu[2] + 1)), dict(anchor_idx=at(an, 0, -1)),
             dict(anchor_idx=at(an, len(an) - 1, n)), dict(anchor_idx=at(an, 3, an[2] - 1)),
             dict(branch_offsets=at(of, 0, 1)), dict(branch_offsets=at(of, 2, of[3] + 1)),
             dict(branch_offsets=at(of, 3, of[2] + 65)), dict(branch_offsets=of[:-1]), dict(parent=at(pa, 5, 4)),
             dict(parent=at(pa, 0, -2)), dict(parent=at(pa, of[2], 0)), dict(parent=pa[:-1])]
    for c in cases:
        with pytest.raises(ba.BranchAttnError) as e:
            ba.Plan(bad(p, **c))
        assert e.value.code == -4, (list(c), e.value)
    assert ba.Plan(p).pairs == W.useful_pairs(p)


@pytest.mark.parametrize("kind", [W.CHAIN, W.BLOCK, W.TREE])
def test_plan_used_from_another_stream(ba, kind):
    p = W.odd_shapes(kind, head_dim=128, dtype="bf16")
    d = to_dev(p, W.make_tensors(p, seed=1, std=0.5))
    want = f32(ba.branch_attn_fwd(ba.Plan(p), d["q_main"], d["q_branch"], d["k"], d["v"])[0])
    busy = torch.randn(4096, 4096, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        busy = busy @ busy.clamp(-1e-3, 1e-3)          # the plan's own kernel waits behind this
    plan = ba.Plan(p)
    with torch.cuda.stream(side):
        o, _ = ba.branch_attn_fwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"])
    torch.cuda.synchronize()
    assert (f32(o) == want).all()


@pytest.mark.parametrize("error_mode", ["global", "thread_local", "relaxed"])
def test_plan_captured_right_after_it_was_built(ba, error_mode):
    """A capture that does not begin with a synchronisation: the plan's kernel waits behind other work on its stream
    while calls that use the plan are captured on another one.  The replay must find the metadata."""
    p = W.odd_shapes(W.TREE, head_dim=128, dtype="bf16")
    d = to_dev(p, W.make_tensors(p, seed=2, std=0.5))
    want = f32(ba.branch_attn_fwd(ba.Plan(p), d["q_main"], d["q_branch"], d["k"], d["v"])[0])
    busy = torch.randn(4096, 4096, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    o, lse = torch.zeros((p.rows, p.h_q, 128), dtype=torch.bfloat16, device="cuda"), torch.zeros((p.rows, p.h_q), device="cuda")
    torch.cuda.synchronize()
    for _ in range(20):
        busy = busy @ busy.clamp(-1e-3, 1e-3)
    plan = ba.Plan(p)
    with torch.cuda.stream(side):
        graph.capture_begin(capture_error_mode=error_mode)
        ba.branch_attn_fwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"], out=o, lse=lse)
        with pytest.raises(RuntimeError):
            ba.Plan(p)                                 # its copy and kernel would run at each replay only
        graph.capture_end()
        assert plan._ready is None                     # the host has waited
        graph.replay()
    torch.cuda.synchronize()
    assert (f32(o) == want).all()


def test_plan_wait(ba):
    p = W.odd_shapes(W.CHAIN)
    busy = torch.randn(4096, 4096, device="cuda")
    for _ in range(20):
        busy = busy @ busy.clamp(-1e-3, 1e-3)
    plan = ba.Plan(p)
    done = torch.cuda.Event()
    done.record()
    plan.wait()
    plan.wait()
    assert plan._ready is None and plan.pairs == W.useful_pairs(p)
    assert ba._lib().ba_host_wait(ba.C.c_void_p(done.cuda_event)) == 0 and done.query()


@pytest.mark.parametrize("kind", [W.CHAIN, W.BLOCK])
@pytest.mark.parametrize("length", [0, 3])
def test_parents_of_chains_and_blocks_are_not_looked_at(ba, kind, length):
    p = W.odd_shapes(kind)
    assert ba.Plan(bad(p, parent=np.full(length, 7))).pairs == W.useful_pairs(p)
