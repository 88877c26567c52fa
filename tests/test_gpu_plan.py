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


def device_plan(ba, p, uniform_len=0):
    """(status, handle, what must stay alive) of ba_plan_create: metadata in device memory, checked there."""
    arrays = [None if a is None else torch.from_numpy(np.asarray(a, np.int32)).cuda()
              for a in (p.cu_seqlens, p.anchor_idx, p.branch_offsets, p.parent)]
    prob = ba._Problem(p.n_main, p.n_branch, p.num_seqs, p.num_branches, p.h_q, p.h_kv, p.head_dim, ba._DT[p.dtype][0], 0.0,
                       int(p.kind), uniform_len, ba.IMPL_AUTO, *[None if a is None else a.data_ptr() for a in arrays])
    nbytes = ba._lib().ba_plan_bytes(ba.C.byref(prob))
    mem = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    handle = ba.C.c_void_p()
    rc = ba._lib().ba_plan_create(ba.C.byref(prob), ba._p(mem), nbytes, ba._stream(), ba.C.byref(handle))
    return rc, handle, (arrays, mem)


@pytest.mark.parametrize("uniform", [False, True])
@pytest.mark.parametrize("kind", [W.CHAIN, W.BLOCK, W.TREE])
def test_device_built_plan_equals_the_host_built_one(ba, kind, uniform):
    p = W.odd_shapes(kind, head_dim=128, dtype="bf16")
    if uniform:
        rng = np.random.default_rng(3)
        parent = np.concatenate([W.random_tree_parents(rng, 5, 3) for _ in p.anchor_idx]).astype(np.int32)
        p = W.Problem(p.cu_seqlens, p.anchor_idx, W.uniform_branch_offsets(p.num_branches, 5), kind,
                      parent if kind == W.TREE else None, 4, 2, 128)
    d = to_dev(p, W.make_tensors(p, seed=4, std=0.5))
    host = ba.Plan(p)
    rc, handle, alive = device_plan(ba, p, 5 if uniform else 0)
    assert rc == 0
    lib = ba._lib()
    assert lib.ba_plan_pairs(handle) == host.pairs == W.useful_pairs(p) and lib.ba_plan_impl(handle) == host.impl
    o, lse = ba.branch_attn_fwd(host, d["q_main"], d["q_branch"], d["k"], d["v"])
    o2, lse2 = torch.zeros_like(o), torch.zeros_like(lse)
    assert lib.branch_attn_fwd(handle, *[ba._p(d[x]) for x in ("q_main", "q_branch", "k", "v")], ba._p(o2), ba._p(lse2), None, 0,
                               ba._stream()) == 0
    assert lib.ba_plan_check(handle, ba._stream()) == 0
    assert torch.equal(o, o2) and torch.equal(lse, lse2)
    lib.ba_plan_destroy(handle)


def test_branches_of_one_length_given_as_offsets(ba):
    """Recognised by ba_plan_create_host (per-depth calls work), taken as they are by ba_plan_create (refused)."""
    p = W.Problem(np.array([0, 40], np.int32), np.arange(10, dtype=np.int32), W.uniform_branch_offsets(10, 3), W.CHAIN, None, 4, 2, 128)
    d = to_dev(p, W.make_tensors(p, seed=5, std=0.5))
    q = torch.zeros((10, 4, 128), dtype=torch.bfloat16, device="cuda")
    ba.branch_attn_fwd_depth(ba.Plan(p), 1, q, d["k"], d["v"])
    for uniform, want in ((0, -2), (3, 0)):
        rc, handle, alive = device_plan(ba, p, uniform)
        assert rc == 0
        o, lse = torch.zeros_like(q), torch.zeros((10, 4), device="cuda")
        assert ba._lib().branch_attn_fwd_depth(handle, 1, ba._p(q), ba._p(d["k"]), ba._p(d["v"]), 0, 10, ba._p(o), ba._p(lse),
                                               ba._stream()) == want
        torch.cuda.synchronize()
        ba._lib().ba_plan_destroy(handle)


def test_bad_metadata_is_refused_on_the_device(ba):
    p = W.odd_shapes(W.TREE)
    cu, an, of, pa = (np.array(x) for x in (p.cu_seqlens, p.anchor_idx, p.branch_offsets, p.parent))

    def at(x, i, v):
        y = x.copy()
        y[i] = v
        return y

    for c in (dict(cu_seqlens=at(cu, 0, 1)), dict(cu_seqlens=at(cu, 1, cu[2] + 1)), dict(anchor_idx=at(an, 0, -1)),
              dict(anchor_idx=at(an, len(an) - 1, p.n_main)), dict(anchor_idx=at(an, 3, an[2] - 1)),
              dict(branch_offsets=at(of, 0, 1)), dict(branch_offsets=at(of, 2, of[3] + 1)), dict(branch_offsets=at(of, 3, of[2] + 65)),
              dict(parent=at(pa, 5, 4)), dict(parent=at(pa, 0, -2)), dict(parent=at(pa, of[2], 0))):
        rc, handle, alive = device_plan(ba, bad(p, **c))
        assert rc == -4 and not handle.value, list(c)
