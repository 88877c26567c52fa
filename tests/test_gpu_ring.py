"""The K/V ring driver on one GPU: ring steps read the received shard from a local
double buffer that a side stream fills while the previous step computes.  Its
results must equal the range-based zigzag driver's bit for bit (same kernels, same
accumulation order), which is itself checked against the oracle."""
import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import ring, zigzag
from paper_2609_07108_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


def inputs(p, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def draw(shape, std):
        return (torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std).to(torch.bfloat16)

    n, m = p.n_main, p.n_branch
    return (draw((n, p.h_q, 128), 0.5), draw((m, p.h_q, 128), 0.5), draw((n + m, p.h_kv, 128), 0.5),
            draw((n + m, p.h_kv, 128), 0.5), draw((n + m, p.h_q, 128), 0.1))


@pytest.mark.parametrize("cp", [2, 8])
def test_ring_equals_zigzag_bit_for_bit(ba, cp):
    p = W.config5(shrink=16)                   # 16,384 tokens: chunks of 1,024 (cp 8) / 4,096 (cp 2)
    plan = ba.Plan(p, impl=ba.IMPL_TC)
    qm, qb, k, v, go = inputs(p, 51)
    o1, l1, _ = zigzag.forward(ba, plan, qm, qb, k, v, cp)
    stats = ring.new_stats()
    bufs = ring.RingBuffers(plan, cp)
    # poison the double buffer: a step that read a slot before its shard arrived would show
    bufs.k.fill_(float("nan")); bufs.v.fill_(float("nan"))
    o2, l2, _ = ring.forward(ba, plan, qm, qb, k, v, cp, bufs=bufs, stats=stats)
    plan.check()
    assert torch.equal(o1, o2) and torch.equal(l1, l2)
    assert stats["copied_bytes"] == cp * ring.shard_bytes_per_rank(p, cp)      # Eq. cp-comm, every rank
    assert len(stats["copies"]) == cp * (cp - 1) and ring.copy_ms(stats) > 0.0
    g1 = zigzag.backward(ba, plan, qm, qb, k, v, o1, l1, go, cp, fused=False)
    g1 = [x.clone() for x in g1[:4]]
    g2 = ring.backward(ba, plan, qm, qb, k, v, o1, l1, go, cp, fused=False, bufs=bufs)
    plan.check()
    for name, a, b in zip(("dQ_main", "dQ_branch", "dK", "dV"), g1, g2[:4]):
        assert torch.equal(a, b), name
    # the one-kernel backward through the ring: dK, dV bit-identical, dQ up to the order of its atomic adds
    g3 = zigzag.backward(ba, plan, qm, qb, k, v, o1, l1, go, cp, fused=True)
    g3 = [x.clone() for x in g3[:4]]
    g4 = ring.backward(ba, plan, qm, qb, k, v, o1, l1, go, cp, fused=True, bufs=bufs)
    plan.check()
    assert torch.equal(g3[2], g4[2]) and torch.equal(g3[3], g4[3])
    for a, b in zip(g3[:2], g4[:2]):
        assert float((a.float() - b.float()).abs().max()) <= 1e-3 * max(1.0, float(a.float().abs().max()))


def test_shard_calls_check_their_ranges(ba):
    p = W.config5(shrink=64)
    plan = ba.Plan(p, impl=ba.IMPL_TC)
    qm, qb, k, v, go = inputs(p, 52)
    lib = ba._lib()
    x = ba._p(k)
    # shard ends must be multiples of 128 (or N): otherwise a key tile would reach outside the shard
    for kv in ((64, 256), (0, 200), (-128, 128), (256, 128), (0, p.n_main + 128)):
        rc = lib.branch_attn_fwd_shard(plan.handle, ba._p(qm), ba._p(qb), x, x, 0, 128, 0, 0, kv[0], kv[1], 0, x, x,
                                       ba._stream())
        assert rc == -1, kv
    torch.cuda.synchronize()


def test_ring_and_zigzag_at_head_dim_64(ba):
    """The steps' fp32 results come from the plain-FMA kernels, merged in their epilogue; the full call is on the
    tensor cores.  Both round O and the gradients to bf16 once."""
    n, cp = 1024, 2
    p = W.Problem(np.array([0, n], np.int32), np.arange(0, n, 3, dtype=np.int32), W.uniform_branch_offsets(342, 3), W.CHAIN, None,
                  4, 2, 64, dtype="bf16")
    plan = ba.Plan(p)
    g = torch.Generator(device="cuda").manual_seed(54)
    draw = lambda rows, heads, std: (torch.randn((rows, heads, 64), generator=g, device="cuda") * std).to(torch.bfloat16)
    qm, qb, k, v, go = draw(n, 4, 0.5), draw(p.n_branch, 4, 0.5), draw(p.rows, 2, 0.5), draw(p.rows, 2, 0.5), draw(p.rows, 4, 0.1)
    o, lse = ba.branch_attn_fwd(plan, qm, qb, k, v)
    want = ba.branch_attn_bwd(plan, qm, qb, k, v, o, lse, go)
    o1, l1, _ = zigzag.forward(ba, plan, qm, qb, k, v, cp)
    o2, l2, _ = ring.forward(ba, plan, qm, qb, k, v, cp)
    assert torch.equal(o1, o2) and torch.equal(l1, l2)
    assert float((o1.float() - o.float()).norm()) <= 4e-3 * float(o.float().norm()) and float((l1 - lse).abs().max()) <= 1e-5
    g1 = [x.clone() for x in zigzag.backward(ba, plan, qm, qb, k, v, o, lse, go, cp)[:4]]
    g2 = ring.backward(ba, plan, qm, qb, k, v, o, lse, go, cp)[:4]
    plan.check()
    for a, b, c in zip(g1, g2, want):      # (2^-9 per rounding)
        assert torch.equal(a, b) and float((a.float() - c.float()).norm()) <= 4e-3 * float(c.float().norm())


# Two sequences, the second one starting inside a shard; N no multiple of 32 or 128.  Behind each shard (in the same
# allocation) lie rows of NaN: a kernel that read them, and multiplied them with a weight of zero, would show.
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("kv", [(0, 256), (256, 512), (256, 733), (640, 733), (0, 733)])
def test_nothing_outside_a_shard_is_read(ba, head_dim, kv):
    n = 733
    p = W.Problem(W.cu_from_lengths([300, 433]), np.arange(0, n, 4, dtype=np.int32), W.uniform_branch_offsets(184, 3), W.CHAIN, None,
                  4, 2, head_dim, dtype="bf16")
    plan = ba.Plan(p)
    g = torch.Generator(device="cuda").manual_seed(53)
    draw = lambda rows, heads, std: (torch.randn((rows, heads, head_dim), generator=g, device="cuda") * std).to(torch.bfloat16)
    qm, qb, k, v, go = draw(n, 4, 0.5), draw(p.n_branch, 4, 0.5), draw(p.rows, 2, 0.5), draw(p.rows, 2, 0.5), draw(p.rows, 4, 0.1)

    def shard(x):
        buf = torch.full((kv[1] - kv[0] + 128, *x.shape[1:]), float("nan"), dtype=x.dtype, device="cuda")
        buf[:kv[1] - kv[0]] = x[kv[0]:kv[1]]
        return buf[:kv[1] - kv[0]]

    qm_range, br = (0, n), (0, p.num_branches)
    o_want, l_want = ba.branch_attn_fwd_partial(plan, qm, qb, k, v, qm_range, br, kv, ba.PART_MAIN)
    acc_o, acc_l = torch.full_like(o_want, 7.0), torch.full_like(l_want, 7.0)
    ba.branch_attn_fwd_shard(plan, qm, qb, shard(k), shard(v), qm_range, br, kv, acc_o, acc_l, merge=False)
    assert torch.equal(acc_o, o_want) and torch.equal(acc_l, l_want)
    o, lse = ba.branch_attn_fwd(plan, qm, qb, k, v)
    zeros = lambda rows, heads: torch.zeros((rows, heads, head_dim), device="cuda")
    for stages in (ba.STAGE_ALL, ba.STAGE_ALL_FUSED):
        if head_dim == 64 and stages == ba.STAGE_ALL_FUSED:
            continue                                   # the one-kernel backward needs head_dim 128
        want = (zeros(n, 4), zeros(p.n_branch, 4), zeros(p.rows, 2), zeros(p.rows, 2))
        ba.branch_attn_bwd(plan, qm, qb, k, v, o, lse, go, qm_range, br, kv, ba.PART_MAIN, accumulate=True, grads=want, stages=stages)
        dq, db, dk, dv = zeros(n, 4), zeros(p.n_branch, 4), zeros(kv[1] - kv[0], 2), zeros(kv[1] - kv[0], 2)
        ba.branch_attn_bwd_shard(plan, qm, qb, shard(k), shard(v), o, lse, go, qm_range, br, kv, dq, db, dk, dv, stages=stages)
        plan.check()
        assert torch.equal(dk, want[2][kv[0]:kv[1]]) and torch.equal(dv, want[3][kv[0]:kv[1]])
        for a, b in ((dq, want[0]), (db, want[1])):
            if stages == ba.STAGE_ALL:
                assert torch.equal(a, b)
            else:          # fp32 atomic adds of up to six key tiles: the order moves the last bits
                assert float((a - b).abs().max()) <= 6 * 2.0 ** -23 * float(b.abs().max())
