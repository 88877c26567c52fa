"""Tensors that start off a 16-byte boundary: refused on the host before any kernel of the call, or (bf16 on the plain-FMA
kernels, and what ba_finalize_grads converts) taken with the same results."""
import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import workloads as W
from paper_2609_07108_b200 import zigzag
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


def moved(x, nbytes):
    skip = nbytes // x.element_size()
    buf = torch.zeros(x.numel() + skip, dtype=x.dtype, device="cuda")
    buf[skip:] = x.flatten()
    return buf[skip:].view(x.shape)


ROWS = ("q_main", "q_branch", "k", "v")
GRADS = ("dq_main", "dq_branch", "dk", "dv")


# head_dim, plain-FMA plan, bytes off; what is refused by the forward and by the backward
@pytest.mark.parametrize("dtype,d,simt,off,fwd,bwd", [
    ("bf16", 128, False, 8, (*ROWS, "o"), (*ROWS, "o", "d_o", *GRADS)),
    ("bf16", 128, True, 8, (), ("o", "d_o")),
    ("bf16", 64, False, 8, (), ("o", "d_o")),
    ("bf16", 64, False, 4, (*ROWS, "o"), (*ROWS, "o", "d_o", *GRADS)),
    ("fp32", 64, False, 8, (*ROWS, "o"), (*ROWS, "o", "d_o", *GRADS)),
])
def test_calls_refuse_what_they_cannot_address(ba, dtype, d, simt, off, fwd, bwd):
    p = W.odd_shapes(W.BLOCK, head_dim=d, dtype=dtype)
    p.h_q, p.h_kv = 3, 1                        # (three heads to a group: no TMA store of O)
    t = to_dev(p, W.make_tensors(p, seed=6, std=0.5))
    plan = ba.Plan(p, impl=ba.IMPL_SIMT if simt else ba.IMPL_AUTO)
    o, lse = ba.branch_attn_fwd(plan, *[t[x] for x in ROWS])
    base = {**{x: t[x] for x in (*ROWS, "d_o")}, "o": o, **dict(zip(GRADS, (torch.full_like(t[x], 7.0) for x in ROWS)))}
    ws = plan.workspace(ba.OP_BWD)

    def call(c):
        ba.branch_attn_fwd(plan, *[c[x] for x in ROWS], out=c["o"], lse=lse.clone())

    def back(c, **k):
        ba.branch_attn_bwd(plan, *[c[x] for x in ROWS], c["o"], lse, c["d_o"], grads=tuple(c[x] for x in GRADS), **k)

    for refused, f, outputs in ((fwd, call, ("o",)), (bwd, back, GRADS)):
        for x in refused:
            c = {**base, x: moved(base[x], off)}
            before = {y: c[y].clone() for y in outputs}
            ws.fill_(0x5a)
            with pytest.raises(ba.BranchAttnError) as e:
                f(c)
            assert e.value.code == -1, x
            assert bool((ws == 0x5a).all()) and all(torch.equal(before[y], c[y]) for y in outputs), x
    # fp32 results: partial outputs and accumulated gradients
    out = moved(torch.zeros((p.rows, 3, d), device="cuda"), 8)
    with pytest.raises(ba.BranchAttnError):
        ba.branch_attn_fwd_partial(plan, *[t[x] for x in ROWS], (0, p.n_main), (0, p.num_branches), (0, p.n_main), ba.PART_ALL, out=out)
    for i in range(4):
        grads = [torch.zeros_like(t[x], dtype=torch.float32) for x in ROWS]
        grads[i] = moved(grads[i], 8)
        with pytest.raises(ba.BranchAttnError):
            ba.branch_attn_bwd(plan, *[t[x] for x in ROWS], o, lse, t["d_o"], accumulate=True, grads=tuple(grads))
    plan.check()
    # what a stage does not touch may be anywhere
    back({**base, **{x: moved(base[x], off) for x in GRADS}}, stages=ba.STAGE_PREP)
    back({**base, "o": moved(o, off), "dk": moved(base["dk"], off)}, stages=ba.STAGE_DQ)
    back(base, stages=ba.STAGE_DKDV)
    want = [base[x].clone() for x in GRADS]
    back(base)
    plan.check()
    for x, w in zip(GRADS, want):      # (head_dim 64: the stages above ran on different kernels, one rounding to bf16 each)
        assert torch.equal(base[x], w) or (d == 64 and float((base[x] - w).float().norm()) <= 2.0 ** -8 * float(w.float().norm()))


@pytest.mark.parametrize("dst", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("count", [1, 3, 4, 5, 4099])
def test_finalize_at_any_element(ba, dst, count):
    g = torch.Generator(device="cuda").manual_seed(count)
    src = torch.randn(count + 8, generator=g, device="cuda")
    for a in (0, 1, 2, 4, 7):
        for b in (0, 1, 4, 7):
            out = torch.full((count + 16,), 7.0, dtype=dst, device="cuda")
            ba.ba_finalize_grads(src[a:a + count], dst=out[b:b + count])
            assert torch.equal(out[b:b + count], src[a:a + count].to(dst))
            assert bool((out[:b] == 7).all()) and bool((out[b + count:] == 7).all())


@pytest.mark.parametrize("n,cp,h_q,h_kv", [(1092, 2, 5, 1), (1084, 2, 3, 1), (1020, 2, 1, 1)])
def test_zigzag_with_rows_of_lse_off_16_bytes(ba, n, cp, h_q, h_kv):
    """Chunks of 273, 271 and 255 rows: the rows of LSE of a chunk, or of its branches, start on any 4-byte boundary."""
    p = W.Problem(np.array([0, n], np.int32), np.arange(0, n, 3, dtype=np.int32), W.uniform_branch_offsets((n + 2) // 3, 3), W.CHAIN,
                  None, h_q, h_kv, 128)
    t = to_dev(p, W.make_tensors(p, seed=7, std=0.5))
    plan = ba.Plan(p)
    qkv = [t[x] for x in ROWS]
    o, lse = ba.branch_attn_fwd(plan, *qkv)
    want = ba.branch_attn_bwd(plan, *qkv, o, lse, t["d_o"])
    o1, lse1, _ = zigzag.forward(ba, plan, *qkv, cp)
    assert float((lse1 - lse).abs().max()) <= 1e-5
    assert float((o1.float() - o.float()).norm()) <= 4e-3 * float(o.float().norm())          # two roundings to bf16
    for fused in (False, True):
        got = zigzag.backward(ba, plan, *qkv, o, lse, t["d_o"], cp, fused=fused)[:4]
        for a, b in zip(got, want):
            # one rounding to bf16 each, and P, dS rounded to bf16 against another running order of the tiles
            assert float((a.float() - b.float()).norm()) <= 6e-3 * float(b.float().norm())
    plan.check()
