"""Tensors that start off a 16-byte boundary: refused on the host before any kernel of the call, or (bf16 on the plain-FMA
kernels) taken with the same results."""
import pytest
import torch

from paper_2609_07108_b200 import workloads as W
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
