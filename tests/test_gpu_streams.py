"""Calls on streams that are not the default one, and captured into graphs: forward and backward (delta and dQ may be launched
while the kernel before them ends), and the zigzag backward that spreads its blocks over two streams."""
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


@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("fp32", 128), ("bf16", 64), ("bf16", 128)])
def test_step_captured(ba, dtype, d):
    """Two steps in one graph, the second on other inputs than the first, replayed on inputs that the capture has not seen."""
    p = W.odd_shapes(W.BLOCK, head_dim=d, dtype=dtype)
    data = [to_dev(p, W.make_tensors(p, seed=s, std=0.5)) for s in (1, 2, 3)]
    plan = ba.Plan(p)

    def step(t):
        o, lse = ba.branch_attn_fwd(plan, t["q_main"], t["q_branch"], t["k"], t["v"])
        return (o, lse, *ba.branch_attn_bwd(plan, t["q_main"], t["q_branch"], t["k"], t["v"], o, lse, t["d_o"]))

    want = [[x.clone() for x in step(t)] for t in data]
    live = [{k: v.clone() for k, v in t.items()} for t in data[:2]]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [step(t) for t in live]
    for order in ((0, 1), (2, 0), (1, 2)):
        for t, i in zip(live, order):
            for k in t:
                t[k].copy_(data[i][k])
        graph.replay()
        for out, i in zip(got, order):
            for a, b in zip(out, want[i]):
                assert torch.equal(a, b)
    plan.check()


@pytest.mark.parametrize("captured", [False, True])
def test_zigzag_backward_on_another_stream(ba, captured):
    n, cp = 2048, 2
    p = W.Problem(np.array([0, n], np.int32), np.arange(n, dtype=np.int32), W.uniform_branch_offsets(n, 3), W.CHAIN, None, 8, 2, 128)
    assert zigzag.two_streams(p, p.rows // (2 * cp))
    t = to_dev(p, W.make_tensors(p, seed=4, std=0.5))
    names = ("q_main", "q_branch", "k", "v", "d_o")
    plan = ba.Plan(p)
    o, lse = ba.branch_attn_fwd(plan, t["q_main"], t["q_branch"], t["k"], t["v"])
    want = [x.clone() for x in zigzag.backward(ba, plan, *[t[x] for x in names[:4]], o, lse, t["d_o"], cp, fused=True)[:4]]
    ws, main = zigzag.Workspace(ba, plan, cp), torch.cuda.Stream()
    live = {x: torch.full_like(t[x], float("nan")) for x in names}

    def run():
        return zigzag.backward(ba, plan, *[live[x] for x in names[:4]], o, lse, live["d_o"], cp, fused=True, ws=ws)[:4]

    graph = torch.cuda.CUDAGraph()
    busy = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(main):
        if captured:
            graph.capture_begin()
            run()
            graph.capture_end()
        for _ in range(20):                      # the inputs arrive behind this, and the results are taken straight away
            busy = busy @ busy.clamp(-1e-3, 1e-3)
        for x in names:
            live[x].copy_(t[x])
        graph.replay() if captured else run()
        got = [x.clone() for x in ws.outs]
    main.synchronize()
    plan.check()
    assert torch.equal(got[2], want[2]) and torch.equal(got[3], want[3])
    for a, b in zip(got[:2], want[:2]):          # fp32 atomic adds in another order, then one rounding to bf16
        assert float((a.float() - b.float()).norm()) <= 2.0 ** -9 * float(b.float().norm())
