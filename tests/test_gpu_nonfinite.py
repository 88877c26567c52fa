"""A NaN or an infinity in one row reaches only the results whose definition contains that row: the plain-FMA
kernels (fp32, any shape) and the head_dim 64 tensor-core kernels leave every other row as it is.  What a row may
reach follows from the oracle's visibility matrix alone."""
import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import workloads as W
from helpers import TOL, REL_RMS, f32, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


def problem(kind, head_dim, dtype, lens, anchors, blen, h_q=4, h_kv=2):
    anchors = np.sort(np.asarray(anchors, np.int32))
    rng = np.random.default_rng(11)
    parent = None
    if kind == W.TREE:
        parent = np.concatenate([W.random_tree_parents(rng, blen, 4) for _ in anchors]).astype(np.int32)
    return W.Problem(W.cu_from_lengths(lens), anchors, W.uniform_branch_offsets(len(anchors), blen), kind, parent, h_q, h_kv,
                     head_dim, dtype=dtype)


# (kind, head_dim, dtype, plain-FMA kernels?): lengths that leave sequences, branches and the poisoned rows in the
# middle of 32-, 64- and 128-row tiles; few rows (tiles shared by clusters) and enough rows to leave tiles whole
SMALL = dict(lens=[70, 131, 300], anchors=list(range(0, 501, 9)), blen=5)
LARGE = dict(lens=[1500, 333, 2200], anchors=list(range(0, 4033, 5)), blen=3, h_q=8, h_kv=8)
SHARED = dict(lens=[40, 600, 5], anchors=list(range(645)), blen=3, h_q=8, h_kv=1)     # dK/dV in clusters of four
CASES = [(W.CHAIN, 64, "fp32", False, SMALL), (W.TREE, 128, "fp32", False, SMALL), (W.BLOCK, 64, "fp32", False, LARGE),
         (W.TREE, 64, "bf16", False, SMALL), (W.CHAIN, 64, "bf16", False, LARGE), (W.CHAIN, 64, "bf16", True, SMALL),
         (W.CHAIN, 64, "bf16", False, SHARED), (W.BLOCK, 128, "bf16", True, SMALL)]


def poisoned(p, d, name, row, value):
    """Tensors with row `row` (global numbering) of tensor `name` set to `value` in the last query / KV head."""
    d = {k: v.clone() for k, v in d.items()}
    if name == "q":
        t, row = (d["q_main"], row) if row < p.n_main else (d["q_branch"], row - p.n_main)
    else:
        t = d[name]
    t[row, -1, 3:7] = value
    return d


def check(name, got, want, hit, dtype):
    """`hit`: [rows, heads] results that the poisoned row may reach (and, all together, does); the others are what
    they were.  (Two sums in another order: bf16 results may round the other way, fp32 sums differ in the last bits.)"""
    bad = ~np.isfinite(got).all(axis=-1)
    assert not (bad & ~hit).any(), f"{name}: {int((bad & ~hit).sum())} rows out of reach are not finite"
    assert bad[hit].any(), f"{name}: the poison reached nothing"
    g, w = got[~hit].astype(np.float64), want[~hit].astype(np.float64)
    assert np.abs(g - w).max() <= TOL[dtype]
    assert np.linalg.norm(g - w) <= REL_RMS[dtype] * np.linalg.norm(w), name


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("kind,head_dim,dtype,simt,size", CASES)
def test_a_poisoned_row_reaches_what_contains_it_only(ba, oracle, kind, head_dim, dtype, simt, size, value):
    p = problem(kind, head_dim, dtype, **size)
    d = to_dev(p, W.make_tensors(p, seed=61, std=0.5))
    plan = ba.Plan(p, impl=ba.IMPL_SIMT if simt else ba.IMPL_AUTO)
    n, group = p.n_main, p.h_q // p.h_kv
    vis = oracle.visibility(p)                          # [query row, key row]
    o, lse = ba.branch_attn_fwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"])

    def backward(d, o):
        g = ba.branch_attn_bwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"], o, lse, d["d_o"])
        return [np.concatenate([f32(g[0]), f32(g[1])]), f32(g[2]), f32(g[3])]

    clean_o, clean = f32(o), backward(d, o)
    q_head = np.arange(p.h_q) >= p.h_q - group          # query heads of the poisoned KV head
    kv_head = np.arange(p.h_kv) >= p.h_kv - 1
    last_q = np.arange(p.h_q) >= p.h_q - 1
    none_q, none_k = np.zeros((p.rows, p.h_q), bool), np.zeros((p.rows, p.h_kv), bool)
    # a key in the middle of a sequence, the first key of the next one, a branch key
    for x in (int(p.cu_seqlens[1]) + 37, int(p.cu_seqlens[2]), n + 2 * (p.n_branch // 5)):
        viewers = vis[:, x]
        q_hit = viewers[:, None] & q_head
        k_hit = (np.arange(p.rows) == x)[:, None] & kv_head
        for name in ("k", "v"):
            dd = poisoned(p, d, name, x, value)
            po, pl = ba.branch_attn_fwd(plan, dd["q_main"], dd["q_branch"], dd["k"], dd["v"])
            check(f"O, poisoned {name}[{x}]", f32(po), clean_o, q_hit, dtype)
            assert torch.equal(pl[torch.from_numpy(~q_hit).cuda()], lse[torch.from_numpy(~q_hit).cuda()])
            dq, dk, dv = backward(dd, o)
            check(f"dQ, poisoned {name}[{x}]", dq, clean[0], q_hit, dtype)
            check(f"dK, poisoned {name}[{x}]", dk, clean[1], k_hit, dtype)
            if name == "k":
                check(f"dV, poisoned k[{x}]", dv, clean[2], k_hit, dtype)
    # a query row: late in a sequence, the last of one, a branch row
    for r in (int(p.cu_seqlens[2]) - 20, int(p.cu_seqlens[1]) - 1, n + p.n_branch // 3):
        q_hit = (np.arange(p.rows) == r)[:, None] & last_q
        k_hit = vis[r][:, None] & kv_head
        for name in ("q", "d_o"):
            dq, dk, dv = backward(poisoned(p, d, name, r, value), o)
            check(f"dQ, poisoned {name}[{r}]", dq, clean[0], q_hit, dtype)
            check(f"dK, poisoned {name}[{r}]", dk, clean[1], k_hit, dtype)
            check(f"dV, poisoned {name}[{r}]", dv, clean[2], k_hit, dtype)
    plan.check()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (64, "fp32")])
def test_a_poisoned_key_of_few_rows_on_long_sequences(ba, oracle, head_dim, dtype, value):
    """Draft rows only: the keys of an item are split over a cluster, both query tiles hold one sequence's rows.  Rows
    that see the poison are not finite, whichever part it is in (head_dim 128: others may be, see branch_attn.h)."""
    p = problem(W.TREE, head_dim, dtype, [2100, 1900], [1800, 2099, 3999], 6)
    d = to_dev(p, W.make_tensors(p, seed=62, std=0.5))
    plan, n, q_head = ba.Plan(p), p.n_main, np.arange(p.h_q) >= p.h_q // 2
    vis = oracle.visibility(p)[n:]
    o, _ = ba.branch_attn_fwd(plan, None, d["q_branch"], d["k"], d["v"])
    for x in (7, 1900, 2050, 2099, 2101, n + 8):
        for name in ("k", "v"):
            dd = poisoned(p, d, name, x, value)
            po, _ = ba.branch_attn_fwd(plan, None, dd["q_branch"], dd["k"], dd["v"])
            hit = vis[:, x][:, None] & q_head
            if name == "v" or np.isnan(value):      # (an infinite key may also make a score of -inf)
                assert not np.isfinite(f32(po)[n:][hit]).all(axis=-1).any(), f"poisoned {name}[{x}] is lost"
            if head_dim == 64:
                check(f"O, poisoned {name}[{x}]", f32(po)[n:], f32(o)[n:], hit, dtype)
    plan.check()



@pytest.mark.parametrize("head_dim,dtype,simt", [(64, "fp32", False), (128, "fp32", False), (64, "bf16", True), (64, "bf16", False), (128, "bf16", False)])
def test_rows_that_see_nan_alone_are_nan(ba, head_dim, dtype, simt):
    """Every key of one KV head is NaN: no score of its rows is a maximum.  O is NaN, not an empty row's zero."""
    p = problem(W.CHAIN, head_dim, dtype, [90, 1], [0, 60, 90], 3)
    d = to_dev(p, W.make_tensors(p, seed=64, std=0.5))
    d["k"][:, -1] = float("nan")
    plan = ba.Plan(p, impl=ba.IMPL_SIMT if simt else ba.IMPL_AUTO)
    o, _ = ba.branch_attn_fwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"])
    plan.check()
    half = p.h_q // 2
    assert np.isnan(f32(o)[:, half:]).all() and np.isfinite(f32(o)[:, :half]).all()


@pytest.mark.parametrize("head_dim,dtype,stages", [(64, "fp32", 7), (64, "bf16", 7), (128, "bf16", 7), (128, "bf16", 9)])
@pytest.mark.parametrize("lens", [[130, 91], [130, 92], [3, 222, 66]])     # N = 221, 222, 291
def test_a_call_without_main_queries_reads_no_main_row_of_d_o(ba, head_dim, dtype, stages, lens):
    p = problem(W.CHAIN, head_dim, dtype, lens, list(range(sum(lens))), 4)
    d = to_dev(p, W.make_tensors(p, seed=63, std=0.5))
    plan, n = ba.Plan(p), p.n_main
    o, lse = ba.branch_attn_fwd(plan, d["q_main"], d["q_branch"], d["k"], d["v"])
    results = []
    for fill in (0.0, float("nan")):
        d["d_o"][:n] = fill
        g = ba.branch_attn_bwd(plan, None, d["q_branch"], d["k"], d["v"], o, lse, d["d_o"], stages=stages)
        results.append([f32(x) for x in g[1:]])
    plan.check()
    for name, a, b in zip(("dQ", "dK", "dV"), *results):
        assert np.isfinite(b).all(), name
        assert np.abs(a - b).max() <= (1e-3 * np.abs(a).max() if stages == 9 else 0.0), name    # (atomic adds, rounded to bf16)
