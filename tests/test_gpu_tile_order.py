"""The order in which kernels take the tiles of a packed batch: formed with the plan, found again by the launch, a permutation,
and heaviest first by weights restated here from the definition of the mask."""
import numpy as np
import pytest
import torch

from paper_2609_07108_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ba():
    from paper_2609_07108_b200 import binding
    assert torch.cuda.is_available()
    return binding


def tile_order(ba, plan, stage, has_main):
    tiling, order = np.zeros(4, np.int64), np.zeros(4096, np.uint16)
    n = ba._lib().ba_plan_tile_order(plan.handle, stage, int(has_main), tiling.ctypes.data, order.ctypes.data, order.size)
    assert n >= 0
    return tiling.tolist(), order[:n].astype(int)


def weights(p, keys, has_main, tiling):
    """Extent of what the rows of each tile see (keys: of what sees them), plus the tile's own branch tokens."""
    mt, ms, bt, bs = tiling
    seq_of = np.repeat(np.arange(len(p.cu_seqlens) - 1), np.diff(p.cu_seqlens))
    lo, end = p.cu_seqlens[:-1][seq_of], p.cu_seqlens[1:][seq_of]            # of every main row
    anchor = np.repeat(p.anchor_idx, np.diff(p.branch_offsets))              # of every branch token
    out = []
    for i in range(mt):
        rows = np.arange(i * ms, min((i + 1) * ms, p.n_main))
        if keys:
            stop = end[rows].max()
            viewers = np.flatnonzero((anchor >= rows[0]) & (anchor < stop)).size
            out.append((stop - rows[0] if has_main else 0) + viewers)
        else:
            out.append(rows[-1] - lo[rows].min() + 1)
    for i in range(bt):
        tok = np.arange(i * bs, min((i + 1) * bs, p.n_branch))
        out.append(tok.size + (0 if keys else anchor[tok].max() - lo[anchor[tok]].min() + 1))
    return np.array(out)


def ragged(kind, d, dtype, h_q, h_kv, uniform):
    rng = np.random.default_rng(11)
    lens = [1, 700, 0, 130, 257, 1411, 0, 64, 900]
    n = sum(lens)
    anchors = np.sort(rng.choice(n, size=200)).astype(np.int32)
    blens = np.full(200, 7) if uniform else rng.integers(0, 23, 200)
    offsets = np.concatenate([[0], np.cumsum(blens)]).astype(np.int32)
    return W.Problem(W.cu_from_lengths(lens), anchors, offsets, kind, None, h_q, h_kv, d, dtype=dtype)


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("d,dtype,h_q,h_kv", [(128, "bf16", 4, 1), (128, "bf16", 3, 3), (64, "bf16", 4, 2), (128, "fp32", 4, 2),
                                              (64, "fp32", 5, 1)])
def test_heaviest_first(ba, d, dtype, h_q, h_kv, uniform):
    p = ragged(W.BLOCK, d, dtype, h_q, h_kv, uniform)
    plan = ba.Plan(p)
    for stage in (0, ba.STAGE_DQ, ba.STAGE_DKDV):
        for has_main in (True, False):
            tiling, order = tile_order(ba, plan, stage, has_main)
            keys, tiles = stage == ba.STAGE_DKDV, tiling[0] + tiling[2]
            if order.size == 0:      # tiles shared by clusters: key tiles of few keys, items of few branch rows
                assert dtype == "bf16" and (keys or not has_main), (stage, has_main)
                continue
            assert sorted(order) == list(range(tiles)), (stage, has_main)
            w = weights(p, keys, has_main, tiling)
            want = sorted(range(tiles), key=lambda i: (-w[i], i if keys else -i))      # (equal ones as without an order)
            assert order.tolist() == want, (stage, has_main)


def test_where_there_is_none(ba):
    one = W.Problem(np.array([0, 2000], np.int32), np.arange(2000, dtype=np.int32), W.uniform_branch_offsets(2000, 3), W.CHAIN, None, 8, 8, 128)
    plan = ba.Plan(one)
    for stage in (0, ba.STAGE_DQ, ba.STAGE_DKDV):
        assert tile_order(ba, plan, stage, True)[1].size == 0
    lib, x = ba._lib(), np.zeros(4, np.int64)
    assert lib.ba_plan_tile_order(None, 0, 1, x.ctypes.data, None, 0) == -1
    assert lib.ba_plan_tile_order(plan.handle, 1, 1, x.ctypes.data, None, 0) == -1
    assert lib.ba_plan_tile_order(plan.handle, 0, 1, x.ctypes.data, None, 5) == -1


def test_medium_batches_have_every_order(ba):
    """A batch that fills the SMs without clusters: forward, dQ and dK/dV all find theirs."""
    lens = [1500, 300, 2048, 77, 900]
    p = W.Problem(W.cu_from_lengths(lens), np.arange(sum(lens), dtype=np.int32), W.uniform_branch_offsets(sum(lens), 3), W.CHAIN, None,
                  8, 8, 128)
    for q in (p, W.Problem(p.cu_seqlens, p.anchor_idx, p.branch_offsets, W.CHAIN, None, 8, 8, 64)):
        plan = ba.Plan(q)
        for stage in (0, ba.STAGE_DQ, ba.STAGE_DKDV):
            for has_main in (True, False):
                tiling, order = tile_order(ba, plan, stage, has_main)
                assert order.size == tiling[0] + tiling[2] > 0
