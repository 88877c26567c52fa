"""Tensor-core backward (and the head_dim 64 forward) at the edges of its tiles: ragged sequence and branch
ends, head groups that do and do not fill a packed tile, and main key tiles shared by clusters of two, four
and eight CTAs, against the fp64 oracle with the gates of the other parity tests."""
import numpy as np
import pytest

from paper_2609_07108_b200 import workloads as W
from test_gpu_fused_bwd import check_fused
from test_gpu_parity import ba, check_full  # noqa: F401  (ba: module-scoped fixture)

pytestmark = pytest.mark.gpu


def problem(lens, anchors, blen, kind, h_q, h_kv, d):
    anchors = np.asarray(sorted(anchors), np.int32)
    parent = None
    if kind == W.TREE:
        rng = np.random.default_rng(blen)
        parent = np.concatenate([W.random_tree_parents(rng, blen, 6) for _ in anchors]).astype(np.int32)
    return W.Problem(W.cu_from_lengths(lens), anchors, W.uniform_branch_offsets(len(anchors), blen), kind, parent, h_q,
                     h_kv, d)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n", [33, 63, 64, 65, 127, 128, 129, 193, 257])
def test_sequence_lengths(ba, oracle, d, n):  # noqa: F811
    check_full(ba, oracle, problem([n], [0, n // 2, n - 1], 3, W.CHAIN, 4, 2, d), seed=n, std=0.5, impl=ba.IMPL_TC)


# dK/dV walk the viewers of a key tile in tiles of 128 rows from a row that is a multiple of 4; a last tile of at most 64
# rows is formed at half width.  A short sequence in front moves the start of the second one's tiles by up to three rows.
# (Few viewers per key: dQ and dK are held to the absolute bound, as below.)
@pytest.mark.parametrize("shift", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [61, 62, 64, 125, 127, 190, 193])
def test_query_row_tiles(ba, oracle, n, shift):  # noqa: F811
    p = problem([shift, n], [shift, shift + n // 3, shift + n - 1], 22, W.BLOCK, 3, 1, 128)
    check_full(ba, oracle, p, seed=n + shift, std=0.5, impl=ba.IMPL_TC, relative_grads=False)


# Trees are held to the absolute bound on dQ and dK.  The backward takes O in bf16, so delta = <dO, O> of a row
# is off by up to 2^-9 sum |dO O|, about 1e-3 here, and each viewer moves a dK row by up to 1e-3 P |q| scale (2e-5
# at P = 0.1, head_dim 64; 3e-6 at P = 1/40, head_dim 128) whatever the kernel; the dK of a tree's leaf has one
# viewer and can be smaller than that (7e-6 to 3e-4 seen; the plain-FMA kernels are off by the same).
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("h_q,h_kv", [(4, 1), (3, 1), (8, 1), (2, 2)])
@pytest.mark.parametrize("kind,blen", [(W.BLOCK, 16), (W.BLOCK, 50), (W.TREE, 33), (W.TREE, 64)])
@pytest.mark.parametrize("q_main", [True, False])
def test_groups_and_branches(ba, oracle, d, h_q, h_kv, kind, blen, q_main):  # noqa: F811
    p = problem([70, 230, 40], [0, 3, 69, 70, 200, 299, 300, 320, 339], blen, kind, h_q, h_kv, d)
    check_full(ba, oracle, p, seed=blen, std=0.5, impl=ba.IMPL_TC, q_main=q_main, relative_grads=kind != W.TREE)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,h_q", [(600, 1), (600, 2), (600, 4)])     # four, eight and eight parts
def test_key_tiles_shared_by_a_cluster(ba, oracle, d, n, h_q):  # noqa: F811
    check_full(ba, oracle, problem([n], np.arange(n), 3, W.CHAIN, h_q, 1, d), seed=h_q, std=0.5, impl=ba.IMPL_TC)


# Two parts of three key tiles; two parts of 88 key tiles, more CTAs than SMs.  dQ and dK are held to the absolute bound:
# the last token of a chain is a key with one viewer, whose delta is off by up to 1e-3 (see trees above), which moves an
# element of its dK row by up to 1e-3 P |q_e| scale, 1.1e-5 at P = 1/8, |q_e| = 1 and head_dim 128 (2.7e-6 seen, at 5 to 12 keys).
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,h_q,h_kv", [(300, 1, 1), (1300, 8, 8)])
def test_key_tiles_in_two_parts(ba, oracle, d, n, h_q, h_kv):  # noqa: F811
    check_full(ba, oracle, problem([n], np.arange(n), 3, W.CHAIN, h_q, h_kv, d), seed=n, std=0.5, impl=ba.IMPL_TC, relative_grads=False)


# dQ and dK are held to the absolute and rel-RMS bounds, for the reason given for trees above: the last token of a
# branch is a key with one viewer, so an error of up to 1e-3 in that row's delta moves its dK row by up to
# 1e-3 P |q| scale (3e-6 at P = 1/150, |q| = 0.5 sqrt(128); 1.8e-6 seen), whatever the size of the row.
@pytest.mark.parametrize("n,h_q", [(590, 1), (600, 2), (600, 4)])     # two, four and eight parts
@pytest.mark.parametrize("q_main", [True, False])
def test_one_kernel_backward_shared_by_a_cluster(ba, oracle, n, h_q, q_main):  # noqa: F811
    check_fused(ba, oracle, problem([n], np.arange(n), 4, W.CHAIN, h_q, 1, 128), seed=h_q, q_main=q_main,
                relative_grads=False)


# The per-row scalars are prepared in tiles of 4 rows and 64 heads.  Sequences this short have near one-hot softmax
# rows, so dQ and dK are held to the absolute bound only.
@pytest.mark.parametrize("n,h_q,d", [(1, 1, 64), (3, 65, 128), (5, 64, 64), (7, 130, 64), (9, 3, 128)])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_row_scalar_tiles(ba, oracle, n, h_q, d, dtype):  # noqa: F811
    p = W.Problem(W.cu_from_lengths([n]), np.array([0, n - 1], np.int32)[:n], W.uniform_branch_offsets(min(n, 2), 3),
                  W.CHAIN, None, h_q, h_q, d, dtype=dtype)
    check_full(ba, oracle, p, seed=n, std=0.5, relative_grads=False)
