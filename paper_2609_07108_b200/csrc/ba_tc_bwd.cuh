// Pieces shared by the tensor-core backward kernels (ba_tc_bwd.cu: split dQ and
// dK/dV kernels; ba_tc_bwd_fused.cu: one key-stationary kernel for all three).
#pragma once

#include <limits.h>
#include <string.h>

#include "ba_common.cuh"
#include "ba_exact.cuh"
#include "ba_sm100.cuh"
#include "ba_tc_items.cuh"

namespace {

constexpr uint32_t kTileBytes = 32768;   // 128 rows x 128 bf16
constexpr float kLog2e = 1.4426950408889634f;

// bits [lo, hi] of a 64-bit word (empty if lo > hi)
__device__ __forceinline__ uint64_t bit_range(int lo, int hi) {
    lo = max(lo, 0);
    hi = min(hi, 63);
    if (lo > hi) return 0ull;
    return (~0ull >> (63 - hi)) & (~0ull << lo);
}

}  // namespace

struct TcBwdParams {
    BaMeta meta;
    BaRange r;
    const float *nlse2_t, *delta_t;   // head-major [h_q, row_pitch]: -LSE log2(e), delta
    int64_t row_pitch;
    void *dq_main, *dq_branch, *dk, *dv;
    int h_q, h_kv, group;
    float scale, scale_log2;
    int accumulate, wide;             // wide: bf16 gradients are 32-byte aligned
    int has_main_q;
    int main_tiles, total_tiles;      // dQ kernel: query row tiles
    int hp, head_chunks, tok;         // dQ with packed heads: heads per tile, chunks of hp heads per group, tokens per tile
    int main_key_tiles, total_key_tiles;  // dK/dV and fused kernels: key tiles
    int branch_key_tiles, step_kb;    // dK/dV: branch key tiles; branch tokens per branch key tile
    int splits, tile_major;           // dK/dV: CTAs per main key tile (cluster size), order of the key tiles
    // Step-major (per-depth) call of the dK/dV kernel: depth > 0.  Query rows are the
    // depth-`depth` tokens of branches [r.tok_begin, r.tok_end) (branch indices), Q / dO / dQ and
    // the per-row scalars are indexed by branch, and branch keys are stored depth-major after the
    // main rows: token (depth j + 1, branch b) is key row N + j * num_branches + b.
    int depth, num_branches, branch_len;
    int *status;
    RowArgs rows;                     // head_dim 64: rows that are formed again one by one
};

namespace {

// Branch tokens per branch key tile.  Branches of one length: a tile that starts and ends with a branch is seen
// by its own tokens only (chains of three: 126 keys and 128 query rows instead of 128 and up to 135, which
// costs a second 128-row step per head, at head_dim 64 a third 64-row one), unless more than an eighth of the lanes would stay empty.
inline int branch_key_step(int len) {
    return len > 1 && 8 * (kTile / len * len) >= 7 * kTile ? kTile / len * len : kTile;
}

// one 32-column chunk of a gradient row: fp32 accumulate (dst += r * mul) or bf16 store (`wide`: the buffer
// is 32-byte aligned, whole sectors per lane)
template <bool ACC_F32>
__device__ __forceinline__ void store_grad_chunk(void *dst, size_t elem_off, const uint32_t (&r)[32], float mul, int wide = 0) {
    using sm100::pack_bf16;
    if (ACC_F32) {
        float4 *d4 = reinterpret_cast<float4 *>((float *)dst + elem_off);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float4 old = d4[i];
            old.x += __uint_as_float(r[4 * i]) * mul;
            old.y += __uint_as_float(r[4 * i + 1]) * mul;
            old.z += __uint_as_float(r[4 * i + 2]) * mul;
            old.w += __uint_as_float(r[4 * i + 3]) * mul;
            d4[i] = old;
        }
    } else {
        __nv_bfloat16 *d = (__nv_bfloat16 *)dst + elem_off;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[e] = pack_bf16(__uint_as_float(r[16 * i + 2 * e]) * mul, __uint_as_float(r[16 * i + 2 * e + 1]) * mul);
            if (wide) sm100::st_global_v8(d + 16 * i, v);
            else {
                reinterpret_cast<uint4 *>(d)[2 * i] = make_uint4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<uint4 *>(d)[2 * i + 1] = make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
    }
}

// One warp: gradient rows [row0, row0 + rows) x heads [h0, h0 + heads) that receive no term (bf16: zeros;
// accumulated: unchanged)
template <int D> __device__ void store_zero_rows(void *dst, int accumulate, int row0, int rows, int h0, int heads, int h_all, int lane) {
    if (accumulate) return;
    constexpr int kChunks = D / 8;        // 16 bytes each
    for (int idx = lane; idx < rows * heads * kChunks; idx += 32) {
        const int r = idx / kChunks;
        const int64_t o = (int64_t)(row0 + r / heads) * h_all + h0 + r % heads;
        reinterpret_cast<uint4 *>(dst)[o * kChunks + idx % kChunks] = make_uint4(0u, 0u, 0u, 0u);
    }
}

__device__ __forceinline__ uint32_t bf16_rest(float2 x, uint32_t hi) {    // x - hi as a bf16 pair
    return sm100::pack_bf16(x.x - __uint_as_float(hi << 16), x.y - __uint_as_float(hi & 0xffff0000u));
}

// What every backward kernel of a call needs
inline TcBwdParams bwd_params(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch, const void *k,
                              const void *v, const float *delta, const void *d_o, int accumulate, void *dq_main,
                              void *dq_branch, void *dk, void *dv, int depth) {
    const ba_problem_t &pr = pl->prob;
    TcBwdParams p;
    memset(&p, 0, sizeof p);
    p.meta = pl->meta;
    p.r = r;
    p.delta_t = delta;
    p.nlse2_t = delta + (size_t)pl->row_pitch * pr.h_q;
    p.row_pitch = pl->row_pitch;
    p.dq_main = dq_main; p.dq_branch = dq_branch; p.dk = dk; p.dv = dv;
    p.h_q = pr.h_q; p.h_kv = pr.h_kv;
    p.group = pr.h_q / pr.h_kv;
    p.scale = pl->scale;
    p.scale_log2 = pl->scale * kLog2e;
    p.accumulate = accumulate;
    p.wide = (((uintptr_t)dq_main | (uintptr_t)dq_branch | (uintptr_t)dk | (uintptr_t)dv) & 31) == 0;
    p.has_main_q = q_main != nullptr;
    p.status = pl->dev_status;
    p.splits = 1;
    p.rows.meta = pl->meta; p.rows.r = r;
    p.rows.q_main = q_main; p.rows.q_branch = q_branch; p.rows.k = k; p.rows.v = v; p.rows.d_o = d_o;
    p.rows.nlse2_t = p.nlse2_t; p.rows.delta_t = p.delta_t; p.rows.row_pitch = p.row_pitch;
    p.rows.h_q = p.h_q; p.rows.h_kv = p.h_kv; p.rows.group = p.group;
    p.rows.scale_log2 = p.scale_log2;
    // depth mode: key rows of depths <= depth only (later rows read as zero); Q, dO hold one row per branch
    p.depth = depth;
    p.num_branches = pr.num_branches;
    p.branch_len = pr.uniform_len;
    return p;
}

// rows of the key tensors that a call may read: without own-branch keys nothing beyond kv_end (a received shard ends there)
inline uint64_t key_rows(const ba_plan *pl, const BaRange &r, int depth) {
    const ba_problem_t &pr = pl->prob;
    return depth ? (uint64_t)(pr.n_main + (int64_t)depth * pr.num_branches)
           : (r.parts & BA_PART_BRANCH) ? (uint64_t)(pr.n_main + pr.n_branch) : (uint64_t)(r.kv_end > r.kv_base ? r.kv_end - r.kv_base : 1);
}

// Maps in the order q_main, q_branch, dO, K, V, branch rows of dO; boxes of `qr` query rows x `qh` heads and `kr` key rows
inline bool bwd_maps(CUtensorMap *tm, const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                     const void *k, const void *v, const void *d_o, int depth, uint32_t qr, uint32_t qh, uint32_t kr) {
    using sm100::make_tmap_rhd;
    const ba_problem_t &pr = pl->prob;
    const int D = pr.head_dim;
    const uint64_t go_rows = depth ? (uint64_t)pr.num_branches : (uint64_t)(pr.n_main + pr.n_branch);
    const void *qm = q_main ? q_main : q_branch;
    const void *qb = (q_branch && pr.n_branch > 0) ? q_branch : q_main;
    const uint64_t qm_rows = depth ? (uint64_t)pr.num_branches : q_main ? (uint64_t)pr.n_main : (uint64_t)pr.n_branch;
    const uint64_t qb_rows = depth ? (uint64_t)pr.num_branches
                             : (q_branch && pr.n_branch > 0) ? (uint64_t)pr.n_branch : (uint64_t)pr.n_main;
    // dO of the branch rows alone: whatever lies in front of branch row 0 (rows of dO that a call without main
    // queries leaves unset) is not loaded
    const bool go_split = !depth && pr.n_branch > 0;
    const void *gob = go_split ? (const char *)d_o + (size_t)pr.n_main * pr.h_q * D * 2 : d_o;
    const uint64_t gob_rows = go_split ? (uint64_t)pr.n_branch : go_rows, kv_rows = key_rows(pl, r, depth);
    return make_tmap_rhd(&tm[0], qm, qm_rows, pr.h_q, D, qr, qh) && make_tmap_rhd(&tm[1], qb, qb_rows, pr.h_q, D, qr, qh) &&
           make_tmap_rhd(&tm[2], d_o, go_rows, pr.h_q, D, qr, qh) && make_tmap_rhd(&tm[3], k, kv_rows, pr.h_kv, D, kr) &&
           make_tmap_rhd(&tm[4], v, kv_rows, pr.h_kv, D, kr) && make_tmap_rhd(&tm[5], gob, gob_rows, pr.h_q, D, qr, qh);
}

// Work items (key tiles) of dK/dV and how they are shared out; returns the number of CTAs
inline int64_t key_items(TcBwdParams &p, const ba_plan *pl, const BaRange &r, bool has_main) {
    const ba_problem_t &pr = pl->prob;
    const int64_t qm_n = has_main ? r.qm_end - r.qm_begin : 0, br_n = r.tok_end - r.tok_begin;
    const int64_t kmt = (r.parts & BA_PART_MAIN) ? (r.kv_end - r.kv_begin + kTile - 1) / kTile : 0;
    p.step_kb = branch_key_step(pr.uniform_len);
    // (step-major: own_branch_kernel)
    const int64_t kbt = (r.parts & BA_PART_BRANCH) && !p.depth ? (br_n + p.step_kb - 1) / p.step_kb : 0;
    p.branch_key_tiles = (int)kbt;
    // Share main key tiles between the CTAs of a cluster while the CTAs are few and a part keeps enough steps (64 streamed
    // rows, by the mean sequence length): ever more of them the more CTAs there are already, because a part costs its
    // set-up and the sum at the end.  Twice as many parts against as many as before, mean / worst of 493 batches (one to
    // sixteen sequences, chains and blocks, five head counts; the same at head_dim 64): up to half a CTA per SM with 3 to 4
    // steps 0.77 / 1.00; up to one with 6 to 8 0.82 / 1.00 (4 to 6: 0.89 / 1.10); up to 1.5 with 8 to 12 0.78 / 0.98 (6 to 8:
    // 0.98 / 1.04); up to 2.5 with 24 to 32 0.76 / 0.96 (16 to 24: 0.88 / 1.24); up to three with 64 0.79 / 0.96 (48 to 64:
    // 0.88 / 1.12); beyond that 1.12 / 1.15 and more.
    const int64_t keys = kmt * kTile, viewers = qm_n + br_n;
    const int64_t seq = pr.num_seqs > 0 ? pr.n_main / pr.num_seqs : 0;
    const int64_t est = keys > 0 ? (seq < keys ? seq : keys) / 2 * viewers / (keys < pr.n_main ? pr.n_main : keys) * p.group / 64 : 0;
    auto worth = [&](int64_t splits) {
        const int64_t halves = (kmt * pr.h_kv * splits * 2 + kSms - 1) / kSms;      // CTAs per SM, in halves
        const int steps = halves <= 1 ? 3 : halves <= 2 ? 6 : halves <= 3 ? 8 : halves <= 5 ? 24 : 64;
        return halves <= 6 && est >= steps * splits;
    };
    while (p.splits < 8 && worth(2 * p.splits)) p.splits *= 2;
    p.main_key_tiles = (int)kmt;
    const int64_t tiles = kmt + (kbt + p.splits - 1) / p.splits;    // work items (clusters) per KV head
    p.total_key_tiles = (int)tiles;
    // Up to 96 work items per SM heaviest first over all KV heads, so that the last items are short; beyond that
    // KV-head-major, whose resident CTAs share one query stream through L2.  KV-head-major against tile-major, chains, blocks
    // and trees, 32/8, 16/4 and 8/8 heads, 1 to 12 sequences: 1.05 to 1.48 times the time at 10 to 14 items per SM, 1.00 to
    // 1.24 at 24, 0.99 to 1.16 at 48, 1.00 to 1.06 at 90, 0.98 to 1.07 at 124.
    p.tile_major = tiles * pr.h_kv <= 96 * kSms;
    return tiles * pr.h_kv * p.splits;
}

inline BaTiling key_tiling(const TcBwdParams &p, bool has_main) {
    return {BA_ORDER_KEYS, has_main, p.main_key_tiles, kTile, p.total_key_tiles - p.main_key_tiles, p.step_kb};
}
inline const BaOrder &key_order(const TcBwdParams &p, const ba_plan *pl, bool has_main) {
    const bool any = !p.depth && p.splits == 1 && p.tile_major && ba_whole_call(pl, p.r, has_main);
    return ba_find_order(pl, any ? key_tiling(p, has_main) : BaTiling{-1});
}

}  // namespace

// dK / dV of a call at head_dim 128 (ba_tc_dkdv.cu): all that can be refused, then the launch; after_dq: it may start
// while the dQ kernel queued just before ends
struct TcDkdvCall {
    TcBwdParams p;
    CUtensorMap tm[6];
    int64_t grid;
    const BaOrder *order;
};
int ba_tc_dkdv_prepare(TcDkdvCall &c, const TcBwdParams &call, const ba_plan *pl, const BaRange &r, const void *q_main,
                       const void *q_branch, const void *k, const void *v, const void *d_o, int dev);
int ba_tc_dkdv_launch(const TcDkdvCall &c, bool after_dq, cudaStream_t st);
// step-major calls: dK / dV of the own-branch keys alone
int ba_tc_own_branch(const TcBwdParams &p, const void *q, const void *k, const void *v, const void *d_o, cudaStream_t st);
