// Work items of the query-stationary tensor-core kernels (forward, dQ): which query rows, which key tiles.
// The tile geometry is described at the head of ba_tc_fwd.cu.
#pragma once

#include <limits.h>

#include "ba_common.cuh"

namespace {

constexpr int kTile = 128;

// Call and item geometry shared by the query-stationary kernels.
struct ItemParams {
    BaMeta meta;
    BaRange r;
    int h_q, h_kv, group;
    int hp, head_chunks;         // heads per query tile; chunks of hp heads per group
    int tok;                     // tokens per query tile (128 / hp)
    int step_m, step_b, off_b;   // tokens per item (main, branch) and first token of tile 1 (branch)
    int main_items, total_items; // row ranges (times h_kv * head_chunks work items)
    int splits;
    int same_rows;               // both query tiles hold the same rows: tile i takes the key tiles of parity i
    // Step-major (per-depth) call: depth > 0.  The query rows are the depth-`depth` tokens of
    // branches [tok_begin, tok_end) (r.tok_* hold BRANCH indices then), the query tensor and the
    // outputs are indexed by branch, and the branch keys are stored depth-major after the main
    // rows: token (depth j + 1, branch b) is key row N + j * num_branches + b.
    int depth, num_branches, branch_len;
};

// What every role knows about one work item (one query row range, one KV head).
struct Item {
    int T;                   // key tiles; -1: no more work
    int jb, je;              // the tiles [jb, je) this CTA handles
    int is_main, g, h0, row0, rows;
    int lo_min, n_full;      // full tile j holds main keys lo_min + 128 j ...
    int tail_k, n_mc, n_ch;  // tail chunks of 32 keys: n_mc from main key tail_k, the rest own-branch keys
    int bs;                  // first own-branch key (token index)
    // query tile i: some row sees full tiles [va, vb), every row sees the whole of full tiles [wa, wb);
    // tail tiles are always visited (if the query tile holds rows)
    int live[2], va[2], vb[2], wa[2], wb[2];
};

// bits [lo, hi] of a 32-bit word (empty if lo > hi)
__device__ __forceinline__ uint32_t bits32(int lo, int hi) {
    lo = max(lo, 0);
    hi = min(hi, 31);
    return lo > hi ? 0u : (~0u >> (31 - hi)) & (~0u << lo);
}

// first token of query tile 1, tokens of query tile i
__device__ __forceinline__ int tile1_off(const ItemParams &p, bool is_main) { return p.same_rows ? 0 : is_main ? p.tok : p.off_b; }
__device__ __forceinline__ int tile_tokens(const ItemParams &p, bool is_main, int i, int rows) {
    const int off1 = tile1_off(p, is_main);
    return p.same_rows ? rows : min(i ? rows - off1 : min(off1, rows), p.tok);
}

__device__ __forceinline__ bool tile_live(const Item &it, int i, int j) {
    return it.live[i] && (j >= it.n_full || (j >= it.va[i] && j < it.vb[i]));
}

__device__ __forceinline__ int tile_chunks(const Item &it, int j) {
    return j < it.n_full ? 4 : min(4, it.n_ch - 4 * (j - it.n_full));
}

// main-key bounds of one query row, clipped to the call's key range (empty: hi < lo)
__device__ __forceinline__ void row_bounds(const ItemParams &p, bool is_main, int row, int &lo, int &hi) {
    const int64_t grow = is_main ? row : p.meta.n_main + (p.depth ? (int64_t)row * p.branch_len : row);
    lo = max(p.meta.row_lo[grow], (int)p.r.kv_begin);
    hi = min(p.meta.row_hi[grow], (int)p.r.kv_end - 1);
    if (!(p.r.parts & BA_PART_MAIN)) { lo = INT_MAX; hi = -1; }
}

// Rows of one call are ordered by position (main) or anchor (branches), so the bounds of a row range
// are those of its first and last row.
__device__ void make_item(const ItemParams &p, const BaOrder &order, uint32_t work, int rank, Item &it) {
    const int per = p.h_kv * p.head_chunks;
    // longest prefixes first (without an order: later rows first); the items of one row range (all KV heads) are adjacent
    const int tile = order.n > 0 ? order.tile[work / per] : p.total_items - 1 - (int)(work / per);
    const int inner = (int)(work % per);
    it.g = inner / p.head_chunks;
    it.h0 = it.g * p.group + (inner % p.head_chunks) * p.hp;
    const bool is_main = tile < p.main_items;
    it.is_main = is_main;
    const int step = is_main ? p.step_m : p.step_b, off1 = tile1_off(p, is_main);
    it.row0 = (int)(is_main ? p.r.qm_begin + (int64_t)tile * step : p.r.tok_begin + (int64_t)(tile - p.main_items) * step);
    const int row_end = (int)(is_main ? p.r.qm_end : p.r.tok_end);
    it.rows = min(step, row_end - it.row0);
    const int first[2] = {it.row0, it.row0 + off1};
    const int last[2] = {it.row0 + (p.same_rows ? it.rows : min(off1, it.rows)) - 1, it.row0 + it.rows - 1};
    int lo_min = INT_MAX, hi_max = -1, lo0[2], hi0[2], lo1[2], hi1[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        it.live[i] = first[i] <= last[i];
        lo0[i] = lo1[i] = INT_MAX; hi0[i] = hi1[i] = -1;
        if (!it.live[i]) continue;
        row_bounds(p, is_main, first[i], lo0[i], hi0[i]);
        row_bounds(p, is_main, last[i], lo1[i], hi1[i]);
        lo_min = min(lo_min, lo0[i]);
        hi_max = max(hi_max, hi1[i]);
    }
    const int keys = max(hi_max - lo_min + 1, 0);
    it.lo_min = keys ? lo_min : 0;
    it.n_full = keys / kTile;
    it.tail_k = it.lo_min + it.n_full * kTile;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        it.va[i] = it.vb[i] = it.wa[i] = it.wb[i] = 0;
        if (hi1[i] >= lo0[i]) {
            it.va[i] = (lo0[i] - it.lo_min) / kTile;
            it.vb[i] = min((hi1[i] - it.lo_min) / kTile + 1, it.n_full);
        }
        if (hi0[i] >= lo1[i]) {
            it.wa[i] = (lo1[i] - it.lo_min + kTile - 1) / kTile;
            it.wb[i] = min((hi0[i] - it.lo_min + 1) / kTile, it.n_full);
        }
    }
    it.n_mc = (keys % kTile + 31) / 32;
    it.n_ch = it.n_mc;
    it.bs = 0;
    if (!is_main && (p.r.parts & BA_PART_BRANCH)) {
        if (p.depth) {       // per depth, the tokens of this item's own branches in branch order
            it.n_ch += p.depth * ((it.rows + 31) / 32);
        } else {
            it.bs = p.meta.br_start[it.row0];
            it.n_ch += (p.meta.br_end[it.row0 + it.rows - 1] - it.bs + 31) / 32;
        }
    }
    it.T = it.n_full + (it.n_ch + 3) / 4;
    it.jb = (int)((int64_t)it.T * rank / p.splits);
    it.je = (int)((int64_t)it.T * (rank + 1) / p.splits);
}

// first row of full key tile j / of tail chunk c in the key tensors
__device__ __forceinline__ int full_row(const ItemParams &p, const Item &it, int j) { return it.lo_min - (int)p.r.kv_base + j * kTile; }
__device__ __forceinline__ int chunk_row(const ItemParams &p, const Item &it, int c) {
    if (c < it.n_mc) return it.tail_k - (int)p.r.kv_base + 32 * c;
    c -= it.n_mc;
    if (!p.depth) return (int)p.meta.n_main + it.bs + 32 * c;
    const int cpd = (it.rows + 31) / 32;
    return (int)p.meta.n_main + (c / cpd) * p.num_branches + it.row0 + 32 * (c % cpd);
}

// The 32 columns of chunk c of key tile j that a query row sees: main keys [lo, hi], and the tokens of its own
// branch in `mask` (bit u = token br_start + u; br_off = first own-branch key of the item - br_start); t_rel =
// the row's token within the item.
__device__ __forceinline__ uint32_t chunk_vis(const ItemParams &p, int j, int c, int n_full, int lo_min, int n_mc, int lo, int hi,
                                              int br_off, uint64_t mask, int t_rel, int rows) {
    const int k0 = lo_min + kTile * j + 32 * c;
    const int q = 4 * (j - n_full) + c;
    if (j < n_full || q < n_mc) return bits32(lo - k0, hi - k0);
    if (p.depth) {       // the token of the row's own branch at every depth <= depth
        const int b = t_rel - 32 * ((q - n_mc) % ((rows + 31) / 32));
        return bits32(b, b);
    }
    const int off = br_off + 32 * (q - n_mc);           // column t = bit t + off of the mask
    return off >= 0 ? (off < 64 ? (uint32_t)(mask >> off) : 0u) : off > -32 ? (uint32_t)(mask << -off) : 0u;
}

// Host: geometry of a call; returns the number of work items.
inline int64_t fill_items(ItemParams &p, const ba_plan *pl, const BaRange &r, bool has_main, int depth, bool same_rows_ok = false) {
    const ba_problem_t &pr = pl->prob;
    p.meta = pl->meta;
    p.r = r;
    p.h_q = pr.h_q;
    p.h_kv = pr.h_kv;
    p.group = pr.h_q / pr.h_kv;
    p.hp = p.group < kTile ? p.group : kTile;
    p.head_chunks = (p.group + p.hp - 1) / p.hp;
    p.tok = kTile / p.hp;
    p.depth = depth;
    p.num_branches = pr.num_branches;
    p.branch_len = pr.uniform_len;
    p.splits = 1;
    p.same_rows = 0;
    p.step_m = p.step_b = 2 * p.tok;
    p.off_b = p.tok;
    // Branches of one length: an item that starts and ends with a branch has no own-branch keys beyond
    // its own tokens (chains of three, 64 tokens per item: 63 tokens and 63 keys instead of 64 and up
    // to 68), unless more than an eighth of the rows would stay empty.  Where it costs no token, tile 1
    // starts with a branch too.
    const int len = depth ? 0 : pr.uniform_len;
    if (len > 1 && len <= p.step_b && 8 * (p.step_b / len * len) >= 7 * p.step_b) {
        p.step_b = p.step_b / len * len;
        if (len <= p.tok && 2 * (p.tok / len * len) == p.step_b) p.off_b = p.tok / len * len;
    }
    // Branch rows only, so few that two query tiles would belong to different sequences and never share a key tile:
    // one tile's worth of rows per item (one sequence's, for branches of one length), in both query tiles.
    if (same_rows_ok && !has_main && !depth && pr.num_seqs > 0 && r.tok_end - r.tok_begin <= (int64_t)pr.num_seqs * p.tok) {
        p.same_rows = 1;
        p.step_b = p.tok;
        const int per_seq = (pr.num_branches + pr.num_seqs - 1) / pr.num_seqs;
        if (len > 0 && len <= p.tok) p.step_b = (per_seq < p.tok / len ? per_seq : p.tok / len) * len;
    }
    const int64_t mt = has_main ? (r.qm_end - r.qm_begin + p.step_m - 1) / p.step_m : 0;
    const int64_t bt = (r.tok_end - r.tok_begin + p.step_b - 1) / p.step_b;
    p.main_items = (int)mt;
    p.total_items = (int)(mt + bt);
    return (mt + bt) * pr.h_kv * p.head_chunks;
}

inline BaTiling item_tiling(const ItemParams &p, bool has_main) {
    return {BA_ORDER_ROWS, has_main, p.main_items, p.step_m, p.total_items - p.main_items, p.step_b};
}
// (Items shared by clusters are few: taken longest first, trees at the ends of 8 sequences, 65,536 tokens, 32/8 heads,
// 88.4 -> 85.4 us, of 9 sequences, 29,883 tokens, 8/8 heads, 80.6 -> 83.7.)
inline const BaOrder &item_order(const ItemParams &p, const ba_plan *pl, bool has_main) {
    static const BaOrder none = {};
    return !p.depth && p.splits == 1 && ba_whole_call(pl, p.r, has_main) ? ba_find_order(pl, item_tiling(p, has_main)) : none;
}

}  // namespace
