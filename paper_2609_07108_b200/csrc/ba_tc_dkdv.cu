// Tensor-core dK / dV (sm_100a, bf16, head_dim 128).
//
// Key-stationary: a CTA keeps 128 key rows of one KV head (K_j, V_j) in shared memory and their gradients (fp32) in
// TMEM, and walks the query rows that can see them -- every query head of the KV head -- as 128-row tiles.
// Everything is transposed so that the key is the TMEM lane:
//   S^T  = K_j Q^T,  dP^T = V_j dO^T                    (128 keys x 128 rows)
//   P^T  = exp2(scale_log2 S^T - lse2[col])             -> TMEM, bf16, over S^T
//   dS^T = P^T o (dP^T - delta[col])                    -> TMEM, bf16, over dP^T
//   dV_j += P^T dO,  dK_j += dS^T Q
// TMEM: dK [0,128) dV [128,256) S^T / P^T [256,384) X = dP^T / dS^T [384,512).
// Warps 0-3 / 4-7 work on query rows [0,64) / [64,128) of every tile: A(t) P^T from S^T, kept in registers as fp32,
// then B(t) dS^T from dP^T.  One thread issues, after A(t): dV(t), S(t+1); after B(t): dK(t), dP(t+1), so the tensor
// core has two contractions to do behind either phase of the warps.
//
// Bound: 2,870 clocks per tile (A 1,320, B 830, the rest handoffs: S(t+1) is there 1,400 clocks after A(t)) against
// 2,048 of MMA; in long runs the power cap (1,180 executed TFLOP/s; library GEMMs 1,438).  Measured against two 64-row
// tiles in flight, one warpgroup each, whose S and dP were N = 64 MMAs at 59 % of the rate and read K_j and V_j twice
// as often: 73,728 tokens with chains 47.3 -> 43.4 ms, 65,536 with trees 7.86 -> 7.41 ms, 32,768 with blocks 1.78 ->
// 1.70 ms (draft rows 448 -> 437 us), 2,048 with chains 124 -> 120 us.
//
// Key tiles of whole branches, clusters that share main key tiles, work fetching: as in ba_tc_bwd.cu.
#include "ba_tc_bwd.cuh"

using namespace sm100;

namespace {

constexpr int kThreads = 384;
constexpr int kRegsCompute = 208, kRegsIssue = 88, kRegsLaunch = 168;
static_assert(256 * kRegsCompute + 128 * kRegsIssue <= kThreads * kRegsLaunch, "register re-split exceeds what the CTA owns");
// the next index is asked for when the loads of the last but this many tiles go out (see the forward)
constexpr int kFetchLead = 2;

// What every role knows about one stationary tile.
struct KeyItem {
    int n_iter;                  // steps (head, streamed tile) of this CTA; -1: no more work
    int n_sub, n_sub_main;       // streamed tiles per head: main part, then branch part
    int s_beg, hh_beg;           // first step: streamed tile and head
    int half;                    // bit 0 / 1: the last tile of the main / branch part holds at most 64 rows
    int is_main, g;
    int row0, row_end;           // keys in the numbering of their part
    int krow0;                   // first key in the key tensors
    int m0, m1, b0, b1;          // streamed rows: main part and branch part
    int ma, ba;                  // first rows of the two parts' tiles
};

constexpr int kQStages = 3, kGoStages = 2;

struct DkdvSmem {
    alignas(1024) uint8_t k[kTileBytes];
    alignas(1024) uint8_t v[kTileBytes];
    alignas(1024) uint8_t q[kQStages][kTileBytes];
    alignas(1024) uint8_t go[kGoStages][kTileBytes];
    alignas(16) float neg_lse2[2][kTile];
    alignas(16) float delta[2][kTile];
    alignas(16) uint4 clc[2];
    KeyItem item[2];
    alignas(8) uint64_t kv_full, kv_empty;
    uint64_t q_full[kQStages], q_empty[kQStages], go_full[kGoStages], go_empty[kGoStages], sc_full[2], sc_empty[2];
    uint64_t s_full, a_done, dp_full, b_done, acc_full, acc_free;
    uint64_t item_full[2], item_empty[2], clc_full[2], loads_out;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(DkdvSmem) <= 232448, "shared memory of the dK/dV kernel");

// the streamed tile of step s of a head: from the last one down, because the rows that see different key tiles of a
// sequence end together, so CTAs that start together share them through L2
__device__ __forceinline__ int walk(int n_sub, int s) { return n_sub - 1 - s; }

// Rows of one call are ordered by position (main) or anchor (branches), so the ranges of a tile are those of its
// first and last row.
__device__ void make_key_item(const TcBwdParams &p, const BaOrder &order, uint32_t work, int rank, KeyItem &it) {
    const int n = (int)p.meta.n_main, S = p.splits;
    int tile;
    // Heaviest first: earlier keys (more viewers)
    if (p.tile_major) {
        tile = order.n > 0 ? order.tile[work / p.h_kv] : (int)(work / p.h_kv);
        it.g = (int)(work % p.h_kv);
    } else {
        // KV-head-major: the CTAs running at one time belong to one or two KV heads and stream the same
        // query rows, so that stream is read from HBM about once per head instead of once per wave
        it.g = (int)(work / p.total_key_tiles);
        tile = (int)(work % p.total_key_tiles);
    }
    const bool is_main = tile < p.main_key_tiles;
    it.is_main = is_main;
    int bt = tile - p.main_key_tiles;
    if (!is_main && S > 1) bt = bt * S + rank;           // a cluster holds S branch key tiles
    const bool past = !is_main && bt >= p.branch_key_tiles;      // the last cluster has ranks to spare: no rows
    const int step = is_main ? kTile : p.step_kb;
    it.row0 = is_main ? (int)p.r.kv_begin + tile * step : (int)p.r.tok_begin + bt * step;
    it.row_end = past ? it.row0 : min(it.row0 + step, (int)(is_main ? p.r.kv_end : p.r.tok_end));
    it.krow0 = is_main ? it.row0 - (int)p.r.kv_base : n + it.row0;
    it.m0 = it.m1 = it.b0 = it.b1 = 0;
    const int first = it.row0, last = it.row_end - 1;
    if (last >= first) {
        if (is_main) {
            if (p.has_main_q) {
                it.m0 = max(first, (int)p.r.qm_begin);
                it.m1 = min(p.meta.key_qend[last], (int)p.r.qm_end);
            }
            it.b0 = p.meta.key_bq_begin[first];
            it.b1 = p.meta.key_bq_end[last];
            if (p.depth) { it.b0 /= p.branch_len; it.b1 /= p.branch_len; }    // token ranges -> branch ranges
        } else {
            it.b0 = p.meta.br_start[first];
            it.b1 = p.meta.br_end[last];
        }
        it.b0 = max(it.b0, (int)p.r.tok_begin);
        it.b1 = min(it.b1, (int)p.r.tok_end);
    }
    // The streamed tiles start at ma / ba: the parts' starts moved back (by < 4 rows) so that every tile's first row
    // is a multiple of 4 in the row numbering of the per-row scalars, whose bulk copies are then 16-byte aligned.
    // The extra leading rows are masked like any other invisible row.
    const int qbase = p.depth ? 0 : n;
    it.ma = it.m0 & ~3;
    it.ba = ((qbase + it.b0) & ~3) - qbase;   // may be as low as -3
    it.n_sub_main = it.m1 > it.m0 ? (it.m1 - it.ma + kTile - 1) / kTile : 0;
    const int n_sub_br = it.b1 > it.b0 ? (it.b1 - it.ba + kTile - 1) / kTile : 0;
    it.n_sub = it.n_sub_main + n_sub_br;
    it.half = (it.m1 - it.ma <= kTile * it.n_sub_main - 64 ? 1 : 0) | (it.b1 - it.ba <= kTile * n_sub_br - 64 ? 2 : 0);
    const int n_all = it.n_sub * p.group;
    const bool part = S > 1 && is_main;
    const int t_beg = part ? (int)((int64_t)n_all * rank / S) : 0;
    it.n_iter = (part ? (int)((int64_t)n_all * (rank + 1) / S) : n_all) - t_beg;
    it.s_beg = it.n_sub > 0 ? t_beg % it.n_sub : 0;
    it.hh_beg = it.n_sub > 0 ? t_beg / it.n_sub : 0;
}
// streamed tile u holds at most 64 rows
__device__ __forceinline__ bool is_half(int half, int n_sub, int n_sub_main, int u) {
    return (u == n_sub_main - 1 && (half & 1)) || (u == n_sub - 1 && u >= n_sub_main && (half & 2));
}

// Which of the rows r0 + [lo, hi] (columns lo .. hi of 64) of a branch see the key `rel` of that branch: bit `rel` of their
// masks.  Eight reads in flight, of the one word of a mask that holds the bit.
__device__ __forceinline__ uint64_t own_rows(const uint64_t *br_mask, int r0, int lo, int hi, int rel) {
    const uint32_t *word = reinterpret_cast<const uint32_t *>(br_mask) + 2 * (int64_t)r0 + (rel >> 5);
    uint32_t v[2] = {0u, 0u};
#pragma unroll
    for (int part = 0; part < 2; ++part) {
        const int last = min(hi, 32 * part + 31);
        for (int c = max(lo, 32 * part); c <= last; c += 8)      // (eight of short branches' rows too: no loop over a remainder)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (c + i <= last) v[part] |= ((word[2 * (c + i)] >> (rel & 31)) & 1u) << ((c + i) & 31);
    }
    return (uint64_t)v[1] << 32 | v[0];
}

// P of 32 columns (fp32 bits, in place of the scores) and its bf16 pairs
template <bool MASKED>
__device__ __forceinline__ void chunk_p(uint32_t (&x)[32], uint32_t mk, float sl2, const float *nl, uint32_t *pk) {
    const float2 s2 = make_float2(sl2, sl2);
    const float4 *nl4 = reinterpret_cast<const float4 *>(nl);
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        const float4 nv = nl4[e >> 2];
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
            const float2 y = ffma2(make_float2(__uint_as_float(x[e + c]), __uint_as_float(x[e + c + 1])), s2,
                                   c ? make_float2(nv.z, nv.w) : make_float2(nv.x, nv.y));
            float2 pp = make_float2(ex2(y.x), ex2(y.y));
            if (MASKED) {      // the scalars of invisible columns may be anything, even NaN
                pp.x = ((mk >> (e + c)) & 1u) ? pp.x : 0.f;
                pp.y = ((mk >> (e + c + 1)) & 1u) ? pp.y : 0.f;
            }
            x[e + c] = __float_as_uint(pp.x);
            x[e + c + 1] = __float_as_uint(pp.y);
            pk[(e + c) >> 1] = pack_bf16(pp.x, pp.y);
        }
    }
}

// dS = P o (dP - delta) of 32 columns as bf16 pairs
template <bool MASKED>
__device__ __forceinline__ void chunk_ds(const uint32_t (&r)[32], const uint32_t (&x)[32], uint32_t mk, const float *dl, uint32_t *pk) {
    const float4 *dl4 = reinterpret_cast<const float4 *>(dl);
    const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        const float4 dv = dl4[e >> 2];
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
            float2 d = fmul2(make_float2(__uint_as_float(x[e + c]), __uint_as_float(x[e + c + 1])),
                             ffma2(c ? make_float2(dv.z, dv.w) : make_float2(dv.x, dv.y), m1,
                                   make_float2(__uint_as_float(r[e + c]), __uint_as_float(r[e + c + 1]))));
            if (MASKED) {
                d.x = ((mk >> (e + c)) & 1u) ? d.x : 0.f;
                d.y = ((mk >> (e + c + 1)) & 1u) ? d.y : 0.f;
            }
            pk[(e + c) >> 1] = pack_bf16(d.x, d.y);
        }
    }
}

template <bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
tc_dkdv_kernel(const __grid_constant__ CUtensorMap tm_q_main, const __grid_constant__ CUtensorMap tm_q_branch,
               const __grid_constant__ CUtensorMap tm_go, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_go_branch,
               const __grid_constant__ TcBwdParams p, const __grid_constant__ BaOrder order) {
    using Smem = DkdvSmem;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &sm.abort_flag;
    if (smem_u32(smem_raw) & 1023u) {   // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicExch(p.status, BA_EUNSUPPORTED);
        return;
    }
    const int S = SPLIT ? p.splits : 1, rank = SPLIT ? (int)(blockIdx.x % S) : 0;
    // global row number of branch query 0 (rows of dO and of the per-row scalars): branch rows follow the main
    // rows, except in depth mode, where those tensors hold one row per branch
    const int qbase = p.depth ? 0 : (int)p.meta.n_main;

    if (tid == 0) {
        mbar_init(&sm.kv_full, 1); mbar_init(&sm.kv_empty, 1);
        for (int s = 0; s < kQStages; ++s) { mbar_init(&sm.q_full[s], 1); mbar_init(&sm.q_empty[s], 1); }
        for (int s = 0; s < kGoStages; ++s) { mbar_init(&sm.go_full[s], 1); mbar_init(&sm.go_empty[s], 1); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sm.sc_full[b], 1);
            mbar_init(&sm.sc_empty[b], 8);
            mbar_init(&sm.item_full[b], 1);
            mbar_init(&sm.item_empty[b], 10);   // producer, MMA thread, one lane of each P / dS warp
            mbar_init(&sm.clc_full[b], 1);
        }
        mbar_init(&sm.s_full, 1);
        mbar_init(&sm.a_done, 256);
        mbar_init(&sm.dp_full, 1);
        mbar_init(&sm.b_done, 256);
        mbar_init(&sm.loads_out, 1);
        mbar_init(&sm.acc_full, 1);
        mbar_init(&sm.acc_free, 256);
        sm.abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 8) {
        tmem_alloc(&sm.tmem_base, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    const uint32_t t_dk = tmem, t_dv = tmem + 128, t_s = tmem + 256, t_x = tmem + 384;
    bool shared_tile = false;      // SPLIT: this CTA walked a part of a main key tile

    if (warp >= 8) {
        reg_dec<kRegsIssue>();
        if (warp == 10) {
            // ================================================= work fetcher (whole warp, as in the forward; an item
            // without steps is finished here and never published)
            uint32_t work = SPLIT ? blockIdx.x / S : blockIdx.x;
            bool more = true;
            for (int n_item = 0, n_clc = 0;;) {
                const int s = n_item & 1, cs = n_clc & 1;
                bool ok = true;
                if (n_item >= 2) ok = mbar_wait(&sm.item_empty[s], ((n_item >> 1) - 1) & 1, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                if (!more) {
                    if (lane == 0) {
                        sm.item[s].n_iter = -1;
                        mbar_arrive(&sm.item_full[s]);
                    }
                    break;
                }
                if (lane == 0) make_key_item(p, order, work, rank, sm.item[s]);
                __syncwarp();
                if (!SPLIT && sm.item[s].n_iter == 0) {
                    const KeyItem &it = sm.item[s];
                    store_zero_rows<128>(p.dk, p.accumulate, it.krow0, it.row_end - it.row0, it.g, 1, p.h_kv, lane);
                    store_zero_rows<128>(p.dv, p.accumulate, it.krow0, it.row_end - it.row0, it.g, 1, p.h_kv, lane);
                } else {
                    if (lane == 0) mbar_arrive(&sm.item_full[s]);
                    if (!SPLIT) ok = mbar_wait(&sm.loads_out, n_item & 1, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    ++n_item;
                }
                if (SPLIT) {
                    more = false;
                } else {
                    if (lane == 0) {
                        fence_proxy_async();
                        mbar_expect_tx(&sm.clc_full[cs], 16);
                        clc_try_cancel(&sm.clc[cs], &sm.clc_full[cs]);
                    }
                    ok = mbar_wait(&sm.clc_full[cs], (n_clc >> 1) & 1, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) {
                        uint32_t spins = 0;      // leave no answer in flight
                        while (!mbar_try_wait(&sm.clc_full[cs], (n_clc >> 1) & 1) && ++spins < (1u << 22)) {}
                        break;
                    }
                    more = clc_answer(&sm.clc[cs], &work);
                    ++n_clc;
                }
                __syncwarp();
            }
        } else if (warp == 9) {
            // ================================================= copies (one thread)
            if (lane == 0) {
                bool ok = true;
                uint32_t n_q = 0, n_go = 0, n_sc = 0, n_kv = 0;      // Q, dO, scalar and stationary tiles loaded so far
                for (int n_item = 0; ok; ++n_item) {
                    const int sl = n_item & 1;
                    ok = mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag);
                    if (!ok) break;
                    const KeyItem it = sm.item[sl];
                    mbar_arrive(&sm.item_empty[sl]);
                    if (it.n_iter < 0) break;
                    if (it.n_iter == 0) continue;
                    struct Rows { bool main; int r0, gr0; };      // streamed tile u: part, first row, its row among all rows
                    auto rows_of = [&](int u) -> Rows {
                        Rows x;
                        x.main = u < it.n_sub_main;
                        x.r0 = x.main ? it.ma + u * kTile : it.ba + (u - it.n_sub_main) * kTile;
                        x.gr0 = x.main ? x.r0 : qbase + x.r0;
                        return x;
                    };
                    int hh = it.hh_beg, s = it.s_beg;  // step = hh * n_sub + s
                    // the query stream comes from HBM: ask for tile i + kPrefetch to be brought into L2 while tile i is loaded
                    constexpr int kPrefetch = 8;
                    int ph = hh, ps = s;
                    for (int i = 0; i < kPrefetch; ++i)
                        if (++ps == it.n_sub) { ps = 0; ++ph; }
                    for (int i = 0; i < it.n_iter; ++i) {
                        if (i == max(it.n_iter - 1 - kFetchLead, 0)) mbar_arrive(&sm.loads_out);
                        const int h = it.g * p.group + hh;
                        const Rows x = rows_of(walk(it.n_sub, s));
                        // a branch tile may start up to three rows before branch row 0: dO by the map that has no rows there
                        const CUtensorMap *tq = x.main ? &tm_q_main : &tm_q_branch, *tg = x.r0 >= 0 ? &tm_go : &tm_go_branch;
                        const int sq = n_q % kQStages, sg = n_go % kGoStages, sc = n_sc & 1;
                        if (n_q >= (uint32_t)kQStages && !(ok = mbar_wait(&sm.q_empty[sq], ((n_q / kQStages) - 1) & 1, abort_flag))) break;
                        mbar_expect_tx(&sm.q_full[sq], kTileBytes);
                        for (int half = 0; half < 2; ++half) tma_load_3d(sm.q[sq] + half * 16384, tq, half * 64, h, x.r0, &sm.q_full[sq]);
                        ++n_q;
                        if (i == 0) {
                            // the stationary pair, once the last S, dP of the item before have been formed
                            if (n_kv > 0 && !(ok = mbar_wait(&sm.kv_empty, (n_kv - 1) & 1, abort_flag))) break;
                            mbar_expect_tx(&sm.kv_full, 2 * kTileBytes);
                            for (int half = 0; half < 2; ++half) {
                                tma_load_3d(sm.k + half * 16384, &tm_k, half * 64, it.g, it.krow0, &sm.kv_full);
                                tma_load_3d(sm.v + half * 16384, &tm_v, half * 64, it.g, it.krow0, &sm.kv_full);
                            }
                            ++n_kv;
                        }
                        if (n_sc >= 2 && !(ok = mbar_wait(&sm.sc_empty[sc], ((n_sc >> 1) - 1) & 1, abort_flag))) break;
                        mbar_expect_tx(&sm.sc_full[sc], 2 * kTile * 4);
                        const size_t off = (size_t)h * p.row_pitch + x.gr0;
                        bulk_load(sm.neg_lse2[sc], p.nlse2_t + off, kTile * 4, &sm.sc_full[sc]);
                        bulk_load(sm.delta[sc], p.delta_t + off, kTile * 4, &sm.sc_full[sc]);
                        ++n_sc;
                        if (n_go >= (uint32_t)kGoStages && !(ok = mbar_wait(&sm.go_empty[sg], ((n_go / kGoStages) - 1) & 1, abort_flag))) break;
                        mbar_expect_tx(&sm.go_full[sg], kTileBytes);
                        for (int half = 0; half < 2; ++half)
                            tma_load_3d(sm.go[sg] + half * 16384, tg, half * 64, h, x.r0 >= 0 ? x.gr0 : x.r0, &sm.go_full[sg]);
                        ++n_go;
                        if (i + kPrefetch < it.n_iter) {
                            const int h2 = it.g * p.group + ph;
                            const Rows y = rows_of(walk(it.n_sub, ps));
                            const CUtensorMap *tq2 = y.main ? &tm_q_main : &tm_q_branch;
                            for (int half = 0; half < 2; ++half) {
                                tma_prefetch_3d(tq2, half * 64, h2, y.r0);
                                tma_prefetch_3d(&tm_go, half * 64, h2, y.gr0);
                            }
                            const size_t off2 = (size_t)h2 * p.row_pitch + y.gr0;
                            bulk_prefetch(p.nlse2_t + off2, kTile * 4);
                            bulk_prefetch(p.delta_t + off2, kTile * 4);
                        }
                        if (++ps == it.n_sub) { ps = 0; ++ph; }
                        if (++s == it.n_sub) { s = 0; ++hh; }
                    }
                }
                if (*abort_flag) {
                    // leave no copy in flight behind: wait (bounded) for what was issued
                    auto drain = [&](uint64_t *bars, uint32_t stages, uint32_t issued) {
                        for (uint32_t k = issued > stages ? issued - stages : 0; k < issued; ++k) {
                            uint32_t spins = 0;
                            while (!mbar_try_wait(&bars[k % stages], (k / stages) & 1) && ++spins < (1u << 22)) {}
                        }
                    };
                    drain(sm.q_full, kQStages, n_q);
                    drain(sm.go_full, kGoStages, n_go);
                    drain(sm.sc_full, 2, n_sc);
                    drain(&sm.kv_full, 1, n_kv);
                }
            }
        } else if (warp == 8) {
            // ================================================= MMA issuer (one elected thread)
            if (elect_one()) {
                constexpr uint32_t kStep = kTileBytes >> 4;
                // low descriptor words; tiles are 64-column halves of 16 KB
                const uint32_t k_km = smem_desc_lo(smem_u32(sm.k), 16), v_km = smem_desc_lo(smem_u32(sm.v), 16);
                const uint32_t q_km0 = smem_desc_lo(smem_u32(sm.q[0]), 16), q_mn0 = smem_desc_lo(smem_u32(sm.q[0]), 16384);
                const uint32_t go_km0 = smem_desc_lo(smem_u32(sm.go[0]), 16), go_mn0 = smem_desc_lo(smem_u32(sm.go[0]), 16384);
                constexpr uint32_t IDESC_ACC = idesc_bf16(128, 128, 1);    // 128 keys x 128, contraction over rows
                auto issue_t = [&](uint32_t d_tmem, uint32_t a_km, uint32_t b_km, bool half) {
                    const uint32_t idesc = half ? idesc_bf16(128, 64, 0) : idesc_bf16(128, 128, 0);
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        mma_ss_lh(d_tmem, a_km + desc_step_kmajor(ks), b_km + desc_step_kmajor(ks), idesc, ks > 0);
                };
                // A: bf16 pairs, rows [0,64) in columns [0,32) and rows [64,128) in columns [64,96)
                auto issue_acc = [&](uint32_t d_tmem, uint32_t a_tmem, uint32_t b_mn, bool half, bool accumulate) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_ts_lh(d_tmem, a_tmem + ks * 8, b_mn + desc_step_mnmajor(ks), IDESC_ACC, accumulate || ks > 0);
                    if (half) return;
#pragma unroll
                    for (int ks = 4; ks < 8; ++ks)
                        mma_ts_lh(d_tmem, a_tmem + 64 + (ks & 3) * 8, b_mn + desc_step_mnmajor(ks), IDESC_ACC, 1);
                };
                // The steps of successive items form one stream: the first S, dP of the next item are formed behind
                // the last accumulation of the current one.
                struct Step { bool valid, first, last, half; };
                int n_item = 0, left = 0, n_sub = 0, n_sub_main = 0, s = 0, half = 0;
                bool ok = true, done = false;
                auto advance = [&](Step &x) {
                    x.first = false;
                    while (left == 0 && !done) {
                        const int sl = n_item & 1;
                        ok = ok && mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag);
                        if (!ok) { done = true; break; }
                        const KeyItem &im = sm.item[sl];
                        left = im.n_iter; n_sub = im.n_sub; n_sub_main = im.n_sub_main; s = im.s_beg; half = im.half;
                        mbar_arrive(&sm.item_empty[sl]);
                        ++n_item;
                        x.first = true;
                        if (left < 0) { done = true; left = 0; }
                    }
                    x.valid = !done;
                    x.half = is_half(half, n_sub, n_sub_main, walk(n_sub, s));
                    if (++s == n_sub) s = 0;
                    --left;
                    x.last = left == 0;
                };
                uint32_t n_kv = 0, n_acc = 0;
                auto issue_s = [&](const Step &x, uint32_t t) {
                    ok = ok && mbar_wait(&sm.q_full[t % kQStages], (t / kQStages) & 1, abort_flag);
                    if (ok && x.first) ok = mbar_wait(&sm.kv_full, n_kv++ & 1, abort_flag);
                    if (!ok) return;
                    tc_fence_after();
                    issue_t(t_s, k_km, q_km0 + (t % kQStages) * kStep, x.half);
                    tc_commit(&sm.s_full);
                };
                auto issue_dp = [&](const Step &x, uint32_t t) {
                    ok = ok && mbar_wait(&sm.go_full[t % kGoStages], (t / kGoStages) & 1, abort_flag);
                    if (!ok) return;
                    tc_fence_after();
                    issue_t(t_x, v_km, go_km0 + (t % kGoStages) * kStep, x.half);
                    tc_commit(&sm.dp_full);
                    if (x.last) tc_commit(&sm.kv_empty);
                };
                Step cur, nxt;
                advance(cur);
                if (cur.valid && ok) { issue_s(cur, 0); issue_dp(cur, 0); }
                for (uint32_t t = 0; ok && cur.valid; ++t, cur = nxt) {
                    const uint32_t go_mn = go_mn0 + (t % kGoStages) * kStep, q_mn = q_mn0 + (t % kQStages) * kStep;
                    advance(nxt);
                    // the accumulators of the item before have been read out
                    if (ok && cur.first && n_acc > 0) ok = mbar_wait(&sm.acc_free, (n_acc - 1) & 1, abort_flag);
                    if (ok) ok = mbar_wait(&sm.a_done, t & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_acc(t_dv, t_s, go_mn, cur.half, !cur.first);                     // dV += P^T dO
                    tc_commit(&sm.go_empty[t % kGoStages]);
                    if (nxt.valid && !nxt.first) issue_s(nxt, t + 1);
                    if (ok) ok = mbar_wait(&sm.b_done, t & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_acc(t_dk, t_x, q_mn, cur.half, !cur.first);                      // dK += dS^T Q
                    tc_commit(&sm.q_empty[t % kQStages]);
                    if (cur.last) {
                        tc_commit(&sm.acc_full);
                        ++n_acc;
                    }
                    if (nxt.valid) {
                        if (nxt.first) issue_s(nxt, t + 1);      // other keys: their copy must not hold up the steps before
                        issue_dp(nxt, t + 1);
                    }
                }
            }
            __syncwarp();
        }
    } else {
        // ================================================= P / dS warps + epilogue
        reg_inc<kRegsCompute>();
        const int hf = warp >> 2;                       // my 64 rows of every streamed tile
        const int r_in = tid & 127;                     // my TMEM lane: key
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t s_addr = t_s + lane_base + 64 * hf, x_addr = t_x + lane_base + 64 * hf;
        const float sl2 = p.scale_log2;
        // what this role needs of an item, and this thread's key; the next item is read while the accumulators of
        // the current one are awaited
        struct Work {
            int n_iter, n_sub, n_sub_main, s_beg, half, g, row_end, krow, m0, m1, b0, b1, ma, ba, row;
            bool is_main, valid;
            int qend, rb0, rb1;          // main rows [row, qend) and branch rows [rb0, rb1) see my key
            // Branch key: which of my rows of streamed tiles 0 and 1 see it, (rb0, rb1) and (qend, m0), and whether the first
            // row of tile 2 does, m1 (its only one: see fetch).  In fields that only main keys need otherwise: with fields of
            // their own the steps of every item got 1 % slower.
        } w, nx;
        auto fetch = [&](int n_item, Work &f) -> bool {
            const int sl = n_item & 1;
            if (!mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag)) return false;
            const KeyItem &im = sm.item[sl];
            f.n_iter = im.n_iter; f.n_sub = im.n_sub; f.n_sub_main = im.n_sub_main; f.s_beg = im.s_beg; f.half = im.half; f.g = im.g;
            f.row_end = im.row_end; f.krow = im.krow0 + r_in;
            f.m0 = im.m0; f.m1 = im.m1; f.b0 = im.b0; f.b1 = im.b1; f.ma = im.ma; f.ba = im.ba;
            f.is_main = im.is_main;
            f.row = im.row0 + r_in;
            f.valid = f.row < f.row_end;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.item_empty[sl]);
            f.qend = f.rb0 = f.rb1 = 0;
            if (f.n_iter > 0 && f.valid) {
                if (f.is_main) {
                    f.qend = p.meta.key_qend[f.row];
                    f.rb0 = p.meta.key_bq_begin[f.row];
                    f.rb1 = p.meta.key_bq_end[f.row];
                    if (p.depth) { f.rb0 /= p.branch_len; f.rb1 /= p.branch_len; }
                } else {
                    const int start = p.meta.br_start[f.row], rbeg = max(start, f.b0), rend = min(p.meta.br_end[f.row], f.b1);
                    // which of my 64 rows from r0 see my key
                    auto own = [&](int r0) { return own_rows(p.meta.br_mask, r0, max(rbeg - r0, 0), min(rend - 1 - r0, 63), f.row - start); };
                    // Once for every head, and for most items while the item before ends (32/8 heads, 16,384 tokens, draft
                    // rows of 256 trees of 48: dK/dV 484 us; found at every step, one row after the other, 625; blocks of 24
                    // on 2,400 tokens 29 and 48).  The 128 keys' branches have at most 63 more rows on either side and the
                    // tiles start at most 3 rows early: 257 rows.
                    const uint64_t own0 = own(f.ba + 64 * hf), own1 = own(f.ba + kTile + 64 * hf);
                    f.rb0 = (int)(uint32_t)own0; f.rb1 = (int)(uint32_t)(own0 >> 32);
                    f.qend = (int)(uint32_t)own1; f.m0 = (int)(uint32_t)(own1 >> 32);
                    f.m1 = hf == 0 && own(f.ba + 2 * kTile) != 0ull;
                }
            }
            return true;
        };
        uint32_t t = 0, n_acc = 0;      // steps and accumulations so far
        bool ok = fetch(0, nx);
        for (int n_item = 0; ok; ++n_item) {
            w = nx;
            if (w.n_iter < 0) break;
            int s = w.s_beg;
            for (int i = 0; i < w.n_iter; ++i, ++t) {
                const int u = walk(w.n_sub, s), sc = t & 1;
                if (++s == w.n_sub) s = 0;
                const bool seg_main = u < w.n_sub_main;
                const int r0 = (seg_main ? w.ma + u * kTile : w.ba + (u - w.n_sub_main) * kTile) + 64 * hf;   // my first row
                const bool idle = hf && is_half(w.half, w.n_sub, w.n_sub_main, u);      // my rows are not there
                // --- which of my 64 rows (columns) see my key
                uint64_t vis = 0ull;
                if (w.valid && !idle) {
                    const int rbeg = seg_main ? w.m0 : w.b0, rend = seg_main ? w.m1 : w.b1;
                    if (w.is_main) {
                        // main rows: same sequence, causal: key <= row < end of the key's sequence; branch tokens
                        // anchored at or after the key, inside its sequence (depth mode: branches)
                        const int v0 = seg_main ? w.row : w.rb0, v1 = seg_main ? w.qend : w.rb1;
                        vis = bit_range(max(v0, rbeg) - r0, min(v1, rend) - 1 - r0);
                    } else {
                        vis = u < 2 ? (uint64_t)(uint32_t)(u ? w.m0 : w.rb1) << 32 | (uint32_t)(u ? w.qend : w.rb0) : (uint64_t)w.m1;
                    }
                }
                const bool masked = !__all_sync(0xffffffffu, vis == ~0ull);
                const uint32_t mk0 = (uint32_t)vis, mk1 = (uint32_t)(vis >> 32);
                const float *nl = sm.neg_lse2[sc] + 64 * hf, *dl = sm.delta[sc] + 64 * hf;
                ok = mbar_wait(&sm.sc_full[sc], (t >> 1) & 1, abort_flag);
                // --- phase A: P^T = exp2(scale_log2 S^T - lse2[col]) -> TMEM (bf16) and registers
                ok = ok && mbar_wait(&sm.s_full, t & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t xa[32], xb[32];       // P, fp32
                if (!idle) {
                    uint32_t pk[32];
                    tmem_ld32(s_addr, xa);
                    tmem_ld32(s_addr + 32, xb);
                    tmem_wait_ld();
                    if (masked) {
                        chunk_p<true>(xa, mk0, sl2, nl, pk);
                        chunk_p<true>(xb, mk1, sl2, nl + 32, pk + 16);
                    } else {
                        chunk_p<false>(xa, 0u, sl2, nl, pk);
                        chunk_p<false>(xb, 0u, sl2, nl + 32, pk + 16);
                    }
                    tmem_st32(s_addr, pk);
                    tmem_wait_st();
                }
                tc_fence_before();
                mbar_arrive(&sm.a_done);
                // --- phase B: dS^T = P^T o (dP^T - delta[col]) -> TMEM (bf16)
                ok = mbar_wait(&sm.dp_full, t & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (!idle) {
                    uint32_t ra[32], rb[32], pk[32];
                    tmem_ld32(x_addr, ra);
                    tmem_ld32(x_addr + 32, rb);
                    tmem_wait_ld();
                    if (masked) {
                        chunk_ds<true>(ra, xa, mk0, dl, pk);
                        chunk_ds<true>(rb, xb, mk1, dl + 32, pk + 16);
                    } else {
                        chunk_ds<false>(ra, xa, 0u, dl, pk);
                        chunk_ds<false>(rb, xb, 0u, dl + 32, pk + 16);
                    }
                    tmem_st32(x_addr, pk);
                    tmem_wait_st();
                }
                tc_fence_before();
                mbar_arrive(&sm.b_done);
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.sc_empty[sc]);
            }
            if (!ok) break;
            if (!SPLIT && !(ok = fetch(n_item + 1, nx))) break;
            // --- epilogue: warpgroup 0 takes dK (x scale), warpgroup 1 dV
            const bool any = w.n_iter > 0;
            if (any) {
                if (!(ok = mbar_wait(&sm.acc_full, n_acc & 1, abort_flag))) break;
                ++n_acc;
                tc_fence_after();
            }
            const uint32_t acc_addr = tmem + lane_base + hf * 128;
            shared_tile = SPLIT && w.is_main;
            void *dst = hf == 0 ? p.dk : p.dv;
            const float mul = hf == 0 ? p.scale : 1.0f;
            const size_t base = ((size_t)w.krow * p.h_kv + w.g) * 128;
            // my part, unscaled, over the streamed stages (acc_full covers every MMA of this CTA, and with them
            // every copy into the stages)
            float4 *part = reinterpret_cast<float4 *>(sm.q[0]) + (size_t)(hf * kTile + r_in) * 32;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                uint32_t r[32];
                if (any) {
                    tmem_ld32(acc_addr + c * 32, r);
                    tmem_wait_ld();
                    if (c == 3) {
                        tc_fence_before();
                        mbar_arrive(&sm.acc_free);       // the next item may accumulate
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) r[e] = 0u;
                }
                if (shared_tile) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)      // 16-byte chunks swizzled by the row: no bank conflicts
                        part[(8 * c + e) ^ (r_in & 31)] =
                            make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]), __uint_as_float(r[4 * e + 2]),
                                        __uint_as_float(r[4 * e + 3]));
                } else if (w.valid) {
                    if (p.accumulate) store_grad_chunk<true>(dst, base + c * 32, r, mul);
                    else store_grad_chunk<false>(dst, base + c * 32, r, mul, p.wide);
                }
            }
            if (SPLIT) break;
        }
    }

    if (SPLIT) {
        // ---- sum the parts: rank r finishes keys [128 r / S, 128 (r + 1) / S) of dK and dV, in rank order
        __syncwarp();
        cluster_sync_all();
        if (warp < 8 && shared_tile && !*abort_flag) {
            const KeyItem &it = sm.item[0];
            const int rows_mine = kTile / S;
            for (int idx = tid; idx < 2 * rows_mine * 32; idx += 256) {
                const int ch = idx & 31, rr = idx >> 5;
                const int which = rr / rows_mine, r = rank * rows_mine + rr % rows_mine;    // dK / dV
                if (it.row0 + r >= it.row_end) continue;
                const uint32_t src = smem_u32(sm.q[0]) + (uint32_t)(((which * kTile + r) * 32 + (ch ^ (r & 31))) * 16);
                float4 y[8];       // all parts in flight at once
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < S) y[q] = cluster_ld_f4(cluster_map(src, q));
                float4 x = y[0];
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    if (q < S) { x.x += y[q].x; x.y += y[q].y; x.z += y[q].z; x.w += y[q].w; }
                const float mul = which == 0 ? p.scale : 1.0f;
                x.x *= mul; x.y *= mul; x.z *= mul; x.w *= mul;
                void *dst = which == 0 ? p.dk : p.dv;
                const size_t off = ((size_t)(it.krow0 + r) * p.h_kv + it.g) * 128 + ch * 4;
                if (p.accumulate) {
                    float4 *d4 = reinterpret_cast<float4 *>((float *)dst + off);
                    const float4 o = *d4;
                    *d4 = make_float4(o.x + x.x, o.y + x.y, o.z + x.z, o.w + x.w);
                } else {
                    *reinterpret_cast<uint2 *>((__nv_bfloat16 *)dst + off) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
                }
            }
        }
        __syncwarp();
        cluster_sync_all();      // no CTA leaves while another may still read its shared memory
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
    wait_prerequisites();      // never done before the dQ kernel that it may overlap
    if (tid == 0 && sm.abort_flag) atomicExch(p.status, BA_ETIMEOUT);
}

// Step-major calls: dK, dV of the own-branch keys.  Token (depth j + 1, branch b) is seen by one query row of the call,
// that of branch b: a term per query head of the group, no contraction over rows.  Sixteen lanes per (branch, KV head),
// 8 of the 128 columns each; P and dS in fp32.
// Bound by memory: Q and dO once, K, V and the fp32 dK, dV of every depth <= depth once.  So everything a lane reads
// of one depth, and Q and dO of four heads, are in flight together (with the heads one after another 280 / 436 / 578 us).
// 18,432 branches, 32/8 heads, depth 1 / 2 / 3: 123 / 185 / 254 us (158 registers and one block per SM: 141 / 227 / 307); as key tiles of the kernel above, 128 keys against 128 rows
// of which each sees one, 155 / 329 / 464 us.
constexpr int kOwnThreads = 256, kOwnHeads = 4;
__device__ __forceinline__ float bf16_at(const uint4 &x, int e) {      // element e of eight
    const uint32_t w = e < 2 ? x.x : e < 4 ? x.y : e < 6 ? x.z : x.w;
    return __uint_as_float((e & 1) ? w & 0xffff0000u : w << 16);
}
__global__ void __launch_bounds__(kOwnThreads, 2) own_branch_kernel(const uint4 *__restrict__ q, const uint4 *__restrict__ go,
                                                                  const uint4 *__restrict__ k, const uint4 *__restrict__ v,
                                                                  const TcBwdParams p) {
    const int64_t unit = ((int64_t)blockIdx.x * kOwnThreads + threadIdx.x) / 16, units = (p.r.tok_end - p.r.tok_begin) * p.h_kv;
    const int sub = threadIdx.x & 15;
    const bool live = unit < units;      // (whole warps go through the shuffles)
    const int64_t b = p.r.tok_begin + (live ? unit / p.h_kv : 0);
    const int g = live ? (int)(unit % p.h_kv) : 0;
    for (int h0 = g * p.group; h0 < (g + 1) * p.group; h0 += kOwnHeads) {
        const int heads = min(kOwnHeads, (g + 1) * p.group - h0);
        uint4 qq[kOwnHeads], gg[kOwnHeads];
        float nl[kOwnHeads], dl[kOwnHeads];
#pragma unroll
        for (int i = 0; i < kOwnHeads; ++i) {
            const int h = h0 + min(i, heads - 1);
            qq[i] = q[((size_t)b * p.h_q + h) * 16 + sub];
            gg[i] = go[((size_t)b * p.h_q + h) * 16 + sub];
            nl[i] = i < heads ? p.nlse2_t[(size_t)h * p.row_pitch + b] : -INFINITY;      // no head: P = 0
            dl[i] = p.delta_t[(size_t)h * p.row_pitch + b];
        }
        for (int j = 0; j < p.depth; ++j) {
            const size_t krow = ((size_t)(p.meta.n_main + (int64_t)j * p.num_branches + b) * p.h_kv + g) * 16 + sub;
            const uint4 kk = k[krow], vv = v[krow];
            float4 *ak = reinterpret_cast<float4 *>(p.dk) + 2 * krow, *av = reinterpret_cast<float4 *>(p.dv) + 2 * krow;
            const float4 k0 = ak[0], k1 = ak[1], v0 = av[0], v1 = av[1];
            float s[kOwnHeads], dp[kOwnHeads], dk[8], dv[8];
#pragma unroll
            for (int i = 0; i < kOwnHeads; ++i) {
                s[i] = dp[i] = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    s[i] = fmaf(bf16_at(qq[i], e), bf16_at(kk, e), s[i]);
                    dp[i] = fmaf(bf16_at(gg[i], e), bf16_at(vv, e), dp[i]);
                }
            }
#pragma unroll
            for (int off = 8; off; off >>= 1)
#pragma unroll
                for (int i = 0; i < kOwnHeads; ++i) {
                    s[i] += __shfl_xor_sync(0xffffffffu, s[i], off);
                    dp[i] += __shfl_xor_sync(0xffffffffu, dp[i], off);
                }
#pragma unroll
            for (int e = 0; e < 8; ++e) dk[e] = dv[e] = 0.f;
#pragma unroll
            for (int i = 0; i < kOwnHeads; ++i) {
                if (i >= heads) break;
                const float pr = ex2(fmaf(s[i], p.scale_log2, nl[i])), ds = pr * (dp[i] - dl[i]);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    dk[e] = fmaf(ds, bf16_at(qq[i], e), dk[e]);
                    dv[e] = fmaf(pr, bf16_at(gg[i], e), dv[e]);
                }
            }
            if (live) {
                const float sc = p.scale;
                ak[0] = make_float4(fmaf(sc, dk[0], k0.x), fmaf(sc, dk[1], k0.y), fmaf(sc, dk[2], k0.z), fmaf(sc, dk[3], k0.w));
                ak[1] = make_float4(fmaf(sc, dk[4], k1.x), fmaf(sc, dk[5], k1.y), fmaf(sc, dk[6], k1.z), fmaf(sc, dk[7], k1.w));
                av[0] = make_float4(v0.x + dv[0], v0.y + dv[1], v0.z + dv[2], v0.w + dv[3]);
                av[1] = make_float4(v1.x + dv[4], v1.y + dv[5], v1.z + dv[6], v1.w + dv[7]);
            }
        }
    }
}

template <bool SPLIT>
int prepare(int dev) {
    // the dynamic shared-memory limit is a per-device attribute of the kernel
    static bool attr_set[64] = {};
    if (attr_set[dev]) return BA_OK;
    // the register re-split hands out what a launch with kRegsLaunch registers per thread owns
    cudaFuncAttributes fa;
    BA_CUDA_CHECK(cudaFuncGetAttributes(&fa, tc_dkdv_kernel<SPLIT>));
    if (fa.numRegs * kThreads < 256 * kRegsCompute + 128 * kRegsIssue) return BA_EUNSUPPORTED;
    BA_CUDA_CHECK(cudaFuncSetAttribute(tc_dkdv_kernel<SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DkdvSmem)));
    attr_set[dev] = true;
    return BA_OK;
}

template <bool SPLIT>
int launch(const TcDkdvCall &c, bool after_dq, cudaStream_t st) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)c.grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sizeof(DkdvSmem);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    if (SPLIT) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)c.p.splits;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    if (after_dq) {     // start when every CTA of the dQ kernel queued just before has started or been taken over
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++cfg.numAttrs;
    }
    cfg.attrs = attr;
    const CUtensorMap *tm = c.tm;
    BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_dkdv_kernel<SPLIT>, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], c.p, *c.order));
    return ba_check_launch();
}

}  // namespace

int ba_tc_dkdv_prepare(TcDkdvCall &c, const TcBwdParams &call, const ba_plan *pl, const BaRange &r, const void *q_main,
                       const void *q_branch, const void *k, const void *v, const void *d_o, int dev) {
    c.p = call;
    c.p.wide = (((uintptr_t)call.dk | (uintptr_t)call.dv) & 31) == 0;
    c.grid = key_items(c.p, pl, r, q_main != nullptr);
    if (c.grid <= 0) return BA_OK;
    if (c.grid > INT_MAX) return BA_EUNSUPPORTED;
    if (!bwd_maps(c.tm, pl, r, q_main, q_branch, k, v, d_o, call.depth, kTile, 1, kTile)) return BA_EINVAL;
    c.order = &key_order(c.p, pl, q_main != nullptr);
    return c.p.splits > 1 ? prepare<true>(dev) : prepare<false>(dev);
}

int ba_tc_dkdv_launch(const TcDkdvCall &c, bool after_dq, cudaStream_t st) {
    if (c.grid <= 0) return BA_OK;
    return c.p.splits > 1 ? launch<true>(c, after_dq, st) : launch<false>(c, after_dq, st);
}

int ba_tc_own_branch(const TcBwdParams &p, const void *q, const void *k, const void *v, const void *d_o, cudaStream_t st) {
    const int64_t blocks = ((p.r.tok_end - p.r.tok_begin) * p.h_kv * 16 + kOwnThreads - 1) / kOwnThreads;
    if (blocks <= 0) return BA_OK;
    if (blocks > INT_MAX) return BA_EUNSUPPORTED;
    own_branch_kernel<<<(unsigned)blocks, kOwnThreads, 0, st>>>((const uint4 *)q, (const uint4 *)d_o, (const uint4 *)k, (const uint4 *)v, p);
    return ba_check_launch();
}
