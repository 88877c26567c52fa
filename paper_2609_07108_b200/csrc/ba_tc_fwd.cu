// Tensor-core forward (sm_100a, bf16, head_dim 64 or 128).
//
// One work item = two query tiles of 128 TMEM lanes.  A tile packs all query heads of one KV head
// (a row of the tile = one (token, head) pair, head fastest), so both tiles share every K / V tile
// whatever the group size, no lane is spent on a duplicated head, and an item spans few tokens: 64
// for four heads per KV head, hence a 64-token causal diagonal and 64 own-branch keys instead of 128.
// Both key sets of the paper's Section 3.2 (causal main prefix, own-branch keys) are walked in ONE
// online-softmax pass, which is Eq. (lse-merge) applied tile by tile.  The keys of an item are
//   full tiles   128 main keys each, from the first key any of its rows sees
//   tail         the rest of the main keys, then the own-branch keys, as 32-key chunks, up to four
//                chunks per tile: a tile costs the tensor core and the softmax only its chunks
// A query tile skips key tiles that none of its rows sees; tiles that all its rows see entirely take
// a mask-free path.
//
// Warp roles (384 threads, registers re-split with setmaxnreg):
//   warps 0-3 / 4-7  softmax of query tile 0 / 1: one thread per row, scores read from TMEM, P
//                    written back to TMEM as bf16 over the scores
//   warp 8           one thread issues tcgen05.mma: S_i = Q_i K^T, O_i += P_i V
//   warp 9           TMA producer: Q of the item, then K_j, V_j through a ring of stages
//   warp 10          fetches work: a CTA that is done takes over the index of one that has not
//                    started (cluster launch control), so set-up, Q loads and the first Q K^T of the
//                    next item run behind the softmax and the output stores of the current one
// TMEM (512 columns): S_0 [0,128) S_1 [128,256) O_0 [256,256+D) O_1 [384,384+D); P_i occupies the
// first 64 columns of S_i; head_dim 64: the 64 columns after O_i hold P_lo.
// head_dim 64 runs in place of a plain-FMA kernel that kept P in fp32.  P goes in as a bf16 pair hi + lo (16 bits of
// mantissa), two products each: against fp64, O rounded to bf16 is then off by what that kernel's is (1.5803e-3
// against 1.5803e-3 in the 2-norm).  O in fp32 would not be, so partial forwards stay with that kernel (ba_use_tc).
// 4,096 tokens, 6 sequences, chains of three, 32/8 heads: 173 us (was 2619).
//
// What bounds it: the chain scores -> maximum -> exponentials -> P -> P V, next Q K^T of each of the
// two tiles (about 2000 clocks of softmax and 1000 of MMA and handoffs per 128 x 128 tile), so the
// tensor pipe is busy a little over half of the time.  See the notes at the MMA issuer and the epilogue for
// what the seams between items cost.
//
// SPLIT variant (few rows, many keys): the CTAs of a cluster share one item, each takes a contiguous
// part of its key tiles, and the partial (O, max, sum) are combined through distributed shared memory.
// Where the two query tiles would hold branches of different sequences, and so never share a key tile, both
// hold the same rows instead and take alternate key tiles: two softmax chains in flight, not one.
#include <limits.h>
#include <string.h>

#include "ba_common.cuh"
#include "ba_exact.cuh"
#include "ba_sm100.cuh"
#include "ba_tc_items.cuh"

using namespace sm100;

namespace {

constexpr int kThreads = 384;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.0f;  // in log2 units: P stays below 2^8
// 128 score columns per thread stay in registers between the maximum and the exponentials
constexpr int kRegsSoftmax = 208, kRegsIssue = 88;
// the next index is asked for when the loads of the item's last but kFetchLead key tile go out
constexpr int kFetchLead = 1;
constexpr int kRegsLaunch = 168;           // what a launch of 384 threads owns per thread
static_assert(256 * kRegsSoftmax + 128 * kRegsIssue <= kThreads * kRegsLaunch, "register re-split exceeds what the CTA owns");

template <int D> struct FwdSmem {
    static constexpr int kStages = D == 128 ? 4 : 8;
    static constexpr uint32_t kTileBytes = kTile * D * 2;
    alignas(1024) uint8_t q[2][kTileBytes];
    alignas(1024) uint8_t kv[kStages][kTileBytes];
    alignas(1024) uint8_t out[8][4096];   // per softmax warp: 32 rows x 64 output columns on their way to memory
    alignas(16) uint4 clc[2];
    Item item[2];
    alignas(8) uint64_t q_full, q_empty;
    uint64_t kv_full[kStages], kv_empty[kStages];
    uint64_t s_full[2], p_half[2], p_full[2], o_full[2], o_free[2];
    uint64_t item_full[2], item_empty[2], clc_full[2], loads_out;
    uint32_t tmem_base;
    int abort_flag;
    // SPLIT: row maximum (log2 units) and sum of the two query tiles, in the idle output staging
    __device__ float2 *ml(int i) { return reinterpret_cast<float2 *>(out[0]) + i * kTile; }
};
static_assert(sizeof(FwdSmem<128>) <= 232448 && sizeof(FwdSmem<64>) <= 232448, "shared memory of the forward kernel");

struct TcFwdParams : ItemParams {
    void *o;
    float *lse;
    float scale_log2;
    int partial_out;
    int wide;                    // outputs are 32-byte aligned
    int warp_tok;                // > 0: a full warp of rows is this many tokens and leaves through a TMA store
    int *status;
    RowArgs rows;                // head_dim 64: rows that are formed again one by one
};


// 32 values of a row -> output (bf16 or fp32), 32-byte stores where the buffer allows
template <bool OUT_F32>
__device__ __forceinline__ void store_row_chunk(void *o, size_t elem_off, const uint32_t (&r)[32], float inv, int wide) {
    if (OUT_F32) {
        float *dst = (float *)o + elem_off;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = __float_as_uint(__uint_as_float(r[8 * i + e]) * inv);
            if (wide) st_global_v8(dst + 8 * i, v);
            else {
                reinterpret_cast<uint4 *>(dst)[2 * i] = make_uint4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<uint4 *>(dst)[2 * i + 1] = make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
    } else {
        __nv_bfloat16 *dst = (__nv_bfloat16 *)o + elem_off;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[e] = pack_bf16(__uint_as_float(r[16 * i + 2 * e]) * inv, __uint_as_float(r[16 * i + 2 * e + 1]) * inv);
            if (wide) st_global_v8(dst + 16 * i, v);
            else {
                reinterpret_cast<uint4 *>(dst)[2 * i] = make_uint4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<uint4 *>(dst)[2 * i + 1] = make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
    }
}

// Eq. (lse-merge) on one 32-column chunk of an fp32 row: dst = dst * w_old + r * w_new
// (dst is not read when w_old is 0: it may be uninitialised then)
__device__ __forceinline__ void merge_row_chunk(void *o, size_t elem_off, const uint32_t (&r)[32], float w_new,
                                                float w_old) {
    float4 *dst = reinterpret_cast<float4 *>((float *)o + elem_off);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (w_old != 0.f) a = dst[i];
        a.x = a.x * w_old + __uint_as_float(r[4 * i]) * w_new;
        a.y = a.y * w_old + __uint_as_float(r[4 * i + 1]) * w_new;
        a.z = a.z * w_old + __uint_as_float(r[4 * i + 2]) * w_new;
        a.w = a.w * w_old + __uint_as_float(r[4 * i + 3]) * w_new;
        dst[i] = a;
    }
}

// max over one 32-column chunk of scores
__device__ __forceinline__ float chunk_max(const uint32_t (&r)[32], float m) {
    float mm[4] = {m, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int e = 0; e < 32; e += 8)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            mm[c] = max3(mm[c], __uint_as_float(r[e + 2 * c]), __uint_as_float(r[e + 2 * c + 1]));
    return max3(fmaxf(mm[0], mm[1]), mm[2], mm[3]);
}

// p = 2^(s * sl2 + neg_ms) for one 32-column chunk -> 16 packed bf16 pairs at TMEM address `hi` (HL: and
// what the rounding left, at `lo`); the row sum is kept as partial sums (packed fp32 adds)
template <bool HL>
__device__ __forceinline__ void chunk_exp(const uint32_t (&r)[32], float sl2, float neg_ms, float2 (&lsum)[2],
                                          uint32_t hi, uint32_t lo) {
    const float2 s2 = make_float2(sl2, sl2), n2 = make_float2(neg_ms, neg_ms);
    uint32_t pk[16], pl[16];
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        const float2 x = ffma2(make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), s2, n2);
        const float2 pp = make_float2(ex2(x.x), ex2(x.y));
        lsum[(e >> 1) & 1] = fadd2(lsum[(e >> 1) & 1], pp);
        const uint32_t h = pack_bf16(pp.x, pp.y);
        pk[e >> 1] = h;
        if (HL) pl[e >> 1] = pack_bf16(pp.x - __uint_as_float(h << 16), pp.y - __uint_as_float(h & 0xffff0000u));
    }
    tmem_st16(hi, pk);
    if (HL) tmem_st16(lo, pl);
}

// columns that the row does not see become -inf
__device__ __forceinline__ void chunk_mask(uint32_t (&r)[32], uint32_t mk) {
#pragma unroll
    for (int e = 0; e < 32; ++e) r[e] = ((mk >> e) & 1u) ? r[e] : 0xff800000u;
}

// row of the outputs that holds query row `row` (main row or branch token; branch in depth mode)
__device__ __forceinline__ int64_t out_row(const TcFwdParams &p, bool is_main, int row) {
    if (p.depth) return row;
    if (p.partial_out) return is_main ? row - p.r.qm_begin : (p.r.qm_end - p.r.qm_begin) + (row - p.r.tok_begin);
    return is_main ? (int64_t)row : p.meta.n_main + row;
}

// One warp: an item whose rows see no key of the call (a merge into running accumulators changes nothing)
template <int D> __device__ void store_empty_item(const TcFwdParams &p, const Item &it, int lane) {
    if (p.partial_out == 2) return;
    const int heads = min(p.hp, (it.g + 1) * p.group - it.h0);
    const int chunks = D / (p.partial_out ? 4 : 8);        // 16 bytes each
    for (int idx = lane; idx < it.rows * heads * chunks; idx += 32) {
        const int row = idx / chunks;
        const int64_t o = out_row(p, it.is_main, it.row0 + row / heads) * p.h_q + it.h0 + row % heads;
        reinterpret_cast<uint4 *>(p.o)[o * chunks + idx % chunks] = make_uint4(0u, 0u, 0u, 0u);
        if (idx % chunks == 0) p.lse[o] = -INFINITY;
    }
}

// The parts of an item's rows, P of them, each with an unnormalised O and (max, sum) in the shared memory of a CTA of
// the cluster: part s is rank s, or query tile s % 2 of rank s / 2 when both tiles hold the same rows.  A rank
// finishes 1 / S of the rows, P threads per row, D / P columns each.  Latency of distributed shared memory is what
// counts here: a thread reads (max, sum) of one part and the row's threads exchange them, and the reads of O of
// four parts are in flight together (a walk from part to part with a test in between: 8 us more at 16 parts).
template <int D, int P>
__device__ __forceinline__ void combine_parts(const TcFwdParams &p, FwdSmem<D> &sm, int tid) {
    constexpr int kCols = D / P, kVec = kCols / 4;
    const int partial_out = D == 128 ? p.partial_out : 0;
    const Item &it = sm.item[0];
    const int lane = tid & 31, dup = p.same_rows, rank = (int)(blockIdx.x % p.splits);
    const int row = rank * (256 / P) + tid / P, part = tid % P;
    const int i = row >> 7, r_in = row & 127;
    const int tok = r_in / p.hp, h = it.h0 + r_in % p.hp;
    const bool valid = tok < tile_tokens(p, it.is_main, i, it.rows) && h < (it.g + 1) * p.group;
    const int my_row = it.row0 + tok + (i ? tile1_off(p, it.is_main) : 0);
    const int64_t orow = out_row(p, it.is_main, my_row);
    // the threads of a row sit in one warp: all have read the old LSE before one of them replaces it
    const float lse_a = valid && partial_out == 2 ? p.lse[orow * p.h_q + h] : -INFINITY;
    __syncwarp();
    auto slot = [&](int s) { return (dup ? s & 1 : i) * kTile + r_in; };
    const float2 ml = cluster_ld_f2(cluster_map(smem_u32(sm.ml(0) + slot(part)), part >> dup));
    float mx = ml.x;
#pragma unroll
    for (int off = P / 2; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float wgt = ml.x == -INFINITY ? 0.f : ex2(ml.x - mx);
    float sum = wgt * ml.y;
#pragma unroll
    for (int off = P / 2; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    float acc[kCols];
#pragma unroll
    for (int e = 0; e < kCols; ++e) acc[e] = 0.f;
#pragma unroll (P < 4 ? 1 : 4)
    for (int s = 0; s < P; ++s) {
        const float w = __shfl_sync(0xffffffffu, wgt, (lane & ~(P - 1)) + s);
        const uint32_t src = cluster_map(smem_u32(sm.kv[0]) + (uint32_t)(slot(s) * D * 4), s >> dup);
#pragma unroll
        for (int e = 0; e < kVec; ++e) {
            const float4 v = cluster_ld_f4(src + (uint32_t)(((part * kVec + e) ^ (r_in & (D / 4 - 1))) * 16));
            if (w != 0.f) {      // a part without visible keys has written no O
                acc[4 * e] += w * v.x; acc[4 * e + 1] += w * v.y;
                acc[4 * e + 2] += w * v.z; acc[4 * e + 3] += w * v.w;
            }
        }
    }
    bool not_finite = false;
    const uint64_t nans = D == 64 && valid ? nan_mask(acc) : 0;
    if (D == 64) not_finite = __any_sync(0xffffffffu, nans != 0);
    if (!valid && !not_finite) return;
    const float inv = sum > 0.f ? 1.0f / sum : sum;      // 0, or NaN although the part that is NaN may weigh nothing
    const float lse_p = sum > 0.f ? (mx + log2f(sum)) * kLn2 : -INFINITY;
    float lse_out = lse_p, w_new = inv, w_old = 0.f;
    if (partial_out == 2) merge_weights(lse_a, lse_p, inv, lse_out, w_old, w_new);
    const size_t base = ((size_t)orow * p.h_q + h) * D + part * kCols;
    if (valid && part == 0) p.lse[orow * p.h_q + h] = lse_out;
#pragma unroll
    for (int e = 0; valid && e < kVec; ++e) {
        float4 v = make_float4(acc[4 * e] * w_new, acc[4 * e + 1] * w_new, acc[4 * e + 2] * w_new, acc[4 * e + 3] * w_new);
        if (partial_out == 0) {
            *reinterpret_cast<uint2 *>((__nv_bfloat16 *)p.o + base + 4 * e) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
        } else {
            float4 *dst = reinterpret_cast<float4 *>((float *)p.o + base + 4 * e);
            if (w_old != 0.f) {
                const float4 o = *dst;
                v.x += o.x * w_old; v.y += o.y * w_old; v.z += o.z * w_old; v.w += o.w * w_old;
            }
            *dst = v;
        }
    }
    if (D == 64 && not_finite)      // does O hold what the row does not see (ba_exact.cuh; bf16 results only)?
        repair_query_row<false, kCols < 8 ? kCols : 8>(p.rows, it.is_main, my_row, h, it.g, -mx, part * kCols, kCols, nans, inv, (__nv_bfloat16 *)p.o + base);
}

template <int D, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd_kernel(const __grid_constant__ CUtensorMap tm_q_main, const __grid_constant__ CUtensorMap tm_q_branch,
              const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
              const __grid_constant__ CUtensorMap tm_k32, const __grid_constant__ CUtensorMap tm_v32,
              const __grid_constant__ CUtensorMap tm_o, const __grid_constant__ TcFwdParams p,
              const __grid_constant__ BaOrder order) {
    using Smem = FwdSmem<D>;
    constexpr int kStages = Smem::kStages;
    constexpr uint32_t kTileBytes = Smem::kTileBytes;
    constexpr int kHalves = D / 64;
    constexpr bool kHL = D == 64;      // P as hi + lo
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &sm.abort_flag;
    constexpr long long kLimit = D == 64 ? kSlowWaitLimitCycles : kWaitLimitCycles;
    if (smem_u32(smem_raw) & 1023u) {   // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicExch(p.status, BA_EUNSUPPORTED);
        return;
    }

    launch_dependents();      // delta of the backward may be launched (it waits for the end of this kernel)
    if (tid == 0) {
        mbar_init(&sm.q_full, 1);
        mbar_init(&sm.q_empty, 1);
        for (int s = 0; s < kStages; ++s) { mbar_init(&sm.kv_full[s], 1); mbar_init(&sm.kv_empty[s], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.s_full[i], 1);
            mbar_init(&sm.p_half[i], 128);
            mbar_init(&sm.p_full[i], 128);
            mbar_init(&sm.o_full[i], 1);
            mbar_init(&sm.o_free[i], 128);
            mbar_init(&sm.item_full[i], 1);
            mbar_init(&sm.item_empty[i], 10);   // TMA thread, MMA thread, one lane of each softmax warp
            mbar_init(&sm.clc_full[i], 1);
        }
        mbar_init(&sm.loads_out, 1);
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

    if (warp >= 8) {
        reg_dec<kRegsIssue>();
        if (warp == 10) {
            // ================================================= work fetcher (whole warp)
            // An item without keys is finished here (O = 0, LSE = -inf) and never published: the MMA thread looks
            // one item ahead of the softmax warps and must not have to pass a run of items that only those release.
            uint32_t work = SPLIT ? blockIdx.x / p.splits : blockIdx.x;
            const int rank = SPLIT ? (int)(blockIdx.x % p.splits) : 0;
            bool more = true;
            for (int n_item = 0, n_clc = 0;;) {
                const int s = n_item & 1, cs = n_clc & 1;
                bool ok = true;
                if (n_item >= 2) ok = mbar_wait(&sm.item_empty[s], ((n_item >> 1) - 1) & 1, abort_flag, kLimit);
                if (!__all_sync(0xffffffffu, ok)) break;
                if (!more) {
                    if (lane == 0) {
                        sm.item[s].T = -1;
                        mbar_arrive(&sm.item_full[s]);
                    }
                    break;
                }
                if (lane == 0) make_item(p, order, work, rank, sm.item[s]);
                __syncwarp();
                if (!SPLIT && sm.item[s].T == 0) {
                    store_empty_item<D>(p, sm.item[s], lane);
                } else {
                    if (lane == 0) mbar_arrive(&sm.item_full[s]);
                    if (!SPLIT) ok = mbar_wait(&sm.loads_out, n_item & 1, abort_flag, kLimit);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    ++n_item;
                }
                if (SPLIT) {
                    more = false;
                } else {
                    // The next index is asked for when the loads of this item are nearly out, a few steps before its
                    // end.  Taken when the item begins, long items queue up behind one another at the end of the grid:
                    // 512 blocks of 16 on 32,768 tokens (draft rows) 230 us that way, 196 this way.
                    if (lane == 0) {
                        fence_proxy_async();
                        mbar_expect_tx(&sm.clc_full[cs], 16);
                        clc_try_cancel(&sm.clc[cs], &sm.clc_full[cs]);
                    }
                    ok = mbar_wait(&sm.clc_full[cs], (n_clc >> 1) & 1, abort_flag, kLimit);
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
            // ================================================= TMA producer
            if (lane == 0) {
                tma_prefetch_desc(&tm_q_main);
                tma_prefetch_desc(&tm_q_branch);
                tma_prefetch_desc(&tm_k);
                tma_prefetch_desc(&tm_v);
                tma_prefetch_desc(&tm_k32);
                tma_prefetch_desc(&tm_v32);
                tma_prefetch_desc(&tm_o);
                const uint32_t q_bytes = (uint32_t)(p.hp * p.tok * D * 2);
                uint32_t nq = 0, kvi = 0;      // items with keys so far, K / V tiles loaded so far
                bool ok = true;
                for (int n = 0; ok; ++n) {
                    const int sl = n & 1;
                    if (!mbar_wait(&sm.item_full[sl], (n >> 1) & 1, abort_flag, kLimit)) break;
                    const Item &it = sm.item[sl];
                    if (it.T < 0) break;
                    if (it.je > it.jb) {
                        if (nq > 0 && !(ok = mbar_wait(&sm.q_empty, (nq - 1) & 1, abort_flag, kLimit))) break;
                        ++nq;
                        const CUtensorMap *tq = it.is_main ? &tm_q_main : &tm_q_branch;
                        mbar_expect_tx(&sm.q_full, q_bytes * (it.live[0] + it.live[1]));
                        for (int i = 0; i < 2; ++i)
                            if (it.live[i])
                                for (int hf = 0; hf < kHalves; ++hf)
                                    tma_load_3d(sm.q[i] + hf * 16384, tq, hf * 64, it.h0,
                                                it.row0 + (i ? tile1_off(p, it.is_main) : 0), &sm.q_full);
                        for (int j = it.jb; j < it.je && ok; ++j) {
                            const int nch = tile_chunks(it, j);
                            if (j == max(it.je - 1 - kFetchLead, it.jb)) mbar_arrive(&sm.loads_out);
                            for (int kv = 0; kv < 2; ++kv, ++kvi) {
                                const int s = kvi % kStages;
                                if (kvi >= (uint32_t)kStages) ok = mbar_wait(&sm.kv_empty[s], ((kvi / kStages) - 1) & 1, abort_flag, kLimit);
                                if (!ok) break;
                                mbar_expect_tx(&sm.kv_full[s], (uint32_t)(nch * 32 * D * 2));
                                if (j < it.n_full) {
                                    for (int hf = 0; hf < kHalves; ++hf)
                                        tma_load_3d(sm.kv[s] + hf * 16384, kv ? &tm_v : &tm_k, hf * 64, it.g,
                                                    full_row(p, it, j), &sm.kv_full[s]);
                                } else {
                                    for (int c = 0; c < nch; ++c) {
                                        const int row = chunk_row(p, it, 4 * (j - it.n_full) + c);
                                        for (int hf = 0; hf < kHalves; ++hf)
                                            tma_load_3d(sm.kv[s] + hf * 16384 + c * 4096, kv ? &tm_v32 : &tm_k32, hf * 64,
                                                        it.g, row, &sm.kv_full[s]);
                                    }
                                }
                            }
                        }
                    }
                    mbar_arrive(&sm.item_empty[sl]);
                }
                if (*abort_flag) {
                    // leave no copy in flight behind: wait (bounded) for what was issued
                    for (uint32_t k = kvi > (uint32_t)kStages ? kvi - kStages : 0; k < kvi; ++k) {
                        uint32_t spins = 0;
                        while (!mbar_try_wait(&sm.kv_full[k % kStages], (k / kStages) & 1) && ++spins < (1u << 22)) {}
                    }
                    if (nq > 0) {
                        uint32_t spins = 0;
                        while (!mbar_try_wait(&sm.q_full, (nq - 1) & 1) && ++spins < (1u << 22)) {}
                    }
                }
            }
        } else if (warp == 8) {
            // ================================================= MMA issuer (one elected thread)
            // This thread is a serial chain between the softmax warps of one step and the next: every
            // instruction between an arrival and the MMAs it releases counts (some 5 clocks each), so the
            // steps are planned, and the K stage of the next one awaited, before the arrival.  (The whole warp
            // running this code and electing a lane per MMA, which is as fast in a bare loop, took 16,384
            // tokens x 4 rows from 7.8 to 8.6 ms: the control flow per step is what costs.)
            if (elect_one()) {
                constexpr uint32_t IDESC_PV = idesc_bf16(128, D, 1);
                const uint32_t q_km = smem_desc_lo(smem_u32(sm.q[0]), 16);
                const uint32_t kv_km0 = smem_desc_lo(smem_u32(sm.kv[0]), 16), kv_mn0 = smem_desc_lo(smem_u32(sm.kv[0]), 16384);
                constexpr uint32_t kStageStep = kTileBytes >> 4;
                auto issue_qk = [&](int i, uint32_t k_km, uint32_t idesc) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        mma_ss_lh(tmem + i * 128, q_km + i * kStageStep + desc_step_kmajor(ks), k_km + desc_step_kmajor(ks), idesc, ks > 0);
                    tc_commit(&sm.s_full[i]);
                };
                auto issue_pv = [&](int i, uint32_t v_mn, int ks0, bool accumulate) {      // two 16-key steps
#pragma unroll
                    for (int ks = ks0; ks < ks0 + 2; ++ks)
                        mma_ts_lh(tmem + 256 + i * 128, tmem + i * 128 + ks * 8, v_mn + desc_step_mnmajor(ks), IDESC_PV,
                                  accumulate || ks > 0);
                    if (kHL)
#pragma unroll
                        for (int ks = ks0; ks < ks0 + 2; ++ks)
                            mma_ts_lh(tmem + 256 + i * 128, tmem + 256 + i * 128 + 64 + ks * 8, v_mn + desc_step_mnmajor(ks), IDESC_PV, 1);
                };
                // The steps (key tiles) of successive items form one stream: the first Q K^T of the next item
                // takes the place of the one that would follow the last step, so no query tile idles at the seam.
                struct Step {
                    uint32_t live;       // bit i: query tile i sees the tile; 0x80: no step
                    uint32_t idesc;      // of Q K^T: N = 32 nch
                    int nch;
                    bool first, last;    // of its item
                };
                Item it;
                int n_item = 0, j_cur = 0;
                it.je = 0;
                bool ok = true, done = false;
                auto advance = [&](Step &st) {
                    st.first = false;
                    ++j_cur;
                    while (j_cur >= it.je && !done) {       // next item with keys
                        const int sl = n_item & 1;
                        ok = ok && mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag, kLimit);
                        if (!ok) { done = true; break; }
                        const Item &im = sm.item[sl];
                        it.T = im.T; it.je = im.je; it.n_full = im.n_full; it.n_ch = im.n_ch;
                        j_cur = im.jb;
#pragma unroll
                        for (int i = 0; i < 2; ++i) { it.live[i] = im.live[i]; it.va[i] = im.va[i]; it.vb[i] = im.vb[i]; }
                        mbar_arrive(&sm.item_empty[sl]);
                        ++n_item;
                        st.first = true;
                        done = it.T < 0;
                    }
                    st.live = done ? 0x80u : (tile_live(it, 0, j_cur) ? 1u : 0u) | (tile_live(it, 1, j_cur) ? 2u : 0u);
                    if (SPLIT && p.same_rows && !done) st.live &= 1u << (j_cur & 1);
                    st.nch = tile_chunks(it, j_cur);
                    st.idesc = idesc_bf16(128, 0, 0) | ((uint32_t)(st.nch * 4) << 17);
                    st.last = j_cur + 1 >= it.je;
                };
                uint32_t nq = 0, kvi = 0;
                uint32_t par_p = 0, par_o = 0, used_o = 0, started = 0;     // bit i: phase parities of query tile i; O_i used
                Step cur, nxt;
                advance(cur);
                if (ok && !done) {
                    ok = mbar_wait(&sm.q_full, 0, abort_flag, kLimit) && mbar_wait(&sm.kv_full[0], 0, abort_flag, kLimit);
                    nq = 1;
                    if (ok) {
                        tc_fence_after();
                        if (cur.live & 1u) issue_qk(0, kv_km0, cur.idesc);
                        if (cur.live & 2u) issue_qk(1, kv_km0, cur.idesc);
                        tc_commit(&sm.kv_empty[0]);
                        if (cur.last) tc_commit(&sm.q_empty);
                    }
                }
                for (; ok && cur.live != 0x80u; kvi += 2, cur = nxt) {
                    const int sv = (kvi + 1) % kStages, sk = (kvi + 2) % kStages;
                    const uint32_t v_mn = kv_mn0 + sv * kStageStep, k_km = kv_km0 + sk * kStageStep;
                    advance(nxt);
                    const bool more = nxt.live != 0x80u;
                    // Steps of different query tiles: the next Q K^T does not wait for the softmax of this one
                    // (its S was released by the P V issued before).
                    const bool early = SPLIT && more && !(nxt.live & cur.live);
                    if (early) {
                        ok = ok && mbar_wait(&sm.kv_full[sk], ((kvi + 2) / kStages) & 1, abort_flag, kLimit);
                        if (!ok) break;
                        tc_fence_after();
                        if (nxt.live & 1u) issue_qk(0, k_km, nxt.idesc);
                        if (nxt.live & 2u) issue_qk(1, k_km, nxt.idesc);
                        tc_commit(&sm.kv_empty[sk]);
                    }
                    ok = ok && mbar_wait(&sm.kv_full[sv], ((kvi + 1) / kStages) & 1, abort_flag, kLimit);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (!ok) break;
                        const bool live = (cur.live >> i) & 1u;
                        if (live) {
                            const bool acc = (started >> i) & 1u;
                            // O of the item before has been read out
                            if (!acc && ((used_o >> i) & 1u) && !(ok = mbar_wait(&sm.o_free[i], ((par_o >> i) & 1u) ^ 1u, abort_flag, kLimit))) break;
                            if (!(ok = mbar_wait(&sm.p_half[i], (par_p >> i) & 1u, abort_flag, kLimit))) break;
                            tc_fence_after();
                            issue_pv(i, v_mn, 0, acc);          // keys 0-63 while the softmax warps finish keys 64-127
                            if (cur.nch > 1) issue_pv(i, v_mn, 2, true);
                            started |= 1u << i;
                        }
                        if (i == 0 && more && !early) {
                            ok = mbar_wait(&sm.kv_full[sk], ((kvi + 2) / kStages) & 1, abort_flag, kLimit);
                            if (ok && nxt.first) ok = mbar_wait(&sm.q_full, nq & 1, abort_flag, kLimit);
                            if (!ok) break;
                        }
                        if (live) {
                            if (!(ok = mbar_wait(&sm.p_full[i], (par_p >> i) & 1u, abort_flag, kLimit))) break;
                            par_p ^= 1u << i;
                            tc_fence_after();
                            if (cur.nch > 2) issue_pv(i, v_mn, 4, true);
                            if (cur.nch > 3) issue_pv(i, v_mn, 6, true);
                        }
                        if (!SPLIT && cur.last && ((started >> i) & 1u)) tc_commit(&sm.o_full[i]);
                        if (more && !early && ((nxt.live >> i) & 1u)) issue_qk(i, k_km, nxt.idesc);
                    }
                    if (!ok) break;
                    if (SPLIT && cur.last) {
                        // both at the end: the softmax warps then write over the K / V stages, which the
                        // last P V of either query tile may still be reading before this point
                        if (started & 1u) tc_commit(&sm.o_full[0]);
                        if (started & 2u) tc_commit(&sm.o_full[1]);
                    }
                    tc_commit(&sm.kv_empty[sv]);
                    if (more) {
                        if (!early) tc_commit(&sm.kv_empty[sk]);
                        if (nxt.last) tc_commit(&sm.q_empty);
                        nq += nxt.first;
                    }
                    if (cur.last) {
                        par_o ^= started;
                        used_o |= started;
                        started = 0;
                    }
                }
            }
            __syncwarp();
        }
    } else {
        // ================================================= softmax + epilogue
        reg_inc<kRegsSoftmax>();
        const int i = warp >> 2;                                   // query tile 0 / 1
        const int r_in = tid & 127;                                // my TMEM lane
        const int my_tok = r_in / p.hp, my_head = r_in % p.hp;     // token and head within the tile
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t s_addr = tmem + lane_base + i * 128;
        const uint32_t o_addr = tmem + lane_base + 256 + i * 128, lo_addr = o_addr + 64;
        const float sl2 = p.scale_log2;
        const int partial_out = D == 128 ? p.partial_out : 0;      // head_dim 64: bf16 results only (ba_use_tc)
        uint32_t n_s = 0, n_o = 0;
        // What this role needs of an item, and this thread's row.  Everything the key loop uses sits in
        // registers (a shared-memory load of these warps waits several hundred clocks behind the operand
        // reads of the Q K^T MMAs), and the next item is read while O of the current one is awaited.
        struct Work {
            int T, jb, je, n_full, lo_min, n_mc, n_ch, bs, va, vb, wa, wb, rows, cnt, h, g, my_row;
            bool is_main, valid;
            int lo, hi, br_start;
            uint64_t bmask;
        } w, nx;
        auto fetch = [&](int nit, Work &f) -> bool {
            const int sl = nit & 1;
            if (!mbar_wait(&sm.item_full[sl], (nit >> 1) & 1, abort_flag, kLimit)) return false;
            const Item &im = sm.item[sl];
            f.T = im.T; f.je = im.je; f.n_full = im.n_full; f.lo_min = im.lo_min; f.n_mc = im.n_mc; f.n_ch = im.n_ch;
            f.bs = im.bs; f.va = im.va[i]; f.vb = im.vb[i]; f.wa = im.wa[i]; f.wb = im.wb[i];
            f.jb = im.live[i] ? im.jb : im.je;
            f.rows = im.rows;
            f.is_main = im.is_main;
            const int off1 = tile1_off(p, f.is_main);
            f.h = im.h0 + my_head;
            f.g = im.g;
            f.cnt = tile_tokens(p, f.is_main, i, f.rows);     // tokens of my query tile
            f.valid = my_tok < f.cnt && f.h < (im.g + 1) * p.group;
            f.my_row = im.row0 + my_tok + (i ? off1 : 0);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.item_empty[sl]);
            f.lo = 1; f.hi = 0; f.br_start = 0; f.bmask = 0;
            if (f.T >= 0 && f.valid) {
                const int64_t grow = f.is_main ? f.my_row : p.meta.n_main + (p.depth ? (int64_t)f.my_row * p.branch_len : f.my_row);
                f.lo = p.meta.row_lo[grow];
                f.hi = p.meta.row_hi[grow];
                if (!f.is_main && (p.r.parts & BA_PART_BRANCH) && !p.depth) {
                    f.br_start = p.meta.br_start[f.my_row];
                    f.bmask = p.meta.br_mask[f.my_row];
                }
            }
            return true;
        };
        bool ok = fetch(0, nx);
        for (int nit = 0; ok; ++nit) {
            w = nx;
            if (w.T < 0) break;
            int lo = 1, hi = 0;
            if (w.valid && (p.r.parts & BA_PART_MAIN)) {
                lo = max(w.lo, (int)p.r.kv_begin);
                hi = min(w.hi, (int)p.r.kv_end - 1);
            }
            const int br_off = w.bs - w.br_start, n_full = w.n_full, je = w.je;
            const int t_rel = my_tok + (i ? tile1_off(p, w.is_main) : 0);
            auto vis = [&](int j, int c) -> uint32_t {
                return w.valid ? chunk_vis(p, j, c, n_full, w.lo_min, w.n_mc, lo, hi, br_off, w.bmask, t_rel, w.rows) : 0u;
            };

            float m_run = -INFINITY, l_run = 0.f, neg_ms = 0.f;
            bool started = false;
            for (int j = w.jb; j < je; ++j) {
                if (j < n_full && (j < w.va || j >= w.vb)) continue;      // no row of this tile sees it
                if (SPLIT && p.same_rows && (j & 1) != i) continue;
                const int nch = j < n_full ? 4 : min(4, w.n_ch - 4 * (j - n_full));
                ok = mbar_wait(&sm.s_full[i], n_s & 1, abort_flag, kLimit);
                ++n_s;
                if (!ok) break;
                tc_fence_after();
                // Running maximum; O and l are rescaled only when it grew by more than the threshold (from -inf
                // on the first visible key; -inf against -inf compares as NaN: nothing happens).
                auto grown = [&](float m_tile) {
                    const bool grow = (m_tile - m_run) * sl2 > kRescaleThreshold;
                    if (__any_sync(0xffffffffu, grow)) {
                        float alpha = 1.0f;
                        if (grow) {
                            alpha = ex2((m_run - m_tile) * sl2);  // m_run = -inf gives 0
                            l_run *= alpha;
                            m_run = m_tile;
                            neg_ms = -m_run * sl2;
                        }
                        if (started) {
                            // O_i is idle: its last P V was finished before this tile's scores were formed
#pragma unroll 1
                            for (int c = 0; c < D / 16; ++c) {
                                uint32_t r[16];
                                tmem_ld16(o_addr + c * 16, r);
                                tmem_wait_ld();
#pragma unroll
                                for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
                                tmem_st16(o_addr + c * 16, r);
                            }
                        }
                    }
                    started = true;
                };
                // P = exp2(s * scale_log2 - m) goes over the first score columns as bf16
                float2 l2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if (nch == 4) {
                    uint32_t r0[32], r1[32], r2[32], r3[32];
                    tmem_ld32(s_addr, r0);
                    tmem_ld32(s_addr + 32, r1);
                    tmem_ld32(s_addr + 64, r2);
                    tmem_ld32(s_addr + 96, r3);
                    tmem_wait_ld();
                    if (j >= n_full || j < w.wa || j >= w.wb) {      // not every row sees the whole tile
                        chunk_mask(r0, vis(j, 0));
                        chunk_mask(r1, vis(j, 1));
                        chunk_mask(r2, vis(j, 2));
                        chunk_mask(r3, vis(j, 3));
                    }
                    float m_tile = chunk_max(r0, -INFINITY);
                    m_tile = chunk_max(r1, m_tile);
                    m_tile = chunk_max(r2, m_tile);
                    m_tile = chunk_max(r3, m_tile);
                    grown(m_tile);
                    chunk_exp<kHL>(r0, sl2, neg_ms, l2, s_addr, lo_addr);
                    chunk_exp<kHL>(r1, sl2, neg_ms, l2, s_addr + 16, lo_addr + 16);
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(&sm.p_half[i]);       // P of keys 0-63 is in place: P V may start
                    chunk_exp<kHL>(r2, sl2, neg_ms, l2, s_addr + 32, lo_addr + 32);
                    chunk_exp<kHL>(r3, sl2, neg_ms, l2, s_addr + 48, lo_addr + 48);
                } else {
                    // a narrow tail tile: chunk by chunk, scores read twice
                    uint32_t r[32];
                    float m_tile = -INFINITY;
#pragma unroll 1
                    for (int c = 0; c < nch; ++c) {
                        tmem_ld32(s_addr + 32 * c, r);
                        const uint32_t mk = vis(j, c);
                        tmem_wait_ld();
                        chunk_mask(r, mk);
                        m_tile = chunk_max(r, m_tile);
                    }
                    grown(m_tile);
#pragma unroll 1
                    for (int c = 0; c < nch; ++c) {
                        tmem_ld32(s_addr + 32 * c, r);
                        const uint32_t mk = vis(j, c);
                        tmem_wait_ld();
                        chunk_mask(r, mk);
                        chunk_exp<kHL>(r, sl2, neg_ms, l2, s_addr + 16 * c, lo_addr + 16 * c);
                        if (c == min(2, nch) - 1) {
                            tmem_wait_st();
                            tc_fence_before();
                            mbar_arrive(&sm.p_half[i]);
                        }
                    }
                }
                l_run += (l2[0].x + l2[0].y) + (l2[1].x + l2[1].y);
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&sm.p_full[i]);
            }
            if (!ok) break;
            if (!SPLIT && !(ok = fetch(nit + 1, nx))) break;
            // --- epilogue: O / l and LSE
            if (started) {
                ok = mbar_wait(&sm.o_full[i], n_o & 1, abort_flag, kLimit);
                ++n_o;
                if (!ok) break;
                tc_fence_after();
            }
            if (SPLIT) {
                // unnormalised O and (max, sum) of my part into shared memory (o_full covers every MMA of
                // this CTA, so the K / V stages are idle)
                // (a sum that is NaN is not an empty part; its maximum may be none)
                const bool any = started && l_run != 0.f;
                sm.ml(i)[r_in] = make_float2(any ? (m_run == -INFINITY ? 0.f : m_run * sl2) : -INFINITY, any ? l_run : 0.f);
                if (started) {
                    float4 *dst = reinterpret_cast<float4 *>(sm.kv[0]) + (size_t)(i * kTile + r_in) * (D / 4);
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(o_addr + c * 32, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 8; ++e)      // 16-byte chunks swizzled by the row: no bank conflicts
                            dst[(8 * c + e) ^ (r_in & (D / 4 - 1))] =
                                make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]),
                                            __uint_as_float(r[4 * e + 2]), __uint_as_float(r[4 * e + 3]));
                    }
                }
                break;       // the merge follows below, with all threads of the cluster
            }
            const int64_t orow = out_row(p, w.is_main, w.my_row);
            const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
            const size_t base = ((size_t)orow * p.h_q + w.h) * D;
            const float lse_p = l_run > 0.f ? (m_run * sl2 + log2f(l_run)) * kLn2 : -INFINITY;
            float w_new = inv, w_old = 0.f;   // partial_out == 2: weights of Eq. (lse-merge)
            if (w.valid) {
                float lse_out = lse_p;
                if (partial_out == 2) merge_weights(p.lse[orow * p.h_q + w.h], lse_p, inv, lse_out, w_old, w_new);
                p.lse[orow * p.h_q + w.h] = lse_out;
            }
            // A warp whose rows are all live hands 64 columns at a time to a TMA store: row by row from
            // registers, a warp instruction touches 32 cache lines and the stores of an item took 4,000
            // (32-byte) to 6,000 clocks (16-byte), as long as two key tiles; this way an epilogue takes 2,500.
            bool by_tma = p.warp_tok > 0 && ((warp & 3) + 1) * p.warp_tok <= w.cnt;
            const uint32_t stage = smem_u32(sm.out[warp]) + lane * 128;
#pragma unroll 1
            for (int hf = 0; hf < D / 64; ++hf) {
                uint32_t ra[32], rb[32];
                if (started) {      // every lane runs the (warp-collective) TMEM loads; only live rows store
                    tmem_ld32(o_addr + hf * 64, ra);
                    tmem_ld32(o_addr + hf * 64 + 32, rb);
                    tmem_wait_ld();
                    if (hf == D / 64 - 1) {
                        tc_fence_before();
                        mbar_arrive(&sm.o_free[i]);   // the next item's P V may overwrite O_i
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) ra[e] = rb[e] = 0u;
                }
                bool not_finite = false;
                uint64_t nans = 0;
                if (D == 64) {
                    const float s = sum32(ra) + sum32(rb);
                    not_finite = __any_sync(0xffffffffu, w.valid && s != s);
                    if (not_finite) {
                        if (w.valid) nans = nan_mask(ra) | nan_mask(rb) << 32;
                        by_tma = false;
                    }
                }
                if (by_tma) {
                    if (lane == 0) tma_store_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint32_t (&r)[32] = c < 4 ? ra : rb;
                        const int e = 8 * (c & 3);
                        st_shared_v4(stage + ((c ^ (lane & 7)) << 4),
                                     pack_bf16(__uint_as_float(r[e]) * inv, __uint_as_float(r[e + 1]) * inv),
                                     pack_bf16(__uint_as_float(r[e + 2]) * inv, __uint_as_float(r[e + 3]) * inv),
                                     pack_bf16(__uint_as_float(r[e + 4]) * inv, __uint_as_float(r[e + 5]) * inv),
                                     pack_bf16(__uint_as_float(r[e + 6]) * inv, __uint_as_float(r[e + 7]) * inv));
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) tma_store_3d(&tm_o, hf * 64, w.h, (int)orow, smem_u32(sm.out[warp]));
                } else if (w.valid) {
                    const size_t off = base + hf * 64;
                    if (partial_out == 2) {
                        merge_row_chunk(p.o, off, ra, w_new, w_old);
                        merge_row_chunk(p.o, off + 32, rb, w_new, w_old);
                    } else if (partial_out) {
                        store_row_chunk<true>(p.o, off, ra, inv, p.wide);
                        store_row_chunk<true>(p.o, off + 32, rb, inv, p.wide);
                    } else {
                        store_row_chunk<false>(p.o, off, ra, inv, p.wide);
                        store_row_chunk<false>(p.o, off + 32, rb, inv, p.wide);
                    }
                }
                if (D == 64 && not_finite)      // does O hold what the row does not see (ba_exact.cuh; bf16 results only)?
                    repair_query_row<false, 8>(p.rows, w.is_main, w.my_row, w.h, w.g, neg_ms, 0, 64, nans, inv, (__nv_bfloat16 *)p.o + base);
            }
        }
        if (lane == 0) tma_store_wait_all();
    }

    if (SPLIT) {
        __syncwarp();
        cluster_sync_all();
        if (warp < 8) {
            switch (p.splits << p.same_rows) {
                case 2: combine_parts<D, 2>(p, sm, tid); break;
                case 4: combine_parts<D, 4>(p, sm, tid); break;
                case 8: combine_parts<D, 8>(p, sm, tid); break;
                default: combine_parts<D, 16>(p, sm, tid); break;
            }
        }
        __syncwarp();
        cluster_sync_all();      // no CTA leaves while another may still read its shared memory
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
    if (tid == 0 && sm.abort_flag) atomicExch(p.status, BA_ETIMEOUT);
}

template <int D, bool SPLIT> int prepare_kernel(int dev) {
    // the dynamic shared-memory limit is a per-device attribute of the kernel
    static bool attr_set[64] = {};
    if (dev < 0 || dev >= 64) return BA_EUNSUPPORTED;
    if (attr_set[dev]) return BA_OK;
    // The register re-split hands out what a launch with kRegsLaunch registers per thread owns: a build
    // that gave the kernel fewer would leave setmaxnreg.inc waiting for registers nobody releases.
    cudaFuncAttributes fa;
    BA_CUDA_CHECK(cudaFuncGetAttributes(&fa, tc_fwd_kernel<D, SPLIT>));
    if (fa.numRegs * kThreads < 256 * kRegsSoftmax + 128 * kRegsIssue) return BA_EUNSUPPORTED;
    BA_CUDA_CHECK(cudaFuncSetAttribute(tc_fwd_kernel<D, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(FwdSmem<D>)));
    attr_set[dev] = true;
    return BA_OK;
}

template <int D>
int launch_fwd(TcFwdParams &p, const BaOrder &order, const CUtensorMap *tm, int64_t work, int dev, cudaStream_t st) {
    const size_t smem = sizeof(FwdSmem<D>);
    if (p.splits == 1) {
        int rc = prepare_kernel<D, false>(dev);
        if (rc != BA_OK) return rc;
        tc_fwd_kernel<D, false><<<(unsigned)work, kThreads, smem, st>>>(tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], p, order);
        return ba_check_launch();
    }
    int rc = prepare_kernel<D, true>(dev);
    if (rc != BA_OK) return rc;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)(work * p.splits));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)p.splits;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_fwd_kernel<D, true>, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], p, order));
    return ba_check_launch();
}

// Work items of a call and their cluster splits; returns the number of items.
// Few items and long key ranges (a handful of branches on long sequences): split the keys of an item over a
// cluster until the SMs are busy, as long as a part keeps at least four tiles.  With branches of different
// sequences in the two query tiles (same_rows), an item per sequence's rows and both tiles on them, unless two
// parts per item already exceed one CTA per SM on short sequences.  Kernel times with the caches flushed, 31-node
// trees at the end of each of 8 / 16 sequences of 8,192 tokens, two sequences per item / same_rows: 154 / 100 and
// 177 / 137 us; 9-node trees, 12 sequences of 8,333: 196 / 88; 16 sequences of 1,024 tokens: 47 / 50, not taken.
// With parts until there are four CTAs per SM: 159 us instead of 100.
int64_t split_items(ItemParams &p, const ba_plan *pl, const BaRange &r, bool has_main, int depth) {
    const ba_problem_t &pr = pl->prob;
    const int64_t est_tiles = (r.parts & BA_PART_MAIN) && pr.num_seqs > 0 ? (r.kv_end - r.kv_begin) / pr.num_seqs / kTile : 0;
    int64_t work;
    auto split = [&](bool same_rows_ok) {
        work = fill_items(p, pl, r, has_main, depth, same_rows_ok);
        p.splits = 1;
        while (p.splits < 8 && work * p.splits * 2 <= 2 * kSms && est_tiles >= 4 * 2 * p.splits) p.splits *= 2;
    };
    split(true);
    // (the kernel for whole items has different rows in its tiles)
    if (p.same_rows && (p.splits == 1 || (work * 2 > kSms && est_tiles < 32))) split(false);
    return work;
}

}  // namespace

bool ba_tc_supported(const ba_problem_t *p) {
    return p->dtype == BA_BF16 && (p->head_dim == 64 || p->head_dim == 128) && encode_tiled_fn() != nullptr;
}

int ba_tc_fwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch, const void *k,
              const void *v, void *o, float *lse, int partial_out, cudaStream_t st, int depth) {
    int dev = 0;
    BA_CUDA_CHECK(cudaGetDevice(&dev));
    const ba_problem_t &pr = pl->prob;
    const int D = pr.head_dim;
    TcFwdParams p;
    memset(&p, 0, sizeof p);
    p.o = o;
    p.lse = lse;
    p.scale_log2 = pl->scale * kLog2e;
    p.partial_out = partial_out;   // 0 final layout, 1 compact fp32, 2 compact fp32 merged in place
    p.wide = ((uintptr_t)o & 31) == 0;
    p.status = pl->dev_status;
    p.rows.meta = pl->meta; p.rows.r = r;
    p.rows.q_main = q_main; p.rows.q_branch = q_branch; p.rows.k = k; p.rows.v = v;
    p.rows.h_q = pr.h_q; p.rows.h_kv = pr.h_kv; p.rows.group = pr.h_q / pr.h_kv;
    p.rows.scale_log2 = p.scale_log2;
    const int64_t work = split_items(p, pl, r, q_main != nullptr, depth);
    if (work == 0) return BA_OK;
    if (work > INT_MAX) return BA_EUNSUPPORTED;

    CUtensorMap tm[7];
    // depth mode: only the key rows of depths <= depth exist yet; rows beyond them read as zero.  Without
    // own-branch keys nothing beyond kv_end is needed (a received shard ends there).
    const uint64_t kv_rows = depth ? (uint64_t)(pr.n_main + (int64_t)depth * pr.num_branches)
                             : (r.parts & BA_PART_BRANCH) ? (uint64_t)(pr.n_main + pr.n_branch)
                                                          : (uint64_t)(r.kv_end > r.kv_base ? r.kv_end - r.kv_base : 1);
    // an absent query tensor still needs a valid map object: alias the other one
    const void *qm = q_main ? q_main : q_branch;
    const void *qb = (q_branch && pr.n_branch > 0) ? q_branch : q_main;
    const uint64_t qm_rows = depth ? (uint64_t)pr.num_branches : q_main ? (uint64_t)pr.n_main : (uint64_t)pr.n_branch;
    uint64_t qb_rows = (q_branch && pr.n_branch > 0) ? (uint64_t)pr.n_branch : (uint64_t)pr.n_main;
    if (depth) qb_rows = (uint64_t)pr.num_branches;     // the queries of one depth: one row per branch
    if (!make_tmap_rhd(&tm[0], qm, qm_rows, pr.h_q, D, p.tok, p.hp) ||
        !make_tmap_rhd(&tm[1], qb, qb_rows, pr.h_q, D, p.tok, p.hp) ||
        !make_tmap_rhd(&tm[2], k, kv_rows, pr.h_kv, D, kTile) || !make_tmap_rhd(&tm[3], v, kv_rows, pr.h_kv, D, kTile) ||
        !make_tmap_rhd(&tm[4], k, kv_rows, pr.h_kv, D, 32) || !make_tmap_rhd(&tm[5], v, kv_rows, pr.h_kv, D, 32))
        return BA_EINVAL;
    // bf16 outputs: the 32 rows of a warp are whole tokens when the group size divides 32
    p.warp_tok = !partial_out && 32 % p.hp == 0 ? 32 / p.hp : 0;
    const uint64_t o_rows = depth ? (uint64_t)pr.num_branches : (uint64_t)(pr.n_main + pr.n_branch);
    if (!p.warp_tok) tm[6] = tm[0];
    else if (!make_tmap_rhd(&tm[6], o, o_rows, pr.h_q, D, p.warp_tok, p.hp)) return BA_EINVAL;
    const BaOrder &order = item_order(p, pl, q_main != nullptr);
    return D == 128 ? launch_fwd<128>(p, order, tm, work, dev, st) : launch_fwd<64>(p, order, tm, work, dev, st);
}

void ba_tc_fwd_orders(ba_plan *pl, const ba_problem_t *host) {
    for (int has_main = 1; has_main >= 0; --has_main) {
        ItemParams p;
        if (fill_items(p, pl, ba_everything(pl), has_main, 0) > 0) ba_add_order(pl, host, item_tiling(p, has_main));
    }
}

const BaOrder &ba_tc_fwd_order(const ba_plan *pl, bool has_main, BaTiling *t) {
    ItemParams p;
    split_items(p, pl, ba_everything(pl), has_main, 0);
    *t = item_tiling(p, has_main);
    return item_order(p, pl, has_main);
}
