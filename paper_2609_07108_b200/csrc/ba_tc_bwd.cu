// Tensor-core backward (sm_100a, bf16): dQ at head_dim 64 and 128, dK/dV at head_dim 64 (128: ba_tc_dkdv.cu).
//
// Gradients of the attention of paper Section 3.2, accumulated over key chunks
// ("replays the same K/V ring and accumulates gradients locally").  With the
// final log-sum-exp l and delta = <dO, O> of each row:
//   P = exp(scale * Q K^T - l),  dP = dO V^T,  dS = P o (dP - delta),
//   dQ = scale * dS K,  dK = scale * dS^T Q,  dV = P^T dO.
// Every output element has exactly one owning CTA, so sums are deterministic.
//
// dQ kernel, head_dim 128: query-stationary, work items and roles of the forward (ba_tc_fwd.cu).  Per key
// tile S -> TMEM, the P / dS warps turn it into P (kept in registers as bf16), the same TMEM columns then
// receive dP, the warps form dS (bf16, written over those columns) and the tensor core adds dS K into the dQ
// accumulator.  Q, dO of an item and two K, one V tile fill the shared memory; the next item's Q is loaded
// behind the last S, its dO behind the last dP of the current one.  Bound by the same chain as the forward, one
// link longer (S -> P -> dP -> dS -> dQ): 4,750 clocks per step of two tiles against 3,072 of MMA.  2,048-token
// chain batch 134 -> 88 us, 32,768 tokens with blocks 1280 -> 1150, 65,536-token trees 5850 -> 5470 (128 rows of
// one head per tile, one CTA per item before).
//   TMEM: R_0 [0,128) R_1 [128,256) (S, then dP, then dS)  dQ_0 [256,384) dQ_1 [384,512)
#include <type_traits>

#include "ba_tc_bwd.cuh"

using namespace sm100;

namespace {

// ============================================================================
// dQ
// ============================================================================
// the next index is asked for when the loads of the last but this many tiles go out (see the forward)
constexpr int kDqFetchLead = 2, kKvFetchLead = 4;
constexpr int kDqThreads = 384;
constexpr int kDqRegsCompute = 208, kDqRegsIssue = 88, kDqRegsLaunch = 168;
static_assert(256 * kDqRegsCompute + 128 * kDqRegsIssue <= kDqThreads * kDqRegsLaunch, "register re-split exceeds what the CTA owns");

struct DqSmem {
    alignas(1024) uint8_t q[2][kTileBytes];
    alignas(1024) uint8_t go[2][kTileBytes];
    alignas(1024) uint8_t kbuf[2][kTileBytes];
    alignas(1024) uint8_t vbuf[kTileBytes];
    alignas(16) uint4 clc[2];
    Item item[2];
    alignas(8) uint64_t q_full, q_empty, go_full, go_empty, v_full, v_empty;
    uint64_t k_full[2], k_empty[2];
    uint64_t s_full[2], a_done[2], dp_full[2], b_done[2], dq_full[2], dq_free[2];
    uint64_t item_full[2], item_empty[2], clc_full[2], loads_out;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(DqSmem) <= 232448, "shared memory of the dQ kernel");

struct TcDqParams : ItemParams {
    const float *nlse2_t, *delta_t;   // head-major [h_q, row_pitch]: -LSE log2(e), delta
    int64_t row_pitch;
    void *dq_main, *dq_branch;
    float scale, scale_log2;
    int accumulate, wide;             // wide: bf16 gradients are 32-byte aligned
    int *status;
};

// P = 2^(s * sl2 + neg_lse2) for one 32-column chunk, as 16 packed bf16 pairs (invisible columns: 0)
template <bool MASKED>
__device__ __forceinline__ void chunk_p(const uint32_t (&r)[32], uint32_t mk, float sl2, float neg_lse2, uint32_t *pr) {
    const float2 s2 = make_float2(sl2, sl2), n2 = make_float2(neg_lse2, neg_lse2);
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        const float2 x = ffma2(make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), s2, n2);
        float p0 = ex2(x.x), p1 = ex2(x.y);
        if (MASKED) {
            p0 = ((mk >> e) & 1u) ? p0 : 0.f;
            p1 = ((mk >> (e + 1)) & 1u) ? p1 : 0.f;
        }
        pr[e >> 1] = pack_bf16(p0, p1);
    }
}

// dS = P o (dP - delta) for one 32-column chunk (P given as packed bf16 pairs)
__device__ __forceinline__ void chunk_ds(const uint32_t (&r)[32], const uint32_t *pr, float dlt,
                                         uint32_t (&pk)[16]) {
    const float2 nd = make_float2(-dlt, -dlt);
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        const uint32_t pp = pr[e >> 1];
        const float2 pf = make_float2(__uint_as_float(pp << 16), __uint_as_float(pp & 0xffff0000u));
        const float2 d = fmul2(pf, fadd2(make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), nd));
        pk[e >> 1] = pack_bf16(d.x, d.y);
    }
}

__global__ void __launch_bounds__(kDqThreads, 1)
tc_dq_kernel(const __grid_constant__ CUtensorMap tm_q_main, const __grid_constant__ CUtensorMap tm_q_branch,
             const __grid_constant__ CUtensorMap tm_go, const __grid_constant__ CUtensorMap tm_k,
             const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k32,
             const __grid_constant__ CUtensorMap tm_v32, const TcDqParams p, const __grid_constant__ BaOrder order) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    DqSmem &sm = *reinterpret_cast<DqSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &sm.abort_flag;
    if (smem_u32(smem_raw) & 1023u) {   // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicExch(p.status, BA_EUNSUPPORTED);
        return;
    }
    // global row number of branch query 0 (rows of dO and of the per-row scalars): branch rows follow the main
    // rows, except in depth mode, where those tensors hold one row per branch
    const int qbase = p.depth ? 0 : (int)p.meta.n_main;

    if (tid == 0) {
        mbar_init(&sm.q_full, 1); mbar_init(&sm.q_empty, 1);
        mbar_init(&sm.go_full, 1); mbar_init(&sm.go_empty, 1);
        mbar_init(&sm.v_full, 1); mbar_init(&sm.v_empty, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.k_full[i], 1);
            mbar_init(&sm.k_empty[i], 1);
            mbar_init(&sm.s_full[i], 1);
            mbar_init(&sm.a_done[i], 128);
            mbar_init(&sm.dp_full[i], 1);
            mbar_init(&sm.b_done[i], 128);
            mbar_init(&sm.dq_full[i], 1);
            mbar_init(&sm.dq_free[i], 128);
            mbar_init(&sm.item_full[i], 1);
            mbar_init(&sm.item_empty[i], 10);   // TMA thread, MMA thread, one lane of each P / dS warp
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
    wait_prerequisites();     // launched while delta ends
    launch_dependents();      // the dK/dV kernel may take the SMs that this one leaves; delta is there for it too

    if (warp >= 8) {
        reg_dec<kDqRegsIssue>();
        if (warp == 10) {
            // ================================================= work fetcher (whole warp, as in the forward; an item
            // without keys is finished here and never published)
            uint32_t work = blockIdx.x;
            bool more = true;
            for (int n_item = 0, n_clc = 0;;) {
                const int s = n_item & 1, cs = n_clc & 1;
                bool ok = true;
                if (n_item >= 2) ok = mbar_wait(&sm.item_empty[s], ((n_item >> 1) - 1) & 1, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                if (!more) {
                    if (lane == 0) {
                        sm.item[s].T = -1;
                        mbar_arrive(&sm.item_full[s]);
                    }
                    break;
                }
                if (lane == 0) make_item(p, order, work, 0, sm.item[s]);
                __syncwarp();
                if (sm.item[s].T == 0) {
                    const Item &it = sm.item[s];
                    store_zero_rows<128>(it.is_main ? p.dq_main : p.dq_branch, p.accumulate, it.row0, it.rows, it.h0,
                                       min(p.hp, (it.g + 1) * p.group - it.h0), p.h_q, lane);
                } else {
                    if (lane == 0) mbar_arrive(&sm.item_full[s]);
                    ok = mbar_wait(&sm.loads_out, n_item & 1, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    ++n_item;
                }
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
                __syncwarp();
            }
        } else if (warp == 9) {
            // ================================================= TMA producer
            if (lane == 0) {
                const uint32_t q_bytes = (uint32_t)(p.hp * p.tok * 256);
                uint32_t nq = 0, kvi = 0, n_go = 0, n_v = 0;      // items, K tiles, dO tiles, V tiles loaded so far
                bool ok = true;
                for (int it_n = 0; ok; ++it_n) {
                    const int sl = it_n & 1;
                    if (!mbar_wait(&sm.item_full[sl], (it_n >> 1) & 1, abort_flag)) break;
                    const Item &it = sm.item[sl];
                    if (it.T < 0) break;
                    if (it.T > 0) {
                        if (nq > 0 && !(ok = mbar_wait(&sm.q_empty, (nq - 1) & 1, abort_flag))) break;
                        const CUtensorMap *tq = it.is_main ? &tm_q_main : &tm_q_branch;
                        const int off1 = it.is_main ? p.tok : p.off_b;
                        mbar_expect_tx(&sm.q_full, q_bytes * (it.live[0] + it.live[1]));
                        for (int i = 0; i < 2; ++i)
                            if (it.live[i])
                                for (int hf = 0; hf < 2; ++hf)
                                    tma_load_3d(sm.q[i] + hf * 16384, tq, hf * 64, it.h0, it.row0 + (i ? off1 : 0), &sm.q_full);
                        ++nq;
                        for (int j = 0; j < it.T && ok; ++j, ++kvi) {
                            const int nch = tile_chunks(it, j);
                            if (j == max(it.T - 1 - kDqFetchLead, 0)) mbar_arrive(&sm.loads_out);
                            auto load = [&](uint8_t *dst, const CUtensorMap *m128, const CUtensorMap *m32, uint64_t *bar) {
                                mbar_expect_tx(bar, (uint32_t)(nch * 8192));
                                if (j < it.n_full) {
                                    for (int hf = 0; hf < 2; ++hf) tma_load_3d(dst + hf * 16384, m128, hf * 64, it.g, full_row(p, it, j), bar);
                                } else {
                                    for (int c = 0; c < nch; ++c) {
                                        const int row = chunk_row(p, it, 4 * (j - it.n_full) + c);
                                        for (int hf = 0; hf < 2; ++hf) tma_load_3d(dst + hf * 16384 + c * 4096, m32, hf * 64, it.g, row, bar);
                                    }
                                }
                            };
                            const int kb = kvi & 1;
                            if (kvi >= 2 && !(ok = mbar_wait(&sm.k_empty[kb], ((kvi >> 1) - 1) & 1, abort_flag))) break;
                            load(sm.kbuf[kb], &tm_k, &tm_k32, &sm.k_full[kb]);
                            if (j == 0) {
                                if (n_go > 0 && !(ok = mbar_wait(&sm.go_empty, (n_go - 1) & 1, abort_flag))) { ++kvi; break; }
                                mbar_expect_tx(&sm.go_full, q_bytes * (it.live[0] + it.live[1]));
                                const int grow = it.is_main ? it.row0 : qbase + it.row0;
                                for (int i = 0; i < 2; ++i)
                                    if (it.live[i])
                                        for (int hf = 0; hf < 2; ++hf)
                                            tma_load_3d(sm.go[i] + hf * 16384, &tm_go, hf * 64, it.h0, grow + (i ? off1 : 0), &sm.go_full);
                                ++n_go;
                            }
                            if (n_v > 0 && !(ok = mbar_wait(&sm.v_empty, (n_v - 1) & 1, abort_flag))) { ++kvi; break; }
                            load(sm.vbuf, &tm_v, &tm_v32, &sm.v_full);
                            ++n_v;
                        }
                    }
                    mbar_arrive(&sm.item_empty[sl]);
                }
                if (*abort_flag) {
                    // leave no copy in flight behind: wait (bounded) for what was issued
                    auto drain = [&](uint64_t *bar, uint32_t parity) {
                        uint32_t spins = 0;
                        while (!mbar_try_wait(bar, parity) && ++spins < (1u << 22)) {}
                    };
                    for (uint32_t k = kvi > 2 ? kvi - 2 : 0; k < kvi; ++k) drain(&sm.k_full[k & 1], (k >> 1) & 1);
                    if (n_v > 0) drain(&sm.v_full, (n_v - 1) & 1);
                    if (n_go > 0) drain(&sm.go_full, (n_go - 1) & 1);
                    if (nq > 0) drain(&sm.q_full, (nq - 1) & 1);
                }
            }
        } else if (warp == 8) {
            // ================================================= MMA issuer (one elected thread, steps as in the forward)
            if (elect_one()) {
                constexpr uint32_t IDESC_MN = idesc_bf16(128, 128, 1);    // dQ += dS K
                constexpr uint32_t kStep = kTileBytes >> 4;
                const uint32_t q_km = smem_desc_lo(smem_u32(sm.q[0]), 16), go_km = smem_desc_lo(smem_u32(sm.go[0]), 16);
                const uint32_t k_km0 = smem_desc_lo(smem_u32(sm.kbuf[0]), 16), k_mn0 = smem_desc_lo(smem_u32(sm.kbuf[0]), 16384);
                const uint32_t v_km = smem_desc_lo(smem_u32(sm.vbuf), 16);
                auto issue_kmajor = [&](int i, uint32_t a_km, uint32_t b_km, uint32_t idesc, uint64_t *bar) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        mma_ss_lh(tmem + i * 128, a_km + i * kStep + desc_step_kmajor(ks), b_km + desc_step_kmajor(ks), idesc, ks > 0);
                    tc_commit(bar);
                };
                struct Step {
                    uint32_t live;       // bit i: query tile i sees the tile; 0x80: no step
                    uint32_t idesc;      // of S and dP: N = 32 nch
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
                        ok = ok && mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag);
                        if (!ok) { done = true; break; }
                        const Item &im = sm.item[sl];
                        it.T = im.T; it.je = im.je; it.n_full = im.n_full; it.n_ch = im.n_ch;
                        j_cur = 0;
#pragma unroll
                        for (int i = 0; i < 2; ++i) { it.live[i] = im.live[i]; it.va[i] = im.va[i]; it.vb[i] = im.vb[i]; }
                        mbar_arrive(&sm.item_empty[sl]);
                        ++n_item;
                        st.first = true;
                        done = it.T < 0;
                    }
                    st.live = done ? 0x80u : (tile_live(it, 0, j_cur) ? 1u : 0u) | (tile_live(it, 1, j_cur) ? 2u : 0u);
                    st.nch = tile_chunks(it, j_cur);
                    st.idesc = idesc_bf16(128, 0, 0) | ((uint32_t)(st.nch * 4) << 17);
                    st.last = j_cur + 1 >= it.je;
                };
                uint32_t nq = 0, n_go = 0, t = 0;                           // t: steps so far
                uint32_t par = 0, par_o = 0, used_o = 0, started = 0;       // bit i: phase parities of query tile i; dQ_i used
                Step cur, nxt;
                advance(cur);
                if (ok && !done) {
                    ok = mbar_wait(&sm.q_full, 0, abort_flag) && mbar_wait(&sm.k_full[0], 0, abort_flag);
                    nq = 1;
                    if (ok) {
                        tc_fence_after();
                        if (cur.live & 1u) issue_kmajor(0, q_km, k_km0, cur.idesc, &sm.s_full[0]);
                        if (cur.live & 2u) issue_kmajor(1, q_km, k_km0, cur.idesc, &sm.s_full[1]);
                        if (cur.last) tc_commit(&sm.q_empty);
                    }
                }
                for (; ok && cur.live != 0x80u; ++t, cur = nxt) {
                    const int kb = t & 1;
                    const uint32_t k_mn = k_mn0 + kb * kStep, k_next = k_km0 + (kb ^ 1) * kStep;
                    advance(nxt);
                    const bool more = nxt.live != 0x80u;
                    if (ok && cur.first) ok = mbar_wait(&sm.go_full, n_go++ & 1, abort_flag);
                    ok = ok && mbar_wait(&sm.v_full, t & 1, abort_flag);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (!ok) break;
                        if ((cur.live >> i) & 1u) {
                            if (!(ok = mbar_wait(&sm.a_done[i], (par >> i) & 1u, abort_flag))) break;
                            tc_fence_after();
                            issue_kmajor(i, go_km, v_km, cur.idesc, &sm.dp_full[i]);
                        }
                    }
                    if (!ok) break;
                    tc_commit(&sm.v_empty);
                    if (cur.last) tc_commit(&sm.go_empty);
                    if (more) {
                        ok = mbar_wait(&sm.k_full[kb ^ 1], ((t + 1) >> 1) & 1, abort_flag);
                        if (ok && nxt.first) ok = mbar_wait(&sm.q_full, nq & 1, abort_flag);
                        if (!ok) break;
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (!ok) break;
                        if ((cur.live >> i) & 1u) {
                            const bool acc = (started >> i) & 1u;
                            // dQ of the item before has been read out
                            if (!acc && ((used_o >> i) & 1u) && !(ok = mbar_wait(&sm.dq_free[i], ((par_o >> i) & 1u) ^ 1u, abort_flag))) break;
                            if (!(ok = mbar_wait(&sm.b_done[i], (par >> i) & 1u, abort_flag))) break;
                            par ^= 1u << i;
                            tc_fence_after();
                            auto issue_dq = [&](int ks0, bool a) {      // two 16-key steps
#pragma unroll
                                for (int ks = ks0; ks < ks0 + 2; ++ks)
                                    mma_ts_lh(tmem + 256 + i * 128, tmem + i * 128 + ks * 8, k_mn + desc_step_mnmajor(ks), IDESC_MN, a || ks > 0);
                            };
                            issue_dq(0, acc);
                            if (cur.nch > 1) issue_dq(2, true);
                            if (cur.nch > 2) issue_dq(4, true);
                            if (cur.nch > 3) issue_dq(6, true);
                            started |= 1u << i;
                        }
                        if (cur.last && ((started >> i) & 1u)) tc_commit(&sm.dq_full[i]);
                        if (more && ((nxt.live >> i) & 1u)) issue_kmajor(i, q_km, k_next, nxt.idesc, &sm.s_full[i]);
                    }
                    if (!ok) break;
                    tc_commit(&sm.k_empty[kb]);
                    if (more) {
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
        // ================================================= P / dS warps + epilogue
        reg_inc<kDqRegsCompute>();
        const int i = warp >> 2;
        const int r_in = tid & 127;                                // my TMEM lane
        const int my_tok = r_in / p.hp, my_head = r_in % p.hp;     // token and head within the tile
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t r_addr = tmem + lane_base + i * 128;
        const uint32_t dq_addr = tmem + lane_base + 256 + i * 128;
        const float sl2 = p.scale_log2;
        uint32_t n_s = 0, n_o = 0;
        // what this role needs of an item, and this thread's row; the next item is read while dQ of the
        // current one is awaited
        struct Work {
            int T, je, n_full, lo_min, n_mc, n_ch, bs, va, vb, wa, wb, rows, h, my_row, t_rel;
            bool is_main, valid;
            int lo, hi, br_start;
            uint64_t bmask;
            float nl, dl;
        } w, nx;
        auto fetch = [&](int nit, Work &f) -> bool {
            const int sl = nit & 1;
            if (!mbar_wait(&sm.item_full[sl], (nit >> 1) & 1, abort_flag)) return false;
            const Item &im = sm.item[sl];
            f.T = im.T; f.n_full = im.n_full; f.lo_min = im.lo_min; f.n_mc = im.n_mc; f.n_ch = im.n_ch;
            f.bs = im.bs; f.va = im.va[i]; f.vb = im.vb[i]; f.wa = im.wa[i]; f.wb = im.wb[i];
            f.je = im.live[i] ? im.T : 0;
            f.rows = im.rows;
            f.is_main = im.is_main;
            const int off1 = f.is_main ? p.tok : p.off_b;
            f.h = im.h0 + my_head;
            f.valid = my_tok < min(i ? f.rows - off1 : min(off1, f.rows), p.tok) && f.h < (im.g + 1) * p.group;
            f.t_rel = my_tok + (i ? off1 : 0);
            f.my_row = im.row0 + f.t_rel;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.item_empty[sl]);
            f.lo = 1; f.hi = 0; f.br_start = 0; f.bmask = 0;
            f.nl = -INFINITY; f.dl = 0.f;      // dead rows: P = exp2(-inf) = 0
            if (f.T >= 0 && f.valid) {
                const int64_t mrow = f.is_main ? f.my_row : p.meta.n_main + (p.depth ? (int64_t)f.my_row * p.branch_len : f.my_row);
                const size_t srow = (size_t)f.h * p.row_pitch + (f.is_main ? f.my_row : qbase + f.my_row);
                f.lo = p.meta.row_lo[mrow];
                f.hi = p.meta.row_hi[mrow];
                f.nl = p.nlse2_t[srow];
                f.dl = p.delta_t[srow];
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
            const int n_full = w.n_full;
            auto vis = [&](int j, int c) -> uint32_t {
                return w.valid ? chunk_vis(p, j, c, n_full, w.lo_min, w.n_mc, lo, hi, w.bs - w.br_start, w.bmask, w.t_rel, w.rows) : 0u;
            };
            bool started = false;
            for (int j = 0; j < w.je; ++j) {
                if (j < n_full && (j < w.va || j >= w.vb)) continue;      // no row of this tile sees it
                const int nch = j < n_full ? 4 : min(4, w.n_ch - 4 * (j - n_full));
                const bool masked = j >= n_full || j < w.wa || j >= w.wb;
                started = true;
                uint32_t pr[64], ra[32], rb[32];
                // --- phase A: P = exp2(scale_log2 * S - lse2), kept as bf16 pairs
                if (!(ok = mbar_wait(&sm.s_full[i], n_s & 1, abort_flag))) break;
                tc_fence_after();
                // straight-line code for whole tiles (the loads of a chunk run behind the math of the one
                // before); narrow tail tiles go chunk by chunk
                if (nch == 4) {
                    tmem_ld32(r_addr, ra);
                    tmem_ld32(r_addr + 32, rb);
                    tmem_wait_ld();
                    if (!masked) {
                        chunk_p<false>(ra, 0u, sl2, w.nl, &pr[0]);
                        tmem_ld32(r_addr + 64, ra);
                        chunk_p<false>(rb, 0u, sl2, w.nl, &pr[16]);
                        tmem_ld32(r_addr + 96, rb);
                        tmem_wait_ld();
                        chunk_p<false>(ra, 0u, sl2, w.nl, &pr[32]);
                        chunk_p<false>(rb, 0u, sl2, w.nl, &pr[48]);
                    } else {
                        chunk_p<true>(ra, vis(j, 0), sl2, w.nl, &pr[0]);
                        tmem_ld32(r_addr + 64, ra);
                        chunk_p<true>(rb, vis(j, 1), sl2, w.nl, &pr[16]);
                        tmem_ld32(r_addr + 96, rb);
                        tmem_wait_ld();
                        chunk_p<true>(ra, vis(j, 2), sl2, w.nl, &pr[32]);
                        chunk_p<true>(rb, vis(j, 3), sl2, w.nl, &pr[48]);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (c < nch) {
                            tmem_ld32(r_addr + 32 * c, ra);
                            const uint32_t mk = vis(j, c);
                            tmem_wait_ld();
                            chunk_p<true>(ra, mk, sl2, w.nl, &pr[16 * c]);
                        }
                }
                tc_fence_before();
                mbar_arrive(&sm.a_done[i]);
                // --- phase B: dS = P o (dP - delta), bf16, over the first columns
                if (!(ok = mbar_wait(&sm.dp_full[i], n_s & 1, abort_flag))) break;
                ++n_s;
                tc_fence_after();
                {
                    uint32_t pk[16];
                    if (nch == 4) {
                        tmem_ld32(r_addr, ra);
                        tmem_ld32(r_addr + 32, rb);
                        tmem_wait_ld();
                        chunk_ds(ra, &pr[0], w.dl, pk);
                        tmem_st16(r_addr, pk);
                        tmem_ld32(r_addr + 64, ra);
                        chunk_ds(rb, &pr[16], w.dl, pk);
                        tmem_st16(r_addr + 16, pk);
                        tmem_ld32(r_addr + 96, rb);
                        tmem_wait_ld();
                        chunk_ds(ra, &pr[32], w.dl, pk);
                        tmem_st16(r_addr + 32, pk);
                        chunk_ds(rb, &pr[48], w.dl, pk);
                        tmem_st16(r_addr + 48, pk);
                    } else {
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            if (c < nch) {
                                tmem_ld32(r_addr + 32 * c, ra);
                                tmem_wait_ld();
                                chunk_ds(ra, &pr[16 * c], w.dl, pk);
                                tmem_st16(r_addr + 16 * c, pk);
                            }
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&sm.b_done[i]);
            }
            if (!ok) break;
            if (!(ok = fetch(nit + 1, nx))) break;
            // --- epilogue: dQ = scale * accumulator
            if (started) {
                if (!(ok = mbar_wait(&sm.dq_full[i], n_o & 1, abort_flag))) break;
                ++n_o;
                tc_fence_after();
            }
            void *dst = w.is_main ? p.dq_main : p.dq_branch;
            const size_t base = ((size_t)w.my_row * p.h_q + w.h) * 128;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                uint32_t r[32];
                if (started) {
                    tmem_ld32(dq_addr + c * 32, r);
                    tmem_wait_ld();
                    if (c == 3) {
                        tc_fence_before();
                        mbar_arrive(&sm.dq_free[i]);   // the next item's dS K may overwrite dQ_i
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) r[e] = 0u;
                }
                if (w.valid) {
                    if (p.accumulate) store_grad_chunk<true>(dst, base + c * 32, r, p.scale);
                    else store_grad_chunk<false>(dst, base + c * 32, r, p.scale, p.wide);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
    if (tid == 0 && sm.abort_flag) atomicExch(p.status, BA_ETIMEOUT);
}


// ============================================================================
// head_dim 64: 64-row streamed tiles, dQ and dK/dV
// ============================================================================
// A CTA keeps 128 stationary rows (pair st1, st2) in shared memory and their gradients (fp32) in TMEM and
// walks the rows of the other side that can see them, or that they see, as 64-row tiles (pair x1, x2):
//   dK/dV  stationary K_j, V_j (128 keys of one KV head); streamed Q, dO of every query head of the group.
//          Everything is transposed so that the key is the TMEM lane: S^T = K_j Q^T, dP^T = V_j dO^T.
//   dQ     stationary Q, dO (128 (token, head) rows of one KV head's group, head fastest); streamed K, V.
//   S = st1 x1^T, dP = st2 x2^T (128 x 64), P = exp2(scale_log2 S - lse2), dS = P o (dP - delta),
//   acc1 += dS x1 (dK / dQ), acc2 += P x2 (dV); P, dS are TMEM A operands.
// Two tiles are in flight (sets 0 / 1, one P / dS warpgroup each).  CTAs fetch further items as in the forward: the
// next stationary pair is loaded and its first S, dP formed behind the last steps and the output of the current
// item (dQ of the batch below 285 -> 205 us).
//   TMEM: acc1 [0,64) acc2 [64,128); set b: XS_b = 256 + 128 b (64 cols: S, its first 32 columns then hold P as
//   bf16), XD_b = XS_b + 64 (dP, then dS); P_lo, dS_lo of set b in 32 columns each from 128 + 64 b.
// This runs in place of plain-FMA kernels that kept P and dS in fp32.  P and dS go in as bf16 pairs hi + lo (16
// bits of mantissa), two products each: against fp64, gradients rounded to bf16 are then off by what those kernels'
// are (dQ, dK, dV 1.64e-3 .. 1.66e-3 in the 2-norm, the same to 1 part in 10,000).  Gradients accumulated in fp32
// would not be, so they stay with those kernels (ba_use_tc).  4,096 tokens, 6 sequences, chains of three, 32/8 heads:
// dQ / dK/dV 187 / 287 us (were 3052 / 8978).  The 128-row tiles of ba_tc_dkdv.cu took 359 us for that dK/dV when this
// form, then without an order of the tiles, took 336: twice the conversions per flop make the warps the limit, and two tiles in flight hide them better.
// dQ is here and not in tc_dq_kernel because that kernel was written for 128 columns of dQ and keeps P
// in registers as bf16; a form of it with hi + lo pairs has not been tried.
//
// Key tiles of dK/dV differ in length (causal) and are few in small batches: the CTAs of a cluster then share
// a main key tile, each walks a contiguous part of its (head, row tile) steps, and the parts are summed through
// distributed shared memory in rank order (one owner per output element, bit-reproducible).
constexpr int kKvThreads = 384;
constexpr int kKvRegsCompute = 208, kKvRegsIssue = 88, kKvRegsLaunch = 168;
static_assert(256 * kKvRegsCompute + 128 * kKvRegsIssue <= kKvThreads * kKvRegsLaunch, "register re-split exceeds what the CTA owns");
constexpr int kSub = 64;           // streamed rows per tile
constexpr int kQStages = 4;

enum { kModeDkdv = 0, kModeDq = 1 };

struct SubMeta {
    float neg_lse2[kSub];
    float delta[kSub];
    int bstart[kSub];
    unsigned long long mask[kSub];
};

// What every role knows about one stationary tile.
struct KvItem {
    int n_iter;                  // steps (head, streamed tile) of this CTA; -1: no more work
    int n_sub, n_sub_main;       // streamed tiles per head: main part, then branch part
    int s_beg, hh_beg;           // first step: streamed tile and head
    int is_main, g, h0;
    int row0, row_end;           // stationary rows in the numbering of their part
    int srow0;                   // first stationary row in its tensor (K, V rows / rows of dO)
    int m0, m1, b0, b1;          // streamed rows: main part and branch part
    int ma, ba;                  // first rows of the two parts' tiles
};

constexpr int kD = 64;
struct KvSmem {
    static constexpr uint32_t kStatBytes = kTile * kD * 2, kSubBytes = kSub * kD * 2;
    alignas(1024) uint8_t st1[kStatBytes];
    alignas(1024) uint8_t st2[kStatBytes];
    alignas(1024) uint8_t xs[kQStages][2 * kSubBytes];  // x1 tile, then x2 tile
    alignas(16) SubMeta meta[kQStages];
    alignas(16) uint4 clc[2];
    KvItem item[2];
    alignas(8) uint64_t st_full, st_empty;
    uint64_t x_full[kQStages], x_empty[kQStages];
    uint64_t sd_full[2], pd_done[2], acc_full, acc_free;
    uint64_t item_full[2], item_empty[2], clc_full[2], loads_out;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(KvSmem) <= 232448, "shared memory of the head_dim 64 backward");
static_assert(kQStages * 2 * kSub * 2 == 2 * kTile * 4, "a cluster's partial accumulators fill the streamed stages exactly");

// 16 columns of a tile: P and dS as 8 packed bf16 pairs each, and the pairs of what rounding left;
// COLS: nl / dl point at the columns' -lse2 and delta in shared memory, otherwise they are the row's own
template <bool MASKED, bool COLS>
__device__ __forceinline__ void quarter_pds(const uint32_t (&rs)[16], const uint32_t (&rd)[16], uint32_t mk, float sl2,
                                            const float *nl, const float *dl, float row_nl, float row_dl,
                                            uint32_t (&pk)[8], uint32_t (&dk8)[8], uint32_t (&pl)[8], uint32_t (&dl8)[8]) {
    const float2 s2 = make_float2(sl2, sl2);
    const float4 *nl4 = reinterpret_cast<const float4 *>(nl);
    const float4 *dl4 = reinterpret_cast<const float4 *>(dl);
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
        const float4 nv = COLS ? nl4[e >> 2] : make_float4(row_nl, row_nl, row_nl, row_nl);
        const float4 dv = COLS ? dl4[e >> 2] : make_float4(row_dl, row_dl, row_dl, row_dl);
        const float2 x0 = ffma2(make_float2(__uint_as_float(rs[e]), __uint_as_float(rs[e + 1])), s2,
                                make_float2(nv.x, nv.y));
        const float2 x1 = ffma2(make_float2(__uint_as_float(rs[e + 2]), __uint_as_float(rs[e + 3])), s2,
                                make_float2(nv.z, nv.w));
        float2 p0 = make_float2(ex2(x0.x), ex2(x0.y)), p1 = make_float2(ex2(x1.x), ex2(x1.y));
        if (MASKED) {
            p0.x = ((mk >> e) & 1u) ? p0.x : 0.f;
            p0.y = ((mk >> (e + 1)) & 1u) ? p0.y : 0.f;
            p1.x = ((mk >> (e + 2)) & 1u) ? p1.x : 0.f;
            p1.y = ((mk >> (e + 3)) & 1u) ? p1.y : 0.f;
        }
        float2 d0 = fmul2(p0, fadd2(make_float2(__uint_as_float(rd[e]), __uint_as_float(rd[e + 1])),
                                    make_float2(-dv.x, -dv.y)));
        float2 d1 = fmul2(p1, fadd2(make_float2(__uint_as_float(rd[e + 2]), __uint_as_float(rd[e + 3])),
                                    make_float2(-dv.z, -dv.w)));
        if (MASKED) {  // the scalars of invisible columns may be anything, even NaN
            d0.x = ((mk >> e) & 1u) ? d0.x : 0.f;
            d0.y = ((mk >> (e + 1)) & 1u) ? d0.y : 0.f;
            d1.x = ((mk >> (e + 2)) & 1u) ? d1.x : 0.f;
            d1.y = ((mk >> (e + 3)) & 1u) ? d1.y : 0.f;
        }
        const int q = e >> 1;
        pk[q] = pack_bf16(p0.x, p0.y);
        pk[q + 1] = pack_bf16(p1.x, p1.y);
        dk8[q] = pack_bf16(d0.x, d0.y);
        dk8[q + 1] = pack_bf16(d1.x, d1.y);
        pl[q] = bf16_rest(p0, pk[q]);
        pl[q + 1] = bf16_rest(p1, pk[q + 1]);
        dl8[q] = bf16_rest(d0, dk8[q]);
        dl8[q + 1] = bf16_rest(d1, dk8[q + 1]);
    }
}

// bits [sh, sh + 64) of a 64-bit mask (sh may be negative)
__device__ __forceinline__ uint64_t shift_mask(uint64_t m, int sh) {
    if (sh >= 0) return sh < 64 ? m >> sh : 0ull;
    return sh > -64 ? m << -sh : 0ull;
}

// Rows of one call are ordered by position (main) or anchor (branches), so the ranges of a tile are those of its
// first and last row.
template <int MODE> __device__ void make_kv_item(const TcBwdParams &p, const BaOrder &order, uint32_t work, int rank, KvItem &it) {
    constexpr bool kDq = MODE == kModeDq;
    const int n = (int)p.meta.n_main, S = p.splits;
    int tile;
    // Heaviest first: earlier keys (more viewers), later query rows (longer prefixes)
    if (kDq) {
        const int per = p.h_kv * p.head_chunks;
        tile = order.n > 0 ? order.tile[work / per] : p.total_tiles - 1 - (int)(work / per);
        it.g = (int)(work % per) / p.head_chunks;
        it.h0 = it.g * p.group + (int)(work % p.head_chunks) * p.hp;
    } else {
        it.h0 = 0;
        if (p.tile_major) {
            tile = order.n > 0 ? order.tile[work / p.h_kv] : (int)(work / p.h_kv);
            it.g = (int)(work % p.h_kv);
        } else {
            // KV-head-major: the CTAs running at one time belong to one or two KV heads and stream the same
            // query rows, so that stream is read from HBM about once per head instead of once per wave
            it.g = (int)(work / p.total_key_tiles);
            tile = (int)(work % p.total_key_tiles);
        }
    }
    const bool is_main = tile < (kDq ? p.main_tiles : p.main_key_tiles);
    it.is_main = is_main;
    int step;
    if (kDq) {
        step = p.tok;
        it.row0 = is_main ? (int)p.r.qm_begin + tile * step : (int)p.r.tok_begin + (tile - p.main_tiles) * step;
        it.row_end = min(it.row0 + step, (int)(is_main ? p.r.qm_end : p.r.tok_end));
    } else {
        int bt = tile - p.main_key_tiles;
        if (!is_main && S > 1) bt = bt * S + rank;           // a cluster holds S branch key tiles
        const bool past = !is_main && bt >= p.branch_key_tiles;      // the last cluster has ranks to spare: no rows
        step = is_main ? kTile : p.step_kb;
        it.row0 = is_main ? (int)p.r.kv_begin + tile * step : (int)p.r.tok_begin + bt * step;
        it.row_end = past ? it.row0 : min(it.row0 + step, (int)(is_main ? p.r.kv_end : p.r.tok_end));
    }
    it.srow0 = is_main ? it.row0 - (kDq ? 0 : (int)p.r.kv_base) : n + it.row0;
    it.m0 = it.m1 = it.b0 = it.b1 = 0;
    const int first = it.row0, last = it.row_end - 1;
    if (last >= first) {
        if (kDq) {
            const int64_t gf = is_main ? first : (int64_t)n + first, gl = is_main ? last : (int64_t)n + last;
            if (p.r.parts & BA_PART_MAIN) {
                it.m0 = max(p.meta.row_lo[gf], (int)p.r.kv_begin);
                it.m1 = min(p.meta.row_hi[gl], (int)p.r.kv_end - 1) + 1;
            }
            if (!is_main && (p.r.parts & BA_PART_BRANCH)) { it.b0 = p.meta.br_start[first]; it.b1 = p.meta.br_end[last]; }
        } else {
            if (is_main) {
                if (p.has_main_q) {
                    it.m0 = max(first, (int)p.r.qm_begin);
                    it.m1 = min(p.meta.key_qend[last], (int)p.r.qm_end);
                }
                it.b0 = p.meta.key_bq_begin[first];
                it.b1 = p.meta.key_bq_end[last];
            } else {
                it.b0 = p.meta.br_start[first];
                it.b1 = p.meta.br_end[last];
            }
            it.b0 = max(it.b0, (int)p.r.tok_begin);
            it.b1 = min(it.b1, (int)p.r.tok_end);
        }
    }
    // In dK/dV the streamed tiles start at ma / ba: the parts' starts moved back (by < 4 rows) so that every
    // tile's first row is a multiple of 4 in the row numbering of the per-row scalars, whose bulk copies are then
    // 16-byte aligned.  The extra leading rows are masked like any other invisible row.
    it.ma = kDq ? it.m0 : it.m0 & ~3;
    it.ba = kDq ? it.b0 : ((n + it.b0) & ~3) - n;   // may be as low as -3
    it.n_sub_main = it.m1 > it.m0 ? (it.m1 - it.ma + kSub - 1) / kSub : 0;
    it.n_sub = it.n_sub_main + (it.b1 > it.b0 ? (it.b1 - it.ba + kSub - 1) / kSub : 0);
    const int n_all = it.n_sub * (kDq ? 1 : p.group);
    const bool part = S > 1 && is_main;
    const int t_beg = part ? (int)((int64_t)n_all * rank / S) : 0;
    it.n_iter = (part ? (int)((int64_t)n_all * (rank + 1) / S) : n_all) - t_beg;
    it.s_beg = it.n_sub > 0 ? t_beg % it.n_sub : 0;
    it.hh_beg = it.n_sub > 0 ? t_beg / it.n_sub : 0;
}

template <int MODE, bool SPLIT>
__global__ void __launch_bounds__(kKvThreads, 1)
tc_kv_kernel(const __grid_constant__ CUtensorMap tm_q_main, const __grid_constant__ CUtensorMap tm_q_branch,
             const __grid_constant__ CUtensorMap tm_go, const __grid_constant__ CUtensorMap tm_k,
             const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_go_branch,
             const __grid_constant__ TcBwdParams p, const __grid_constant__ BaOrder order) {
    using Smem = KvSmem;
    constexpr bool kDq = MODE == kModeDq;
    constexpr int D = kD;
    constexpr uint32_t kSubBytes = Smem::kSubBytes;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &sm.abort_flag;
    constexpr long long kLimit = kSlowWaitLimitCycles;
    if (smem_u32(smem_raw) & 1023u) {   // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicExch(p.status, BA_EUNSUPPORTED);
        return;
    }
    const int S = SPLIT ? p.splits : 1, rank = SPLIT ? (int)(blockIdx.x % S) : 0;
    const int n = (int)p.meta.n_main;      // global row number of branch row 0

    if (tid == 0) {
        mbar_init(&sm.st_full, 1); mbar_init(&sm.st_empty, 1);
        for (int s = 0; s < kQStages; ++s) { mbar_init(&sm.x_full[s], kDq ? 1 : 2); mbar_init(&sm.x_empty[s], 1); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sm.sd_full[b], 1);
            mbar_init(&sm.pd_done[b], 128);
            mbar_init(&sm.item_full[b], 1);
            mbar_init(&sm.item_empty[b], 10);   // producer, MMA thread, one lane of each P / dS warp
            mbar_init(&sm.clc_full[b], 1);
        }
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
    bool shared_tile = false;      // SPLIT: this CTA walked a part of a main key tile
    if (kDq) wait_prerequisites();      // launched while delta ends

    if (warp >= 8) {
        reg_dec<kKvRegsIssue>();
        if (warp == 10) {
            // ================================================= work fetcher (whole warp, as in the forward; an item
            // without steps is finished here and never published)
            uint32_t work = SPLIT ? blockIdx.x / S : blockIdx.x;
            bool more = true;
            for (int n_item = 0, n_clc = 0;;) {
                const int s = n_item & 1, cs = n_clc & 1;
                bool ok = true;
                if (n_item >= 2) ok = mbar_wait(&sm.item_empty[s], ((n_item >> 1) - 1) & 1, abort_flag, kLimit);
                if (!__all_sync(0xffffffffu, ok)) break;
                if (!more) {
                    if (lane == 0) {
                        sm.item[s].n_iter = -1;
                        mbar_arrive(&sm.item_full[s]);
                    }
                    break;
                }
                if (lane == 0) make_kv_item<MODE>(p, order, work, rank, sm.item[s]);
                __syncwarp();
                if (!SPLIT && sm.item[s].n_iter == 0) {
                    const KvItem &it = sm.item[s];
                    const int rows = it.row_end - it.row0;
                    if (kDq) {
                        store_zero_rows<D>(it.is_main ? p.dq_main : p.dq_branch, 0, it.row0, rows, it.h0,
                                         min(p.hp, (it.g + 1) * p.group - it.h0), p.h_q, lane);
                    } else {
                        store_zero_rows<D>(p.dk, 0, it.srow0, rows, it.g, 1, p.h_kv, lane);
                        store_zero_rows<D>(p.dv, 0, it.srow0, rows, it.g, 1, p.h_kv, lane);
                    }
                } else {
                    if (lane == 0) mbar_arrive(&sm.item_full[s]);
                    if (!SPLIT) ok = mbar_wait(&sm.loads_out, n_item & 1, abort_flag, kLimit);
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
            // ================================================= producer (whole warp)
            bool ok = true;
            uint32_t t = 0, n_st = 0;      // streamed tiles and stationary tiles loaded so far
            for (int n_item = 0; ok; ++n_item) {
                const int sl = n_item & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag, kLimit));
                if (!ok) break;
                const KvItem it = sm.item[sl];
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.item_empty[sl]);
                if (it.n_iter < 0) break;
                if (it.n_iter == 0) continue;
                int hh = it.hh_beg, s = it.s_beg;  // step = hh * n_sub + s
                // the query stream comes from HBM: ask for tile i + kPrefetch to be brought into L2 while tile i is loaded
                constexpr int kPrefetch = 16;
                int ph = hh, ps = s;
                for (int i = 0; i < kPrefetch; ++i)
                    if (++ps == it.n_sub) { ps = 0; ++ph; }
                for (int i = 0; i < it.n_iter; ++i, ++t) {
                    const int st = t % kQStages;
                    if (t >= (uint32_t)kQStages) ok = mbar_wait(&sm.x_empty[st], ((t / kQStages) - 1) & 1, abort_flag, kLimit);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (lane == 0 && i == max(it.n_iter - 1 - kKvFetchLead, 0)) mbar_arrive(&sm.loads_out);
                    const bool seg_main = s < it.n_sub_main;
                    const int r0 = seg_main ? it.ma + s * kSub : it.ba + (s - it.n_sub_main) * kSub;
                    SubMeta &mt = sm.meta[st];
                    if (kDq) {
                        if (lane == 0) {
                            const int kr = seg_main ? r0 - (int)p.r.kv_base : (int)p.meta.n_main + r0;
                            mbar_expect_tx(&sm.x_full[st], 2 * kSubBytes);
                            tma_load_3d(sm.xs[st], &tm_k, 0, it.g, kr, &sm.x_full[st]);
                            tma_load_3d(sm.xs[st] + kSubBytes, &tm_v, 0, it.g, kr, &sm.x_full[st]);
                        }
                    } else {
                        const int h = it.g * p.group + hh;
                        const int gr0 = seg_main ? r0 : n + r0;
                        if (lane == 0) {
                            // a branch tile may start up to three rows before branch row 0: dO by the map that has no rows there
                            const CUtensorMap *tq = seg_main ? &tm_q_main : &tm_q_branch, *tg = r0 >= 0 ? &tm_go : &tm_go_branch;
                            mbar_expect_tx(&sm.x_full[st], 2 * kSubBytes + 2 * kSub * 4);
                            tma_load_3d(sm.xs[st], tq, 0, h, r0, &sm.x_full[st]);
                            tma_load_3d(sm.xs[st] + kSubBytes, tg, 0, h, r0 >= 0 ? gr0 : r0, &sm.x_full[st]);
                            const size_t off = (size_t)h * p.row_pitch + gr0;
                            bulk_load(mt.neg_lse2, p.nlse2_t + off, kSub * 4, &sm.x_full[st]);
                            bulk_load(mt.delta, p.delta_t + off, kSub * 4, &sm.x_full[st]);
                            if (i + kPrefetch < it.n_iter) {
                                const int h2 = it.g * p.group + ph;
                                const bool main2 = ps < it.n_sub_main;
                                const int r2 = main2 ? it.ma + ps * kSub : it.ba + (ps - it.n_sub_main) * kSub;
                                const int g2 = main2 ? r2 : n + r2;
                                const CUtensorMap *tq2 = main2 ? &tm_q_main : &tm_q_branch;
                                tma_prefetch_3d(tq2, 0, h2, r2);
                                tma_prefetch_3d(&tm_go, 0, h2, g2);
                                const size_t off2 = (size_t)h2 * p.row_pitch + g2;
                                bulk_prefetch(p.nlse2_t + off2, kSub * 4);
                                bulk_prefetch(p.delta_t + off2, kSub * 4);
                            }
                        }
                        if (!it.is_main) {
                            // own-branch tiles: branch start and mask of each query token
                            for (int c = lane; c < kSub; c += 32) {
                                const int tok = r0 + c;
                                const bool live = tok >= it.b0 && tok < it.b1;
                                mt.bstart[c] = live ? p.meta.br_start[tok] : 0;
                                mt.mask[c] = live ? p.meta.br_mask[tok] : 0ull;
                            }
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sm.x_full[st]);  // second arrival: plain stores are in place
                    }
                    if (i == 0) {
                        // the stationary pair, once the last S, dP of the item before have been formed
                        if (n_st > 0) ok = mbar_wait(&sm.st_empty, (n_st - 1) & 1, abort_flag, kLimit);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) { ++t; break; }
                        if (lane == 0) {
                            if (kDq) {
                                const CUtensorMap *tq = it.is_main ? &tm_q_main : &tm_q_branch;
                                mbar_expect_tx(&sm.st_full, (uint32_t)(2 * p.hp * p.tok * D * 2));
                                tma_load_3d(sm.st1, tq, 0, it.h0, it.row0, &sm.st_full);
                                tma_load_3d(sm.st2, &tm_go, 0, it.h0, it.srow0, &sm.st_full);
                            } else {
                                mbar_expect_tx(&sm.st_full, 2 * Smem::kStatBytes);
                                tma_load_3d(sm.st1, &tm_k, 0, it.g, it.srow0, &sm.st_full);
                                tma_load_3d(sm.st2, &tm_v, 0, it.g, it.srow0, &sm.st_full);
                            }
                        }
                        ++n_st;
                    }
                    if (++ps == it.n_sub) { ps = 0; ++ph; }
                    if (++s == it.n_sub) { s = 0; ++hh; }
                }
            }
            if (*abort_flag && lane == 0) {
                // leave no copy in flight behind: wait (bounded) for what was issued
                for (uint32_t k = t > (uint32_t)kQStages ? t - kQStages : 0; k < t; ++k) {
                    uint32_t spins = 0;
                    while (!mbar_try_wait(&sm.x_full[k % kQStages], (k / kQStages) & 1) && ++spins < (1u << 22)) {}
                }
                if (n_st > 0) {
                    uint32_t spins = 0;
                    while (!mbar_try_wait(&sm.st_full, (n_st - 1) & 1) && ++spins < (1u << 22)) {}
                }
            }
        } else if (warp == 8) {
            // ================================================= MMA issuer (one elected thread)
            if (elect_one()) {
                constexpr uint32_t IDESC_T = idesc_bf16(128, kSub, 0);   // 128 x 64, K = D
                constexpr uint32_t IDESC_ACC = idesc_bf16(128, D, 1);    // 128 x D, K = 64 rows
                // low descriptor words; a stage holds the x1 tile, then the x2 tile, each in 64-column halves of 8 KB
                const uint32_t st1_km = smem_desc_lo(smem_u32(sm.st1), 16), st2_km = smem_desc_lo(smem_u32(sm.st2), 16);
                const uint32_t xs_km0 = smem_desc_lo(smem_u32(sm.xs[0]), 16), xs_mn0 = smem_desc_lo(smem_u32(sm.xs[0]), 8192);
                constexpr uint32_t kStageStep = (2 * kSubBytes) >> 4, kHalfStage = kSubBytes >> 4;
                auto issue_t = [&](uint32_t d_tmem, uint32_t a_km, uint32_t b_km) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        mma_ss_lh(d_tmem, a_km + desc_step_kmajor(ks), b_km + (uint32_t)((ks >> 2) * 512 + (ks & 3) * 2), IDESC_T, ks > 0);
                };
                auto issue_acc = [&](uint32_t d_tmem, uint32_t a_tmem, uint32_t b_mn, bool accumulate) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_ts_lh(d_tmem, a_tmem + ks * 8, b_mn + desc_step_mnmajor(ks), IDESC_ACC, accumulate || ks > 0);
                };
                // The steps of successive items form one stream: S, dP of step t + 2 are formed after the
                // accumulation of step t, whichever item they belong to.
                struct Step { bool valid, first, last; };
                int n_item = 0, left = 0;
                bool ok = true, done = false;
                auto advance = [&](Step &x) {
                    x.first = false;
                    while (left == 0 && !done) {
                        const int sl = n_item & 1;
                        ok = ok && mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag, kLimit);
                        if (!ok) { done = true; break; }
                        left = sm.item[sl].n_iter;
                        mbar_arrive(&sm.item_empty[sl]);
                        ++n_item;
                        x.first = true;
                        if (left < 0) { done = true; left = 0; }
                    }
                    x.valid = !done;
                    --left;
                    x.last = left == 0;
                };
                uint32_t n_st = 0, n_acc = 0;
                auto issue_sd = [&](const Step &x, uint32_t t) {
                    const uint32_t km = xs_km0 + (t % kQStages) * kStageStep, xs = tmem + 256 + (t & 1) * 128;
                    if (x.first) ok = mbar_wait(&sm.st_full, n_st++ & 1, abort_flag, kLimit);
                    if (!ok) return;
                    tc_fence_after();
                    issue_t(xs, st1_km, km);                        // S
                    issue_t(xs + 64, st2_km, km + kHalfStage);      // dP
                    tc_commit(&sm.sd_full[t & 1]);
                    if (x.last) tc_commit(&sm.st_empty);
                };
                Step s0, s1, s2;
                advance(s0);
                if (s0.valid && ok && (ok = mbar_wait(&sm.x_full[0], 0, abort_flag, kLimit))) issue_sd(s0, 0);
                s1.valid = false;
                if (s0.valid && ok) {
                    advance(s1);
                    if (s1.valid && ok && (ok = mbar_wait(&sm.x_full[1], 0, abort_flag, kLimit))) issue_sd(s1, 1);
                }
                for (uint32_t t = 0; ok && s0.valid; ++t, s0 = s1, s1 = s2) {
                    const int b = t & 1;
                    const uint32_t stage_mn = xs_mn0 + (t % kQStages) * kStageStep, xs = tmem + 256 + b * 128;
                    s2.valid = false;
                    if (s1.valid) advance(s2);
                    if (ok && s2.valid) ok = mbar_wait(&sm.x_full[(t + 2) % kQStages], ((t + 2) / kQStages) & 1, abort_flag, kLimit);
                    // the accumulators of the item before have been read out
                    if (ok && s0.first && n_acc > 0) ok = mbar_wait(&sm.acc_free, (n_acc - 1) & 1, abort_flag, kLimit);
                    if (ok) ok = mbar_wait(&sm.pd_done[b], (t >> 1) & 1, abort_flag, kLimit);
                    if (!ok) break;
                    tc_fence_after();
                    if (!kDq) issue_acc(tmem + D, xs, stage_mn + kHalfStage, !s0.first);     // dV += P^T dO
                    issue_acc(tmem, xs + 64, stage_mn, !s0.first);                           // dK += dS^T Q / dQ += dS K
                    if (!kDq) issue_acc(tmem + D, tmem + 128 + b * 64, stage_mn + kHalfStage, true);         // + P_lo, dS_lo
                    issue_acc(tmem, tmem + 128 + b * 64 + 32, stage_mn, true);
                    tc_commit(&sm.x_empty[t % kQStages]);
                    if (s0.last) {
                        tc_commit(&sm.acc_full);
                        ++n_acc;
                    }
                    if (s2.valid) issue_sd(s2, t + 2);
                }
            }
            __syncwarp();
        }
    } else {
        // ================================================= P / dS warps + epilogue
        reg_inc<kKvRegsCompute>();
        const int b = warp >> 2;
        const int r_in = tid & 127;
        const int my_tok = kDq ? r_in / p.hp : r_in, my_head = kDq ? r_in % p.hp : 0;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t xs_addr = tmem + lane_base + 256 + b * 128;
        const uint32_t xd_addr = xs_addr + 64;
        const uint32_t lo_addr = tmem + lane_base + 128 + b * 64;
        const float sl2 = p.scale_log2;
        // what this role needs of an item, and this thread's stationary row; the next item is read while the
        // accumulators of the current one are awaited
        struct Work {
            int n_iter, n_sub, n_sub_main, s_beg, g, row0, row_end, srow, m0, m1, b0, b1, ma, ba, row, h;
            bool is_main, valid;
            int lo, hi, rb0, rb1;        // main range (keys / query rows) and branch range of my row
            uint64_t mask;
            float nl, dl;
        } w, nx;
        auto fetch = [&](int n_item, Work &f) -> bool {
            const int sl = n_item & 1;
            if (!mbar_wait(&sm.item_full[sl], (n_item >> 1) & 1, abort_flag, kLimit)) return false;
            const KvItem &im = sm.item[sl];
            f.n_iter = im.n_iter; f.n_sub = im.n_sub; f.n_sub_main = im.n_sub_main; f.s_beg = im.s_beg; f.g = im.g;
            f.row0 = im.row0; f.row_end = im.row_end; f.srow = im.srow0 + r_in;
            f.m0 = im.m0; f.m1 = im.m1; f.b0 = im.b0; f.b1 = im.b1; f.ma = im.ma; f.ba = im.ba;
            f.is_main = im.is_main;
            f.h = im.h0 + my_head;
            f.row = im.row0 + my_tok;
            f.valid = f.row < f.row_end && (!kDq || (my_tok < p.tok && f.h < (f.g + 1) * p.group));
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.item_empty[sl]);
            f.lo = 1; f.hi = 0; f.rb0 = f.rb1 = 0; f.mask = 0;
            f.nl = -INFINITY; f.dl = 0.f;        // dead rows of dQ: P = exp2(-inf) = 0
            if (f.n_iter > 0 && f.valid) {
                if (kDq) {
                    const int64_t gr = f.is_main ? f.row : (int64_t)p.meta.n_main + f.row;
                    if (p.r.parts & BA_PART_MAIN) {
                        f.lo = max(p.meta.row_lo[gr], (int)p.r.kv_begin);
                        f.hi = min(p.meta.row_hi[gr], (int)p.r.kv_end - 1);
                    }
                    if (!f.is_main && (p.r.parts & BA_PART_BRANCH)) {
                        f.rb0 = p.meta.br_start[f.row];
                        f.mask = p.meta.br_mask[f.row];
                    }
                    f.nl = p.nlse2_t[(size_t)f.h * p.row_pitch + gr];
                    f.dl = p.delta_t[(size_t)f.h * p.row_pitch + gr];
                } else if (f.is_main) {
                    f.lo = f.row;
                    f.hi = p.meta.key_qend[f.row] - 1;
                    f.rb0 = p.meta.key_bq_begin[f.row];
                    f.rb1 = p.meta.key_bq_end[f.row];
                } else {
                    f.rb0 = p.meta.br_start[f.row];
                    f.rb1 = p.meta.br_end[f.row];
                }
            }
            return true;
        };
        uint32_t t0 = 0, n_acc = 0;      // steps and accumulations before this item
        bool ok = fetch(0, nx);
        for (int n_item = 0; ok; ++n_item) {
            w = nx;
            if (w.n_iter < 0) break;
            int s = w.s_beg + (int)((b - t0) & 1u);      // streamed tile of my next step within its head
            while (w.n_iter > 0 && s >= w.n_sub) s -= w.n_sub;
            for (uint32_t t = t0 + ((b - t0) & 1u); t < t0 + (uint32_t)w.n_iter; t += 2) {
                const int st = t % kQStages;
                const bool seg_main = s < w.n_sub_main;
                const int r0 = seg_main ? w.ma + s * kSub : w.ba + (s - w.n_sub_main) * kSub;
                const SubMeta &mt = sm.meta[st];
                s += 2;
                while (s >= w.n_sub) s -= w.n_sub;
                // --- which of the 64 streamed rows (columns) my row sees, or is seen by (needs only the
                // stage's scalars, so it runs while the MMAs are still in flight)
                if (!kDq) {
                    ok = mbar_wait(&sm.x_full[st], (t / kQStages) & 1, abort_flag, kLimit);
                    if (!ok) break;
                }
                uint64_t vis = 0ull;
                if (w.valid) {
                    if (kDq) {
                        vis = seg_main ? bit_range(w.lo - r0, w.hi - r0) : shift_mask(w.mask, r0 - w.rb0);
                    } else if (w.is_main) {
                        // main rows: same sequence, causal: key <= row < end of the key's sequence; branch tokens
                        // anchored at or after the key, inside its sequence
                        const int v0 = seg_main ? w.lo : w.rb0, v1 = seg_main ? w.hi + 1 : w.rb1;
                        const int rbeg = seg_main ? w.m0 : w.b0, rend = seg_main ? w.m1 : w.b1;
                        vis = bit_range(max(v0, rbeg) - r0, min(v1, rend) - 1 - r0);
                    } else {
                        // own-branch tokens whose mask has my bit
                        const int lo_c = max(max(w.rb0, w.b0) - r0, 0), hi_c = min(min(w.rb1, w.b1) - 1 - r0, kSub - 1);
                        for (int c = lo_c; c <= hi_c; ++c) {
                            const int rel = w.row - mt.bstart[c];
                            if (rel >= 0 && rel < 64 && ((mt.mask[c] >> rel) & 1ull)) vis |= 1ull << c;
                        }
                    }
                }
                const bool masked = !__all_sync(0xffffffffu, vis == ~0ull);
                ok = mbar_wait(&sm.sd_full[b], (t >> 1) & 1, abort_flag, kLimit);
                if (!ok) break;
                tc_fence_after();
                // --- P, dS 16 columns at a time, the next pair of loads in flight behind the math
                {
                    uint32_t sa[16], da[16], sb[16], db[16], pk[8], dk8[8], pl[8], dl8[8];
                    auto quarters = [&](auto msk) {
                        constexpr bool MASKED = decltype(msk)::value;
                        auto quarter = [&](const uint32_t (&rs)[16], const uint32_t (&rd)[16], int q) {
                            quarter_pds<MASKED, !kDq>(rs, rd, (uint32_t)(vis >> (16 * q)) & 0xffffu, sl2, mt.neg_lse2 + 16 * q,
                                                           mt.delta + 16 * q, w.nl, w.dl, pk, dk8, pl, dl8);
                            if (!kDq) tmem_st8(xs_addr + 8 * q, pk);
                            tmem_st8(xd_addr + 8 * q, dk8);
                            if (!kDq) tmem_st8(lo_addr + 8 * q, pl);
                            tmem_st8(lo_addr + 32 + 8 * q, dl8);
                        };
                        tmem_ld16(xs_addr, sa);
                        tmem_ld16(xd_addr, da);
                        tmem_ld16(xs_addr + 16, sb);
                        tmem_ld16(xd_addr + 16, db);
                        tmem_wait_ld();
                        quarter(sa, da, 0);
                        tmem_ld16(xs_addr + 32, sa); tmem_ld16(xd_addr + 32, da);
                        quarter(sb, db, 1);
                        tmem_ld16(xs_addr + 48, sb); tmem_ld16(xd_addr + 48, db);
                        tmem_wait_ld();
                        quarter(sa, da, 2);
                        quarter(sb, db, 3);
                    };
                    if (masked) quarters(std::true_type{});
                    else quarters(std::false_type{});
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&sm.pd_done[b]);
            }
            if (!ok) break;
            t0 += (uint32_t)w.n_iter;
            if (!SPLIT && !(ok = fetch(n_item + 1, nx))) break;
            // --- epilogue: dK/dV: warpgroup 0 takes dK (x scale), warpgroup 1 dV; dQ: half the columns each
            const bool any = w.n_iter > 0;
            if (any) {
                if (!(ok = mbar_wait(&sm.acc_full, n_acc & 1, abort_flag, kLimit))) break;
                ++n_acc;
                tc_fence_after();
            }
            constexpr int kChunks = kDq ? D / 64 : D / 32;
            const uint32_t acc_addr = tmem + lane_base + (kDq ? b * (D / 2) : b * D);
            shared_tile = SPLIT && !kDq && w.is_main;
            void *dst = kDq ? (w.is_main ? p.dq_main : p.dq_branch) : b == 0 ? p.dk : p.dv;
            const float mul = kDq || b == 0 ? p.scale : 1.0f;
            const size_t base = kDq ? ((size_t)w.row * p.h_q + w.h) * D + b * (D / 2) : ((size_t)w.srow * p.h_kv + w.g) * D;
            // my part, unscaled, over the streamed stages (acc_full covers every MMA of this CTA, and with them
            // every copy into the stages)
            float4 *part = reinterpret_cast<float4 *>(sm.xs[0]) + (size_t)(b * kTile + r_in) * (D / 4);
#pragma unroll 1
            for (int c = 0; c < kChunks; ++c) {
                uint32_t r[32];
                if (any) {
                    tmem_ld32(acc_addr + c * 32, r);
                    tmem_wait_ld();
                    if (c == kChunks - 1) {
                        tc_fence_before();
                        mbar_arrive(&sm.acc_free);       // the next item may accumulate
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) r[e] = 0u;
                }
                bool not_finite = false;
                uint64_t nans = 0;
                if (!shared_tile) {
                    const float s = sum32(r);
                    not_finite = __any_sync(0xffffffffu, w.valid && s != s);
                    if (not_finite && w.valid) nans = nan_mask(r);
                }
                if (shared_tile) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)      // 16-byte chunks swizzled by the row: no bank conflicts
                        part[(8 * c + e) ^ (r_in & (D / 4 - 1))] =
                            make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]), __uint_as_float(r[4 * e + 2]),
                                        __uint_as_float(r[4 * e + 3]));
                } else if (w.valid) {
                    store_grad_chunk<false>(dst, base + c * 32, r, mul, p.wide);
                }
                if (not_finite) {      // does it hold rows out of its reach (ba_exact.cuh; bf16 results only)?
                    __nv_bfloat16 *row = (__nv_bfloat16 *)dst + base + c * 32;
                    if (kDq) repair_query_row<true, 8>(p.rows, w.is_main, w.row, w.h, w.g, w.nl, b * 32, 32, nans, mul, row);
                    else repair_key_row<8>(p.rows, w.is_main, w.row, w.g, b == 1, c * 32, 32, nans, mul, row);
                }
            }
            if (SPLIT) break;
        }
    }

    if (SPLIT && !kDq) {
        // ---- sum the parts: rank r finishes keys [128 r / S, 128 (r + 1) / S) of dK and dV, in rank order
        __syncwarp();
        cluster_sync_all();
        if (warp < 8 && shared_tile && !*abort_flag) {
            const KvItem &it = sm.item[0];
            const int rows_mine = kTile / S;
            float chk = 0.f;      // NaN: some result is
            for (int idx = tid; idx < 2 * rows_mine * (D / 4); idx += 256) {
                const int ch = idx % (D / 4), rr = idx / (D / 4);
                const int which = rr / rows_mine, r = rank * rows_mine + rr % rows_mine;    // dK / dV
                if (it.row0 + r >= it.row_end) continue;
                const uint32_t src = smem_u32(sm.xs[0]) + (uint32_t)(((which * kTile + r) * (D / 4) + (ch ^ (r & (D / 4 - 1)))) * 16);
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
                const size_t off = ((size_t)(it.srow0 + r) * p.h_kv + it.g) * D + ch * 4;
                *reinterpret_cast<uint2 *>((__nv_bfloat16 *)dst + off) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
                chk += x.x + x.y + x.z + x.w;
            }
            if (__any_sync(0xffffffffu, chk != chk)) {      // do they hold rows out of their reach (ba_exact.cuh; bf16 results only)?
#pragma unroll 1
                for (int idx = tid; idx < 2 * rows_mine * (D / 4); idx += 256) {
                    const int ch = idx % (D / 4), rr = idx / (D / 4), which = rr / rows_mine, r = rank * rows_mine + rr % rows_mine;
                    __nv_bfloat16 *row = (__nv_bfloat16 *)(which == 0 ? p.dk : p.dv) + ((size_t)(it.srow0 + r) * p.h_kv + it.g) * D + ch * 4;
                    uint64_t nans = 0;
                    if (it.row0 + r < it.row_end)
                        for (int e = 0; e < 4; ++e) nans |= is_nan(__bfloat162float(row[e])) ? 1ull << e : 0ull;
                    repair_key_row<4>(p.rows, true, it.row0 + r, it.g, which == 1, ch * 4, 4, nans, which == 0 ? p.scale : 1.0f, row);
                }
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

template <int MODE, bool SPLIT>
int launch_kv(const TcBwdParams &p, const BaOrder &order, const CUtensorMap *tm, int64_t grid, int dev, cudaStream_t st, bool after_delta = false) {
    if (grid <= 0) return BA_OK;
    // the dynamic shared-memory limit is a per-device attribute of the kernel
    static bool attr_set[64] = {};
    const size_t smem = sizeof(KvSmem);
    if (!attr_set[dev]) {
        // the register re-split hands out what a launch with kKvRegsLaunch registers per thread owns
        cudaFuncAttributes fa;
        BA_CUDA_CHECK(cudaFuncGetAttributes(&fa, tc_kv_kernel<MODE, SPLIT>));
        if (fa.numRegs * kKvThreads < 256 * kKvRegsCompute + 128 * kKvRegsIssue) return BA_EUNSUPPORTED;
        BA_CUDA_CHECK(cudaFuncSetAttribute(tc_kv_kernel<MODE, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    dependent_launch(cfg, attr, dim3((unsigned)grid), kKvThreads, smem, st);
    if (SPLIT) {
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)p.splits;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    } else if (!after_delta) {
        cfg.numAttrs = 0;
    }
    BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_kv_kernel<MODE, SPLIT>, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], p, order));
    return ba_check_launch();
}

// dQ at head_dim 64: 128-row tiles
inline void row_tiles(TcBwdParams &p, int64_t qm_n, int64_t br_n) {
    p.hp = p.group < kTile ? p.group : kTile;
    p.head_chunks = (p.group + p.hp - 1) / p.hp;
    p.tok = kTile / p.hp;
    p.main_tiles = (int)((qm_n + p.tok - 1) / p.tok);
    p.total_tiles = p.main_tiles + (int)((br_n + p.tok - 1) / p.tok);
}
inline BaTiling row_tiling(const TcBwdParams &p, bool has_main) {
    return {BA_ORDER_ROWS, has_main, p.main_tiles, p.tok, p.total_tiles - p.main_tiles, p.tok};
}
inline const BaOrder &row_order(const TcBwdParams &p, const ba_plan *pl, bool has_main) {
    return ba_find_order(pl, ba_whole_call(pl, p.r, has_main) ? row_tiling(p, has_main) : BaTiling{-1});
}

}  // namespace

void ba_tc_bwd_orders(ba_plan *pl, const ba_problem_t *host) {
    const int64_t n = pl->prob.n_main, m = pl->prob.n_branch;
    const BaRange r = ba_everything(pl);
    for (int has_main = 1; has_main >= 0; --has_main) {
        TcBwdParams p = bwd_params(pl, r, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr, nullptr, 0);
        if (key_items(p, pl, r, has_main) > 0 && p.splits == 1 && p.tile_major) ba_add_order(pl, host, key_tiling(p, has_main));
        if (pl->prob.head_dim == 64) {
            row_tiles(p, has_main ? n : 0, m);
            ba_add_order(pl, host, row_tiling(p, has_main));
        }
    }
}

const BaOrder &ba_tc_bwd_order(const ba_plan *pl, int stage, bool has_main, BaTiling *t) {
    BaRange r = ba_everything(pl);
    if (!has_main) r.qm_end = 0;
    TcBwdParams p = bwd_params(pl, r, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr, nullptr, 0);
    if (stage == BA_STAGE_DKDV) {
        key_items(p, pl, r, has_main);
        *t = key_tiling(p, has_main);
        return key_order(p, pl, has_main);
    }
    if (pl->prob.head_dim == 64) {
        row_tiles(p, r.qm_end, r.tok_end);
        *t = row_tiling(p, has_main);
        return row_order(p, pl, has_main);
    }
    ItemParams q;
    fill_items(q, pl, r, has_main, 0);
    *t = item_tiling(q, has_main);
    return item_order(q, pl, has_main);
}

int ba_tc_bwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch, const void *k,
              const void *v, const BaDelta &prep, int accumulate, void *dq_main, void *dq_branch, void *dk, void *dv,
              cudaStream_t st, int stages, int depth) {
    // depth > 0: dQ is written (bf16, one row per branch), dK / dV accumulate
    int dev = 0;
    BA_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return BA_EUNSUPPORTED;
    const ba_problem_t &pr = pl->prob;
    const void *d_o = prep.d_o;
    TcBwdParams p = bwd_params(pl, r, q_main, q_branch, k, v, prep.delta_t, d_o, accumulate, dq_main, dq_branch, dk, dv, depth);
    const bool has_main = q_main != nullptr, do_dq = stages & BA_STAGE_DQ, do_dkdv = stages & BA_STAGE_DKDV;
    const int64_t qm_n = has_main ? r.qm_end - r.qm_begin : 0, br_n = r.tok_end - r.tok_begin;
    auto maps = [&](CUtensorMap *tm, uint32_t qr, uint32_t qh, uint32_t kr) {
        return bwd_maps(tm, pl, r, q_main, q_branch, k, v, d_o, depth, qr, qh, kr);
    };
    // dQ may be launched while delta ends, but not with about one item to an SM behind a delta that fills the SMs: the CTAs
    // that start first take the items of those that cannot start yet, and work them off one after the other, while dK/dV
    // takes the SMs that come free (not at head_dim 64, where it comes after dQ: 2,738 rows, 5/1 heads, 88 / 91).  Whole steps of
    // draft rows, launched early / behind delta: 3,045 rows, 12/4 heads (148 items) 331 / 277 us, 3,430, 8/8 (112) 734 /
    // 630, 7,347, 5/1 (147) 267 / 239; with more items or a small delta early is 1 to 4 % better (372 items 129 / 131,
    // 1,372 rows 77 / 80), at worst 1.5 % slower (1,048 items 364 / 359).
    auto early_dq = [&](int64_t items) { return (stages & BA_STAGE_PREP) && !depth && (items > kSms || ba_delta_small(prep)); };
    auto prepare_rows = [&] { return stages & BA_STAGE_PREP ? ba_delta(prep, st) : BA_OK; };
    CUtensorMap tm[6];      // dQ
    if (pr.head_dim == 64) {
        CUtensorMap tk[6];  // dK/dV
        TcBwdParams pq = p;
        row_tiles(pq, qm_n, br_n);
        const int64_t dq_grid = (int64_t)pq.total_tiles * pr.h_kv * pq.head_chunks, grid = key_items(p, pl, r, has_main);
        if ((do_dq && dq_grid > INT_MAX) || (do_dkdv && grid > INT_MAX)) return BA_EUNSUPPORTED;
        if ((do_dq && !maps(tm, pq.tok, pq.hp, kSub)) || (do_dkdv && !maps(tk, kSub, 1, kTile))) return BA_EINVAL;
        int rc = prepare_rows();
        if (rc == BA_OK && do_dq)
            rc = launch_kv<kModeDq, false>(pq, row_order(pq, pl, has_main), tm, dq_grid, dev, st, (stages & BA_STAGE_PREP) != 0);
        if (rc != BA_OK || !do_dkdv) return rc;
        // (both kernels overlapped, as at head_dim 128: 605 us instead of 548 for the 4,096-token chains)
        const BaOrder &order = key_order(p, pl, has_main);
        return p.splits > 1 ? launch_kv<kModeDkdv, true>(p, order, tk, grid, dev, st) : launch_kv<kModeDkdv, false>(p, order, tk, grid, dev, st);
    }
    TcDqParams q;
    CUtensorMap k32, v32;
    int64_t dq_grid = 0;
    if (do_dq) {
        static bool attr_set[64] = {};
        if (!attr_set[dev]) {
            // the register re-split hands out what a launch with kDqRegsLaunch registers per thread owns
            cudaFuncAttributes fa;
            BA_CUDA_CHECK(cudaFuncGetAttributes(&fa, tc_dq_kernel));
            if (fa.numRegs * kDqThreads < 256 * kDqRegsCompute + 128 * kDqRegsIssue) return BA_EUNSUPPORTED;
            BA_CUDA_CHECK(cudaFuncSetAttribute(tc_dq_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DqSmem)));
            attr_set[dev] = true;
        }
        memset(&q, 0, sizeof q);
        dq_grid = fill_items(q, pl, r, has_main, depth);
        q.nlse2_t = p.nlse2_t; q.delta_t = p.delta_t; q.row_pitch = p.row_pitch;
        q.dq_main = dq_main; q.dq_branch = dq_branch;
        q.scale = p.scale; q.scale_log2 = p.scale_log2;
        q.accumulate = depth ? 0 : accumulate;
        q.wide = p.wide;
        q.status = p.status;
        if (dq_grid > INT_MAX) return BA_EUNSUPPORTED;
        const uint64_t kv_rows = key_rows(pl, r, depth);
        if (!maps(tm, q.tok, q.hp, kTile) || !make_tmap_rhd(&k32, k, kv_rows, pr.h_kv, 128, 32) ||
            !make_tmap_rhd(&v32, v, kv_rows, pr.h_kv, 128, 32))
            return BA_EINVAL;
    }
    TcDkdvCall dkdv;
    int rc = do_dkdv ? ba_tc_dkdv_prepare(dkdv, p, pl, r, q_main, q_branch, k, v, d_o, dev) : BA_OK;
    // nothing has been launched so far, and nothing is refused from here on
    if (rc == BA_OK) rc = prepare_rows();
    if (rc == BA_OK && depth && do_dkdv) rc = ba_tc_own_branch(p, q_branch, k, v, d_o, st);
    if (rc != BA_OK) return rc;
    if (dq_grid > 0) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        dependent_launch(cfg, attr, dim3((unsigned)dq_grid), kDqThreads, sizeof(DqSmem), st);
        if (!early_dq(dq_grid)) cfg.numAttrs = 0;
        BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_dq_kernel, tm[0], tm[1], tm[2], tm[3], tm[4], k32, v32, q, item_order(q, pl, has_main)));
        if ((rc = ba_check_launch()) != BA_OK) return rc;
    }
    // dK/dV: the two kernels write different tensors and need the same inputs: the second may start on the SMs that the
    // last items of the first leave idle (not when no row of dQ was launched: the kernel before is then the
    // caller's, or delta).  Both kernels, overlapped / one after the other: 2,048-token chains 222 / 231 us, draft
    // rows of 512 blocks 658 / 680.
    return do_dkdv ? ba_tc_dkdv_launch(dkdv, do_dq && qm_n + br_n > 0, st) : BA_OK;
}
