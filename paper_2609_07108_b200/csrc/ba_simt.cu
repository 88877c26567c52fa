// Plain-FMA (CUDA-core) branch attention: forward, dQ and dK/dV.
//
// This is the fp32 path (tensor cores cannot meet a 1e-4 absolute bound on N(0,1) inputs in a single
// tf32 pass) and the fallback for every supported shape.  Same metadata and same semantics as the
// tensor-core path: both key sets of a branch query (causal main prefix, own-branch keys; paper Section
// 3.2) go through ONE online-softmax pass, i.e. Eq. (lse-merge) applied tile by tile.
//
// One kernel, three modes.  A CTA of four warps owns 32 stationary rows and walks tiles of 32 streamed rows
// through shared memory:
//   forward, dQ   stationary = query rows (token, head of one KV head; head fastest, so the heads of a
//                 group share every K / V tile), streamed = keys
//   dK/dV         stationary = keys of one KV head, streamed = query rows, head by head
// Each tile is two or three small matrix products with register tiles of 8 x 4 (scores, contraction over D split
// four ways) and 4 x D/16 (accumulators, contraction over the tile), packed fp32 FMAs (fma.rn.f32x2) throughout.
// Scores pass between the two layouts of a warp through its own buffer: no barrier, only the two or
// three per tile that hand over the streamed tiles, whose copies (cp.async) run behind the other operand's
// products.  All operands stay in their natural [row][D] layout, padded by 16 bytes per row: 16-byte reads
// of 8 consecutive rows then touch all 32 banks once.
//
// Bound: latency, with three CTAs (twelve warps) per SM by registers: forward / dK/dV of the 2,048-token batch below
// issue in 49 / 42 % of the cycles, the FMA pipe is 48 / 48 % busy (60 / 61 % on the fullest SM), shared memory 40 /
// 50 %.  So more warps beat bigger tiles: 64 stationary rows (two
// CTAs per SM) read less shared memory per FMA and are slower, 8,192 tokens, 300 blocks of 8, 8/8 heads, D 128,
// forward / dQ / dK/dV: 1390 / 1837 / 2416 us against 1193 / 1725 / 2029.  Measured against kernels that walked the
// keys one by one with a row's dot product spread over D/32 lanes: 2,048 tokens with 64 blocks of 16, 8/2 heads,
// D 128: 162 / 211 / 271 us (were 399 / 424 / 1805); 640 tokens, 4/4 heads, D 64: 25 / 30 / 32 us (were 166 / 162 /
// 147).
//
// Few stationary tiles (small batches; few KV heads in dK/dV): the CTAs of a cluster share one tile, each
// takes a contiguous part of its streamed tiles, and the parts are summed through distributed shared
// memory in rank order, so every output element still has one owner and results are reproducible.
#include <limits.h>
#include <string.h>

#include "ba_common.cuh"
#include "ba_exact.cuh"
#include "ba_sm100.cuh"

using sm100::cluster_ld_f2;
using sm100::cluster_ld_f4;
using sm100::cluster_map;
using sm100::cluster_sync_all;
using sm100::ffma2;
using sm100::fmul2;
using sm100::launch_dependents;
using sm100::smem_u32;
using sm100::wait_prerequisites;

namespace {

constexpr int kThreads = 128;
constexpr int kRows = 32;      // stationary rows per CTA
constexpr int kBN = 32;        // streamed rows per tile
constexpr int kPPitch = kBN + 4;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

enum { kFwd = 0, kDq = 1, kDkdv = 2 };

struct SimtArgs : RowArgs {
    const float *lse_in;
    void *o;          // forward output
    float *lse_out;
    void *dq_main, *dq_branch, *dk, *dv;
    int partial_out;  // forward: compact fp32 outputs (2: merged in place)
    int accumulate;   // backward: fp32 += outputs
    int hp, head_chunks, tok;      // forward, dQ: heads per tile, chunks of hp heads per group, tokens per tile
    int main_tiles, total_tiles;   // stationary tiles (of one KV head and head chunk)
    int splits;                    // CTAs per tile (cluster size)
};

template <typename T> __device__ __forceinline__ void store4(T *p, float4 x);
template <> __device__ __forceinline__ void store4<float>(float *p, float4 x) {
    *reinterpret_cast<float4 *>(p) = x;
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *p, float4 x) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
    uint2 r;
    r.x = *reinterpret_cast<uint32_t *>(&lo);
    r.y = *reinterpret_cast<uint32_t *>(&hi);
    *reinterpret_cast<uint2 *>(p) = r;
}

// NaN or opposite infinities among four results
__device__ __forceinline__ bool not_finite(float4 x) {
    const float s = x.x + x.y + x.z + x.w;
    return s != s;
}
__device__ __forceinline__ uint64_t nan_bits(float4 x) {
    return (x.x != x.x ? 1u : 0u) | (x.y != x.y ? 2u : 0u) | (x.z != x.z ? 4u : 0u) | (x.w != x.w ? 8u : 0u);
}

// four elements global -> shared as fp32 (zeros when !live): asynchronous for fp32 sources
__device__ __forceinline__ void copy4(float *dst, const float *src, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy4(float *dst, const __nv_bfloat16 *src, bool live) {
    const float4 x = live ? load4<__nv_bfloat16>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(dst) = x;
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int D> __device__ __forceinline__ constexpr int pitch() { return D + 4; }

// ROWS rows -> shared tile [ROWS][D + 4]; row(r) = element offset of row r in `src`, or -1 (zeros)
template <typename T, int D, int ROWS, typename RowFn>
__device__ __forceinline__ void load_rows(float *dst, const T *src, RowFn row) {
    constexpr int CPR = D / 4;  // float4 chunks per row
#pragma unroll 4
    for (int idx = threadIdx.x; idx < ROWS * CPR; idx += kThreads) {
        const int r = idx / CPR, ch = idx % CPR;
        const int64_t off = row(r);
        copy4(dst + r * pitch<D>() + ch * 4, src + (off < 0 ? 0 : off + ch * 4), off >= 0);
    }
}

// s[i][j] = <a row (2 rg + i), b row (cg + 8 j)>, rg = lane / 8, cg = lane % 8, of the warp's 8 x 32 tile.  A lane
// first forms 8 x 4 products over a quarter of the contraction (chunks of four, dealt to the four row groups), then
// the lanes exchange halves until each holds its two rows.  Shared memory fills 32 lane registers per cycle whatever
// the pattern, so what counts is loads per FMA: 12 float4 for 64 packed FMAs here, 6 for 16 with tiles of 2 x 4 over
// the whole contraction (640 tokens, D 64, whole step: 75.1 -> 68.1 us; 300 tokens, D 128, dQ: 48 -> 41 us).
template <int D> __device__ __forceinline__ void scores(const float *a, const float *b, int lane, float (&s)[2][4]) {
    a += 4 * (lane >> 3);
    b += 4 * (lane >> 3);
    float2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int k = 0; k < D; k += 16) {
        float4 y[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = *reinterpret_cast<const float4 *>(b + 8 * j * pitch<D>() + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 x = *reinterpret_cast<const float4 *>(a + i * pitch<D>() + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[i][j] = ffma2(make_float2(x.x, x.y), make_float2(y[j].x, y[j].y), acc[i][j]);
                acc[i][j] = ffma2(make_float2(x.z, x.w), make_float2(y[j].z, y[j].w), acc[i][j]);
            }
        }
    }
    float t[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) t[i][j] = acc[i][j].x + acc[i][j].y;
#pragma unroll
    for (int half = 4; half >= 2; half >>= 1) {      // keep half of the rows, add the partner's part of them
        const int off = 4 * half;                    // partner: lane ^ 16, then lane ^ 8
        const bool upper = lane & off;
#pragma unroll
        for (int i = 0; i < half; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float other = __shfl_xor_sync(0xffffffffu, upper ? t[i][j] : t[half + i][j], off);
                t[i][j] = (upper ? t[half + i][j] : t[i][j]) + other;
            }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = t[i][j];
}

// acc[r][...] += sum_n p[4 ag + r][n] * v[n][cols], ag = lane / 16; columns 4 (lane % 16) + 64 q + 0 .. 3
template <int D> struct Acc { float2 v[4][D / 32]; };
template <int D> __device__ __forceinline__ void accumulate(const float *p, const float *v, Acc<D> &acc) {
#pragma unroll 2
    for (int n = 0; n < kBN; n += 4) {
        float4 w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = *reinterpret_cast<const float4 *>(p + r * kPPitch + n);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int q = 0; q < D / 64; ++q) {
                const float4 x = *reinterpret_cast<const float4 *>(v + (n + e) * pitch<D>() + 64 * q);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float pe = e == 0 ? w[r].x : e == 1 ? w[r].y : e == 2 ? w[r].z : w[r].w;
                    const float2 p2 = make_float2(pe, pe);
                    acc.v[r][2 * q] = ffma2(p2, make_float2(x.x, x.y), acc.v[r][2 * q]);
                    acc.v[r][2 * q + 1] = ffma2(p2, make_float2(x.z, x.w), acc.v[r][2 * q + 1]);
                }
            }
    }
}

template <int D, int MODE> struct SimtSmem {
    static constexpr int kX1 = MODE == kDq ? 2 : 1;             // dQ keeps K of the next tile in a second buffer
    float st1[kRows * pitch<D>()];                              // stationary: Q / K
    float st2[MODE == kFwd ? 4 : kRows * pitch<D>()];           // stationary: - / dO / V
    float x1[kX1][kBN * pitch<D>()];                           // streamed: K / Q
    float x2[kBN * pitch<D>()];                                 // streamed: V / dO
    float p[4][kRows / 4 * kPPitch];                             // per warp
    float alpha[4][kRows / 4];
    float2 ml[kRows];
    // dK/dV: scalars of the streamed query rows
    float lse2[kBN], dlt[kBN];
    int lo[kBN], hi[kBN], bst[kBN];
    unsigned long long mask[kBN];
    int lo_min, hi_max, bs_min, be_max;
};

template <typename T, int D, int MODE>
__global__ void __launch_bounds__(kThreads, 3) simt_kernel(const __grid_constant__ SimtArgs a, const __grid_constant__ BaOrder order) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    using Smem = SimtSmem<D, MODE>;
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    constexpr int WR = kRows / 4, AR = 4;     // rows per warp, per accumulator lane
    constexpr bool kMerges = MODE == kFwd && D == 64 && sizeof(T) == 2;      // partial results merged in place
    constexpr int P = pitch<D>();
    if (MODE == kDq) wait_prerequisites();      // launched while delta ends
    if (MODE != kDkdv) launch_dependents();     // dQ: dK/dV may start beside it; forward: delta may be launched
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t n = a.meta.n_main;
    const int rank = (int)(blockIdx.x % a.splits);
    const int work = (int)(blockIdx.x / a.splits);

    // ---- stationary tile: kRows rows of the main or the branch part.  Heaviest first: later query rows
    // (longer prefixes), earlier keys (more viewers).
    const int per = MODE == kDkdv ? a.h_kv : a.h_kv * a.head_chunks;
    const int inner = work % per;
    const int tile = order.n > 0 ? order.tile[work / per] : MODE == kDkdv ? work / per : a.total_tiles - 1 - work / per;
    const bool is_main = tile < a.main_tiles;
    const int g = MODE == kDkdv ? inner : inner / a.head_chunks;
    const int h0 = MODE == kDkdv ? 0 : g * a.group + (inner % a.head_chunks) * a.hp;
    const int64_t first = MODE == kDkdv ? (is_main ? a.r.kv_begin : a.r.tok_begin) : (is_main ? a.r.qm_begin : a.r.tok_begin);
    const int64_t end = MODE == kDkdv ? (is_main ? a.r.kv_end : a.r.tok_end) : (is_main ? a.r.qm_end : a.r.tok_end);
    const int step = MODE == kDkdv ? kRows : a.tok;
    const int64_t base = first + (int64_t)(is_main ? tile : tile - a.main_tiles) * step;
    // row r of the tile: token (key) base + r / hp, query head h0 + r % hp
    auto live_row = [&](int r) -> bool {
        if (MODE == kDkdv) return base + r < end;
        const int t = r / a.hp;
        return t < a.tok && base + t < end && h0 + r % a.hp < (g + 1) * a.group;
    };
    auto row_tok = [&](int r) -> int64_t { return MODE == kDkdv ? base + r : base + r / a.hp; };

    if (tid == 0) { sm.lo_min = INT_MAX; sm.hi_max = -1; sm.bs_min = INT_MAX; sm.be_max = -1; }
    __syncthreads();
    if (tid < kRows && live_row(tid)) {
        const int64_t t = row_tok(tid);
        if (MODE == kDkdv) {
            if (is_main) {
                atomicMax(&sm.hi_max, a.meta.key_qend[t]);
                atomicMin(&sm.bs_min, a.meta.key_bq_begin[t]);
                atomicMax(&sm.be_max, a.meta.key_bq_end[t]);
            } else {
                atomicMin(&sm.bs_min, a.meta.br_start[t]);
                atomicMax(&sm.be_max, a.meta.br_end[t]);
            }
        } else {
            const int64_t gr = is_main ? t : n + t;
            const int lo = max(a.meta.row_lo[gr], (int)a.r.kv_begin), hi = min(a.meta.row_hi[gr], (int)a.r.kv_end - 1);
            if ((a.r.parts & BA_PART_MAIN) && hi >= lo) { atomicMin(&sm.lo_min, lo); atomicMax(&sm.hi_max, hi); }
            if (!is_main && (a.r.parts & BA_PART_BRANCH)) {
                atomicMin(&sm.bs_min, a.meta.br_start[t]);
                atomicMax(&sm.be_max, a.meta.br_end[t]);
            }
        }
    }
    // stationary operands
    {
        const T *src1 = MODE == kDkdv ? (const T *)a.k : is_main ? (const T *)a.q_main : (const T *)a.q_branch;
        load_rows<T, D, kRows>(sm.st1, src1, [&](int r) -> int64_t {
            if (!live_row(r)) return -1;
            if (MODE == kDkdv) return (((is_main ? -a.r.kv_base : n) + base + r) * a.h_kv + g) * D;
            return (row_tok(r) * a.h_q + h0 + r % a.hp) * D;
        });
        if (MODE != kFwd) {
            const T *src2 = MODE == kDkdv ? (const T *)a.v : (const T *)a.d_o;
            load_rows<T, D, kRows>(sm.st2, src2, [&](int r) -> int64_t {
                if (!live_row(r)) return -1;
                if (MODE == kDkdv) return (((is_main ? -a.r.kv_base : n) + base + r) * a.h_kv + g) * D;
                return (((is_main ? 0 : n) + row_tok(r)) * a.h_q + h0 + r % a.hp) * D;
            });
        }
    }
    __syncthreads();

    // ---- streamed tiles: main part [m0, m1), branch part [b0, b1) (main keys / own-branch keys, or main
    // query rows / branch tokens); dK/dV walks them once per query head of the group
    int64_t m0 = 0, m1 = 0, b0 = 0, b1 = 0;
    if (MODE == kDkdv) {
        if (is_main && a.q_main != nullptr) {
            m0 = max(base, a.r.qm_begin);
            m1 = min((int64_t)sm.hi_max, a.r.qm_end);
        }
        b0 = max((int64_t)sm.bs_min, a.r.tok_begin);
        b1 = min((int64_t)sm.be_max, a.r.tok_end);
    } else {
        m0 = sm.lo_min; m1 = (int64_t)sm.hi_max + 1;
        b0 = sm.bs_min; b1 = sm.be_max;
    }
    const int nm = m1 > m0 ? (int)((m1 - m0 + kBN - 1) / kBN) : 0;
    const int nb = b1 > b0 ? (int)((b1 - b0 + kBN - 1) / kBN) : 0;
    const int n_tiles = nm + nb;
    const int n_iter = n_tiles * (MODE == kDkdv ? a.group : 1);
    const int t_beg = (int)((int64_t)n_iter * rank / a.splits), t_end = (int)((int64_t)n_iter * (rank + 1) / a.splits);

    struct Tile { int r0, cnt, h; bool main; };
    auto tile_of = [&](int t) -> Tile {
        Tile x;
        const int s = MODE == kDkdv ? t % n_tiles : t;
        x.h = MODE == kDkdv ? g * a.group + t / n_tiles : g;
        x.main = s < nm;
        x.r0 = (int)(x.main ? m0 : b0) + (x.main ? s : s - nm) * kBN;
        x.cnt = min(kBN, (int)(x.main ? m1 : b1) - x.r0);
        return x;
    };
    auto load_x1 = [&](int t) {
        if (t >= t_end) return;
        const Tile x = tile_of(t);
        float *dst = sm.x1[t % Smem::kX1];
        if (MODE == kDkdv) {
            load_rows<T, D, kBN>(dst, x.main ? (const T *)a.q_main : (const T *)a.q_branch,
                            [&](int r) -> int64_t { return r < x.cnt ? ((int64_t)(x.r0 + r) * a.h_q + x.h) * D : -1; });
            if (tid < kBN) {
                const bool live = tid < x.cnt;
                const int64_t row = x.r0 + tid, gr = (x.main ? 0 : n) + row;
                sm.lse2[tid] = live ? a.lse_in[gr * a.h_q + x.h] * kLog2e : 0.f;
                sm.dlt[tid] = live ? a.delta_t[(size_t)x.h * a.row_pitch + gr] : 0.f;
                sm.lo[tid] = live ? a.meta.row_lo[gr] : INT_MAX;
                sm.hi[tid] = live ? a.meta.row_hi[gr] : -1;
                sm.bst[tid] = live && !x.main ? a.meta.br_start[row] : 0;
                sm.mask[tid] = live && !x.main ? a.meta.br_mask[row] : 0ull;
            }
        } else {
            const int row0 = (int)(x.main ? -a.r.kv_base : n) + x.r0;      // in the key tensors
            load_rows<T, D, kBN>(dst, (const T *)a.k,
                            [&](int r) -> int64_t { return r < x.cnt ? ((int64_t)(row0 + r) * a.h_kv + g) * D : -1; });
        }
    };
    auto load_x2 = [&](int t) {
        if (t >= t_end) return;
        const Tile x = tile_of(t);
        const int heads = MODE == kDkdv ? a.h_q : a.h_kv, row0 = (int)(!x.main ? n : MODE == kDkdv ? 0 : -a.r.kv_base) + x.r0;
        load_rows<T, D, kBN>(sm.x2, MODE == kDkdv ? (const T *)a.d_o : (const T *)a.v,
                        [&](int r) -> int64_t { return r < x.cnt ? ((int64_t)(row0 + r) * heads + x.h) * D : -1; });
    };

    // ---- per-thread views: score lanes hold rows 2 rg + i and columns cg + 8 j of the warp's WR x 32 tile,
    // accumulator lanes rows AR ag + r and 4-column chunks
    const int rg = lane >> 3, cg = lane & 7, ag = lane >> 4, ac = (lane & 15) * 4;
    const float *a1 = sm.st1 + warp * WR * P, *a2 = sm.st2 + (MODE == kFwd ? 0 : warp * WR * P);
    float *pw = sm.p[warp];
    float *p_st = pw + 2 * rg * kPPitch + cg;                    // my score elements: + i * kPPitch + 8 j
    const float *p_ld = pw + AR * ag * kPPitch;
    // my stationary rows
    int lo[2], hi[2], bst[2], key[2];
    uint64_t mask[2];
    bool valid[2];
    float lse2[2], dlt[2], m_run[2], l_run[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int r = warp * WR + 2 * rg + i;
        lse2[i] = dlt[i] = l_run[i] = 0.f;
        m_run[i] = -INFINITY;
        valid[i] = live_row(r);
        lo[i] = INT_MAX; hi[i] = -1; bst[i] = 0; mask[i] = 0; key[i] = (int)row_tok(r);
        if (MODE != kDkdv && valid[i]) {
            const int64_t t = row_tok(r), gr = is_main ? t : n + t;
            const int h = h0 + r % a.hp;
            if (a.r.parts & BA_PART_MAIN) {
                lo[i] = max(a.meta.row_lo[gr], (int)a.r.kv_begin);
                hi[i] = min(a.meta.row_hi[gr], (int)a.r.kv_end - 1);
            }
            if (!is_main && (a.r.parts & BA_PART_BRANCH)) { bst[i] = a.meta.br_start[t]; mask[i] = a.meta.br_mask[t]; }
            if (MODE == kDq) {
                lse2[i] = a.lse_in[gr * a.h_q + h] * kLog2e;
                dlt[i] = a.delta_t[(size_t)h * a.row_pitch + gr];
            }
        }
    }
    Acc<D> acc0, acc1;     // O / dQ / dK, and dV
#pragma unroll
    for (int r = 0; r < AR; ++r)
#pragma unroll
        for (int c = 0; c < D / 32; ++c) { acc0.v[r][c] = make_float2(0.f, 0.f); acc1.v[r][c] = make_float2(0.f, 0.f); }

    auto visible = [&](const Tile &x, int i, int c) -> bool {
        if (!valid[i]) return false;
        if (MODE != kDkdv) {
            if (x.main) { const int kk = x.r0 + c; return kk >= lo[i] && kk <= hi[i]; }
            const int rel = x.r0 + c - bst[i];
            return c < x.cnt && rel >= 0 && rel < 64 && ((mask[i] >> rel) & 1ull);
        }
        if (is_main) return key[i] >= sm.lo[c] && key[i] <= sm.hi[c];
        const int rel = key[i] - sm.bst[c];
        return rel >= 0 && rel < 64 && ((sm.mask[c] >> rel) & 1ull);
    };

    load_x1(t_beg);
    if (MODE == kDq) load_x2(t_beg);
    copies_done();
    __syncthreads();
    if (MODE != kDq) load_x2(t_beg);
    for (int t = t_beg; t < t_end; ++t) {
        const Tile x = tile_of(t);
        const float *x1 = sm.x1[t % Smem::kX1];
        float s[2][4];
        if (MODE == kDq) load_x1(t + 1);           // into the other buffer
        scores<D>(a1, x1 + cg * P, lane, s);
        if (MODE == kFwd) {
            // --- online softmax of the warp's eight rows
            float alpha[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float mt = -INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    s[i][j] = visible(x, i, cg + 8 * j) ? s[i][j] * a.scale_log2 : -INFINITY;
                    mt = fmaxf(mt, s[i][j]);
                }
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 4));
                const float mn = fmaxf(m_run[i], mt);
                alpha[i] = mn == -INFINITY ? 1.f : exp2f(m_run[i] - mn);
                float sum = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    s[i][j] = s[i][j] == -INFINITY ? 0.f : exp2f(s[i][j] - mn);
                    sum += s[i][j];
                    p_st[i * kPPitch + 8 * j] = s[i][j];
                }
                l_run[i] = l_run[i] * alpha[i] + sum;      // my columns only; summed over the lanes at the end
                m_run[i] = mn;
                if (cg == 0) sm.alpha[warp][2 * rg + i] = alpha[i];
            }
            copies_done();
            __syncthreads();                       // V has arrived, K is free
            load_x1(t + 1);
#pragma unroll
            for (int r = 0; r < AR; ++r) {
                const float f = sm.alpha[warp][AR * ag + r];
#pragma unroll
                for (int c = 0; c < D / 32; ++c) acc0.v[r][c] = fmul2(acc0.v[r][c], make_float2(f, f));
            }
            accumulate<D>(p_ld, sm.x2 + ac, acc0);
            copies_done();
            __syncthreads();                       // next K has arrived, V is free
            load_x2(t + 1);
        } else if (MODE == kDq) {
            float dp[2][4];
            scores<D>(a2, sm.x2 + cg * P, lane, dp);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float pr = exp2f(s[i][j] * a.scale_log2 - lse2[i]);
                    p_st[i * kPPitch + 8 * j] = visible(x, i, cg + 8 * j) ? pr * (dp[i][j] - dlt[i]) : 0.f;
                }
            __syncthreads();                       // V is free
            load_x2(t + 1);
            accumulate<D>(p_ld, x1 + ac, acc0);    // dQ += dS K
            copies_done();
            __syncthreads();                       // next K, V have arrived
        } else {
            copies_done();
            __syncthreads();                       // dO has arrived
            float dp[2][4];
            scores<D>(a2, sm.x2 + cg * P, lane, dp);
            float pr[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = cg + 8 * j;
                    const bool vis = visible(x, i, c);
                    pr[i][j] = vis ? exp2f(s[i][j] * a.scale_log2 - sm.lse2[c]) : 0.f;
                    p_st[i * kPPitch + 8 * j] = vis ? pr[i][j] * (dp[i][j] - sm.dlt[c]) : 0.f;
                }
            __syncwarp();
            accumulate<D>(p_ld, x1 + ac, acc0);    // dK += dS^T Q
            __syncthreads();                       // Q is free
            load_x1(t + 1);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) p_st[i * kPPitch + 8 * j] = pr[i][j];
            __syncwarp();
            accumulate<D>(p_ld, sm.x2 + ac, acc1); // dV += P^T dO
            copies_done();
            __syncthreads();                       // next Q has arrived, dO is free
            load_x2(t + 1);
        }
    }

    // ---- epilogue: the parts' accumulators in shared memory, summed by row over the cluster
    copies_done();
    __syncthreads();
    float *out0 = sm.st1, *out1 = sm.st2;
#pragma unroll
    for (int r = 0; r < AR; ++r)
#pragma unroll
        for (int q = 0; q < D / 64; ++q) {
            const int off = (warp * WR + AR * ag + r) * P + ac + 64 * q;
            *reinterpret_cast<float4 *>(out0 + off) =
                make_float4(acc0.v[r][2 * q].x, acc0.v[r][2 * q].y, acc0.v[r][2 * q + 1].x, acc0.v[r][2 * q + 1].y);
            if (MODE == kDkdv)
                *reinterpret_cast<float4 *>(out1 + off) =
                    make_float4(acc1.v[r][2 * q].x, acc1.v[r][2 * q].y, acc1.v[r][2 * q + 1].x, acc1.v[r][2 * q + 1].y);
        }
    if (MODE == kFwd) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float l = l_run[i];
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            l += __shfl_xor_sync(0xffffffffu, l, 4);
            if (cg == 0) sm.ml[warp * WR + 2 * rg + i] = make_float2(m_run[i], l);
        }
    }
    __syncwarp();
    if (a.splits > 1) cluster_sync_all(); else __syncthreads();
    constexpr int CPR = D / 4;
    const int rows_mine = kRows / a.splits;
    for (int idx = tid; idx < rows_mine * CPR; idx += kThreads) {
        const int r = rank * rows_mine + idx / CPR, ch = (idx % CPR) * 4;
        const int64_t t = row_tok(r), gr = is_main ? t : n + t;
        auto out_row = [&]() -> int64_t {
            return a.partial_out ? is_main ? t - a.r.qm_begin : (a.r.qm_end - a.r.qm_begin) + (t - a.r.tok_begin) : gr;
        };
        const bool live = live_row(r);
        float lse_a = -INFINITY;
        if (kMerges && a.partial_out == 2) {      // the lanes of a row (of one warp) read the old LSE before one replaces it
            if (live) lse_a = a.lse_out[out_row() * a.h_q + h0 + r % a.hp];
            __syncwarp();
        }
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        const uint32_t src0 = smem_u32(out0 + r * P + ch), src1 = smem_u32(out1 + r * P + ch), src_ml = smem_u32(&sm.ml[r]);
        if (MODE == kFwd) {
            float mx = -INFINITY, l = 0.f;
            for (int s = 0; s < a.splits; ++s) mx = fmaxf(mx, cluster_ld_f2(cluster_map(src_ml, s)).x);
            for (int s = 0; s < a.splits; ++s) {
                const float2 ml = cluster_ld_f2(cluster_map(src_ml, s));
                if (ml.y == 0.f) continue;      // sees nothing (a sum that is NaN is not an empty part)
                const float w = exp2f(ml.x - mx);
                const float4 v = cluster_ld_f4(cluster_map(src0, s));
                l += w * ml.y;
                x.x += w * v.x; x.y += w * v.y; x.z += w * v.z; x.w += w * v.w;
            }
            const float inv = l > 0.f ? 1.0f / l : 0.f;
            const int h = h0 + r % a.hp;
            if (__any_sync(0xffffffffu, live && not_finite(x)))      // does it hold what it does not see (ba_exact.cuh)?
                x = repair_query4<T, D, false>(a, is_main, (int)t, h, g, -mx, ch, live ? nan_bits(x) : 0, x);
            if (!live) continue;
            float lse_new = l > 0.f ? (mx + log2f(l)) * kLn2 : -INFINITY, w_new = inv, w_old = 0.f;
            if (kMerges && a.partial_out == 2) merge_weights(lse_a, lse_new, inv, lse_new, w_old, w_new);
            x.x *= w_new; x.y *= w_new; x.z *= w_new; x.w *= w_new;
            const int64_t orow = out_row();
            if (ch == 0) a.lse_out[orow * a.h_q + h] = lse_new;
            const size_t off = ((size_t)orow * a.h_q + h) * D + ch;
            if (kMerges && w_old != 0.f) {
                const float4 o = load4<float>((float *)a.o + off);
                x.x += o.x * w_old; x.y += o.y * w_old; x.z += o.z * w_old; x.w += o.w * w_old;
            }
            if (a.partial_out) store4<float>((float *)a.o + off, x);
            else store4<T>((T *)a.o + off, x);
        } else {
            for (int s = 0; s < a.splits; ++s) {
                const float4 v = cluster_ld_f4(cluster_map(src0, s));
                x.x += v.x; x.y += v.y; x.z += v.z; x.w += v.w;
                if (MODE == kDkdv) {
                    const float4 u = cluster_ld_f4(cluster_map(src1, s));
                    y.x += u.x; y.y += u.y; y.z += u.z; y.w += u.w;
                }
            }
            // do they hold rows out of their reach (ba_exact.cuh)?
            if (MODE == kDq && __any_sync(0xffffffffu, live && not_finite(x))) {
                const int h = h0 + r % a.hp;
                const float nl = live ? a.nlse2_t[h * a.row_pitch + gr] : 0.f;
                x = repair_query4<T, D, true>(a, is_main, (int)t, h, g, nl, ch, live ? nan_bits(x) : 0, x);
            }
            if (MODE == kDkdv) {
                if (__any_sync(0xffffffffu, live && not_finite(x)))
                    x = repair_key4<T, D>(a, is_main, (int)t, g, false, ch, live ? nan_bits(x) : 0, x);
                if (__any_sync(0xffffffffu, live && not_finite(y)))
                    y = repair_key4<T, D>(a, is_main, (int)t, g, true, ch, live ? nan_bits(y) : 0, y);
            }
            if (!live) continue;
            x.x *= a.scale; x.y *= a.scale; x.z *= a.scale; x.w *= a.scale;
            void *dst0 = MODE == kDkdv ? a.dk : is_main ? a.dq_main : a.dq_branch;
            const size_t off = MODE == kDkdv ? ((size_t)(is_main ? t - a.r.kv_base : gr) * a.h_kv + g) * D + ch : ((size_t)t * a.h_q + h0 + r % a.hp) * D + ch;
            if (a.accumulate) {
                const float4 o = load4<float>((float *)dst0 + off);
                store4<float>((float *)dst0 + off, make_float4(o.x + x.x, o.y + x.y, o.z + x.z, o.w + x.w));
                if (MODE == kDkdv) {
                    const float4 u = load4<float>((float *)a.dv + off);
                    store4<float>((float *)a.dv + off, make_float4(u.x + y.x, u.y + y.y, u.z + y.z, u.w + y.w));
                }
            } else {
                store4<T>((T *)dst0 + off, x);
                if (MODE == kDkdv) store4<T>((T *)a.dv + off, y);
            }
        }
    }
    __syncwarp();
    if (a.splits > 1) cluster_sync_all();      // no CTA leaves while another may still read its shared memory
    if (MODE == kDkdv) wait_prerequisites();   // never done before the dQ kernel that it may overlap
}

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

template <typename T, int D, int MODE>
int launch(SimtArgs &a, const BaOrder &order, int64_t work, bool after_dq, cudaStream_t st) {
    // the dynamic shared-memory limit is a per-device attribute of the kernel
    static bool attr_set[64] = {};
    int dev = 0;
    BA_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return BA_EUNSUPPORTED;
    const size_t smem = sizeof(SimtSmem<D, MODE>);
    if (!attr_set[dev]) {
        BA_CUDA_CHECK(cudaFuncSetAttribute(simt_kernel<T, D, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)(work * a.splits));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    if (a.splits > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)a.splits;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    if (after_dq) {     // start when every CTA of the kernel queued just before has started (dQ: it then waits for delta)
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++cfg.numAttrs;
    }
    cfg.attrs = attr;
    BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, simt_kernel<T, D, MODE>, a, order));
    return ba_check_launch();
}

// tile geometry; returns the number of tiles
template <int MODE> int64_t tile_work(SimtArgs &a) {
    int64_t mt, bt, per;
    if (MODE == kDkdv) {
        mt = (a.r.parts & BA_PART_MAIN) ? ceil_div(a.r.kv_end - a.r.kv_begin, kRows) : 0;
        bt = (a.r.parts & BA_PART_BRANCH) ? ceil_div(a.r.tok_end - a.r.tok_begin, kRows) : 0;
        per = a.h_kv;
    } else {
        a.hp = a.group < kRows ? a.group : kRows;
        a.head_chunks = (a.group + a.hp - 1) / a.hp;
        a.tok = kRows / a.hp;
        mt = a.q_main ? ceil_div(a.r.qm_end - a.r.qm_begin, a.tok) : 0;
        bt = ceil_div(a.r.tok_end - a.r.tok_begin, a.tok);
        per = (int64_t)a.h_kv * a.head_chunks;
    }
    a.main_tiles = (int)mt;
    a.total_tiles = (int)(mt + bt);
    return (mt + bt) * per;
}

template <int MODE> BaTiling tiling(const SimtArgs &a, bool has_main) {
    const int step = MODE == kDkdv ? kRows : a.tok;
    return {MODE == kDkdv ? BA_ORDER_KEYS : BA_ORDER_ROWS, has_main, a.main_tiles, step, a.total_tiles - a.main_tiles, step};
}

template <int MODE> const BaOrder &tile_order(const ba_plan *pl, const SimtArgs &a) {
    const bool has_main = a.q_main != nullptr;
    return ba_find_order(pl, ba_whole_call(pl, a.r, has_main) ? tiling<MODE>(a, has_main) : BaTiling{-1});
}

template <typename T, int D, int MODE>
int launch_tiles(const ba_plan *pl, SimtArgs a, bool after_dq, cudaStream_t st) {
    const ba_problem_t &pr = pl->prob;
    const int64_t seq = pr.num_seqs > 0 ? pr.n_main / pr.num_seqs : 0;
    const int64_t rows_per_key = pr.n_main > 0 ? 1 + pr.n_branch / pr.n_main : 1;
    // streamed tiles of a long row: a whole sequence (dK/dV: of every head)
    const int64_t est = MODE == kDkdv ? seq * rows_per_key * a.group / kBN : seq / kBN;
    const int64_t work = tile_work<MODE>(a);
    if (work == 0) return BA_OK;
    // Split a tile's walk over a cluster until there are about eight CTAs per SM as long as the walk of a whole
    // sequence leaves every part two streamed tiles (300 tokens, dQ: 48 us; 67 us with parts of one tile), and on to
    // sixteen, for the balance between the SMs, while it leaves every part four (2,048 tokens with 64 blocks, dK/dV:
    // 303 us with eight, 270 with sixteen; 3,500 tokens, 200 chains of 20, 8/4 heads, D 64: 1625 and 980; 1,000
    // tokens with 60 trees, dQ: 138 us in parts of four, 162 in parts of two).
    a.splits = 1;
    while (a.splits < 8 && ((work * a.splits * 2 <= kSms * 8 && est >= 2 * 2 * a.splits) ||
                            (work * a.splits * 2 <= kSms * 16 && est >= 2 * 4 * a.splits)))
        a.splits *= 2;
    if (work * a.splits > INT_MAX) return BA_EUNSUPPORTED;
    return launch<T, D, MODE>(a, tile_order<MODE>(pl, a), work, after_dq, st);
}

template <int MODE> int dispatch(const ba_plan *pl, const SimtArgs &a, cudaStream_t st, bool after_dq = false) {
    const int d = pl->prob.head_dim;
    if (pl->prob.dtype == BA_FP32)
        return d == 64 ? launch_tiles<float, 64, MODE>(pl, a, after_dq, st) : launch_tiles<float, 128, MODE>(pl, a, after_dq, st);
    return d == 64 ? launch_tiles<__nv_bfloat16, 64, MODE>(pl, a, after_dq, st) : launch_tiles<__nv_bfloat16, 128, MODE>(pl, a, after_dq, st);
}

SimtArgs base_args(const ba_plan *pl, const BaRange &r) {
    SimtArgs a;
    memset(&a, 0, sizeof a);
    a.meta = pl->meta;
    a.r = r;
    a.h_q = pl->prob.h_q;
    a.h_kv = pl->prob.h_kv;
    a.group = pl->prob.h_q / pl->prob.h_kv;
    a.scale = pl->scale;
    a.scale_log2 = pl->scale * kLog2e;
    return a;
}

}  // namespace

void ba_simt_orders(ba_plan *pl, const ba_problem_t *host) {
    for (int has_main = 1; has_main >= 0; --has_main) {
        SimtArgs a = base_args(pl, ba_everything(pl));
        a.q_main = has_main ? pl : nullptr;      // (only asked whether it is there)
        tile_work<kFwd>(a);                      // forward and dQ
        ba_add_order(pl, host, tiling<kFwd>(a, has_main));
        tile_work<kDkdv>(a);
        ba_add_order(pl, host, tiling<kDkdv>(a, has_main));
    }
}

const BaOrder &ba_simt_order(const ba_plan *pl, int stage, bool has_main, BaTiling *t) {
    SimtArgs a = base_args(pl, ba_everything(pl));
    a.q_main = has_main ? pl : nullptr;
    if (stage == BA_STAGE_DKDV) {
        tile_work<kDkdv>(a);
        *t = tiling<kDkdv>(a, has_main);
        return tile_order<kDkdv>(pl, a);
    }
    tile_work<kFwd>(a);
    *t = tiling<kFwd>(a, has_main);
    return tile_order<kFwd>(pl, a);
}

int ba_simt_fwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                const void *k, const void *v, void *o, float *lse, int partial_out,
                cudaStream_t st) {
    SimtArgs a = base_args(pl, r);
    a.q_main = q_main; a.q_branch = q_branch; a.k = k; a.v = v;
    a.o = o; a.lse_out = lse; a.partial_out = partial_out;
    return dispatch<kFwd>(pl, a, st);
}

int ba_simt_bwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                const void *k, const void *v, const float *lse, const float *delta,
                const void *d_o, int accumulate, void *dq_main, void *dq_branch, void *dk,
                void *dv, cudaStream_t st, int stages) {
    SimtArgs a = base_args(pl, r);
    a.q_main = q_main; a.q_branch = q_branch; a.k = k; a.v = v; a.d_o = d_o;
    a.lse_in = lse; a.delta_t = delta; a.row_pitch = pl->row_pitch; a.accumulate = accumulate;
    a.nlse2_t = delta + (size_t)pl->row_pitch * a.h_q;
    a.dq_main = dq_main; a.dq_branch = dq_branch; a.dk = dk; a.dv = dv;
    int rc = BA_OK;
    if (stages & BA_STAGE_DQ) rc = dispatch<kDq>(pl, a, st, (stages & BA_STAGE_PREP) != 0);
    // The two kernels write different tensors and need the same inputs: the second may run beside the first
    // (not when no row of dQ was launched: the kernel before is then the caller's, or delta)
    const bool dq_rows = (q_main && r.qm_end > r.qm_begin) || r.tok_end > r.tok_begin;
    if (rc == BA_OK && (stages & BA_STAGE_DKDV)) rc = dispatch<kDkdv>(pl, a, st, (stages & BA_STAGE_DQ) && dq_rows);
    return rc;
}
