// Single result rows, summed over their visible pairs only.
//
// The kernels multiply whole tiles: a pair that a mask excludes enters with weight 0, and 0 x NaN (or infinity) is
// NaN.  So a row of a tile may come out as NaN although nothing that it sees is.  The kernels whose results must
// not mix rows that way (plain FMA, and head_dim 64 on the tensor cores) look at what they are about to store: a
// NaN that came by a weight of 0 cannot leave a sum any more, so finite results need no further look.  Otherwise
//   *_row_mixed   look among the rows that a result does see for the term that makes it NaN, 32 rows at a time
//   *_row_sum     form a result again, pair by pair, where there is no such term
// Inputs without NaN or infinity never get here.  head_dim 64, one chain batch of 16,384 tokens, one infinity that
// most rows see, forward / backward: 7.0 / 22.5 ms without it, 9.3 / 90 ms with it (909 / 4421 ms when every such row
// was formed again).
#pragma once

#include <limits.h>

#include "ba_common.cuh"

// What the sums read.
struct RowArgs {
    BaMeta meta;
    BaRange r;
    const void *q_main, *q_branch, *k, *v, *d_o;
    const float *nlse2_t, *delta_t;   // backward: -LSE log2(e) and delta, head-major [h_q, row_pitch]
    int64_t row_pitch;
    int h_q, h_kv, group;
    float scale, scale_log2;
};

namespace {

template <int C> struct Cols {
    float v[C];
    __device__ __forceinline__ bool all_nan() const {      // no term can change the sums any more
        bool all = true;
#pragma unroll
        for (int c = 0; c < C; ++c) all = all && v[c] != v[c];
        return all;
    }
};

// four elements as fp32
template <typename T> __device__ __forceinline__ float4 load4(const T *p);
template <> __device__ __forceinline__ float4 load4<float>(const float *p) {
    return *reinterpret_cast<const float4 *>(p);
}
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16 *p) {
    const uint2 raw = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

template <typename T, int D> __device__ __forceinline__ float row_dot(const T *a, const T *b) {
    float s = 0.f;
#pragma unroll 4
    for (int i = 0; i < D; i += 4) {
        const float4 x = load4(a + i), y = load4(b + i);
        s = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, s))));
    }
    return s;
}
template <typename T, int C> __device__ __forceinline__ void add_row(Cols<C> &out, float w, const T *p) {
#pragma unroll
    for (int c = 0; c < C; c += 4) {
        const float4 x = load4(p + c);
        out.v[c] = fmaf(w, x.x, out.v[c]);
        out.v[c + 1] = fmaf(w, x.y, out.v[c + 1]);
        out.v[c + 2] = fmaf(w, x.z, out.v[c + 2]);
        out.v[c + 3] = fmaf(w, x.w, out.v[c + 3]);
    }
}

// Columns [col0, col0 + C) of query row `row` (main row or branch token), head h:
//   forward   sum P v,  P = 2^(scale_log2 q.k + neg2) with neg2 = -maximum of the row
//   BWD       sum dS k, dS = P (dP - delta)           with neg2 = -LSE log2(e); without the factor `scale`
template <typename T, int D, bool BWD, int C>
__device__ __forceinline__ Cols<C> query_row_sum(const RowArgs &a, bool is_main, int row, int h, float neg2, int col0) {
    Cols<C> out;
#pragma unroll
    for (int c = 0; c < C; ++c) out.v[c] = 0.f;
    const int64_t n = a.meta.n_main, gr = is_main ? row : n + row;
    const T *q = (const T *)(is_main ? a.q_main : a.q_branch) + ((int64_t)row * a.h_q + h) * D;
    const T *go = BWD ? (const T *)a.d_o + (gr * a.h_q + h) * D : nullptr;
    const float dlt = BWD ? a.delta_t[h * a.row_pitch + gr] : 0.f;
    auto add = [&](int64_t key_row) {
        const int64_t off = (key_row * a.h_kv + h / a.group) * D;
        const T *k = (const T *)a.k + off, *v = (const T *)a.v + off;
        float w = exp2f(fmaf(row_dot<T, D>(q, k), a.scale_log2, neg2));
        if (BWD) w *= row_dot<T, D>(go, v) - dlt;
        add_row<T, C>(out, w, (BWD ? k : v) + col0);
    };
    if (a.r.parts & BA_PART_MAIN) {
        const int64_t lo = max((int64_t)a.meta.row_lo[gr], a.r.kv_begin), hi = min((int64_t)a.meta.row_hi[gr], a.r.kv_end - 1);
#pragma unroll 1
        for (int64_t x = lo; x <= hi; ++x) {
            add(x - a.r.kv_base);
            if ((x & 31) == 0 && out.all_nan()) break;
        }
    }
    if (!is_main && (a.r.parts & BA_PART_BRANCH)) {
#pragma unroll 1
        for (uint64_t m = a.meta.br_mask[row]; m; m &= m - 1) add(n + a.meta.br_start[row] + __ffsll((long long)m) - 1);
    }
    return out;
}

// Columns [col0, col0 + C) of the gradient of key `key` (main key or branch token) of KV head g, over the selected
// query rows that see it: dV = sum P dO, or dK = sum dS q without the factor `scale`
template <typename T, int D, int C>
__device__ __forceinline__ Cols<C> key_row_sum(const RowArgs &a, bool is_main, int key, int g, bool want_dv, int col0) {
    Cols<C> out;
#pragma unroll
    for (int c = 0; c < C; ++c) out.v[c] = 0.f;
    const int64_t n = a.meta.n_main;
    const int64_t off = ((is_main ? key - a.r.kv_base : n + key) * a.h_kv + g) * D;
    const T *k = (const T *)a.k + off, *v = (const T *)a.v + off;
    int64_t m0 = 0, m1 = 0;
    if (is_main && a.q_main) { m0 = max((int64_t)key, a.r.qm_begin); m1 = min((int64_t)a.meta.key_qend[key], a.r.qm_end); }
    const int64_t b0 = max((int64_t)(is_main ? a.meta.key_bq_begin[key] : a.meta.br_start[key]), a.r.tok_begin);
    const int64_t b1 = min((int64_t)(is_main ? a.meta.key_bq_end[key] : a.meta.br_end[key]), a.r.tok_end);
#pragma unroll 1
    for (int h = g * a.group; h < (g + 1) * a.group; ++h) {
        auto add = [&](const T *q, int64_t gr) {
            const T *go = (const T *)a.d_o + (gr * a.h_q + h) * D;
            float w = exp2f(fmaf(row_dot<T, D>(q, k), a.scale_log2, a.nlse2_t[h * a.row_pitch + gr]));
            if (!want_dv) w *= row_dot<T, D>(go, v) - a.delta_t[h * a.row_pitch + gr];
            add_row<T, C>(out, w, (want_dv ? go : q) + col0);
        };
#pragma unroll 1
        for (int64_t x = m0; x < m1; ++x) {
            add((const T *)a.q_main + (x * a.h_q + h) * D, x);
            if ((x & 31) == 0 && out.all_nan()) return out;
        }
#pragma unroll 1
        for (int64_t t = b0; t < b1; ++t) {
            if (!is_main && !((a.meta.br_mask[t] >> (key - a.meta.br_start[t])) & 1ull)) continue;
            add((const T *)a.q_branch + (t * a.h_q + h) * D, n + t);
            if ((t & 31) == 0 && out.all_nan()) return out;
        }
    }
    return out;
}

template <typename T, int D> __device__ __forceinline__ bool row_bad(const T *p) {      // holds NaN or infinity
    float s = 0.f;
#pragma unroll 4
    for (int i = 0; i < D; i += 4) {
        const float4 x = load4(p + i);
        s = fmaf(x.x, 0.f, fmaf(x.y, 0.f, fmaf(x.z, 0.f, fmaf(x.w, 0.f, s))));
    }
    return s != 0.f;
}
// the bits of `need` whose term w x[c] is finite
template <typename T, int C> __device__ __forceinline__ uint64_t still_needed(uint64_t need, float w, const T *p) {
#pragma unroll
    for (int c = 0; c < C; c += 4) {
        const float4 x = load4(p + c);
        const float t[4] = {w * x.x, w * x.y, w * x.z, w * x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (t[e] * 0.f != 0.f) need &= ~(1ull << (c + e));
    }
    return need;
}

// Whole warp, one KV head: `need` marks NaN columns of this lane's row (0: nothing asked).  True if some of them has
// no term that is not finite.
template <typename T, int D, bool BWD, int C>
__device__ __forceinline__ bool query_row_mixed(const RowArgs &a, bool is_main, int row, int h, int g, float neg2, int col0, uint64_t need) {
    const int lane = threadIdx.x & 31;
    const int64_t n = a.meta.n_main, gr = is_main ? row : n + row;
    const T *q = (const T *)(is_main ? a.q_main : a.q_branch) + ((int64_t)row * a.h_q + h) * D;
    auto term = [&](int64_t key_row) {
        const int64_t off = (key_row * a.h_kv + g) * D;
        const T *k = (const T *)a.k + off, *v = (const T *)a.v + off;
        float w = exp2f(fmaf(row_dot<T, D>(q, k), a.scale_log2, neg2));
        if (BWD) w *= row_dot<T, D>((const T *)a.d_o + (gr * a.h_q + h) * D, v) - a.delta_t[h * a.row_pitch + gr];
        need = still_needed<T, C>(need, w, (BWD ? k : v) + col0);
    };
    int lo = INT_MAX, hi = -1;
    if (need && (a.r.parts & BA_PART_MAIN)) {
        lo = max(a.meta.row_lo[gr], (int)a.r.kv_begin);
        hi = min(a.meta.row_hi[gr], (int)a.r.kv_end - 1);
    }
    const int first = __reduce_min_sync(0xffffffffu, lo), last = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll 1
    for (int x0 = first; x0 <= last; x0 += 32) {
        const int64_t off = ((x0 + lane - a.r.kv_base) * a.h_kv + g) * D;
        const bool bad = x0 + lane <= last && (row_bad<T, D>((const T *)a.k + off) || row_bad<T, D>((const T *)a.v + off));
#pragma unroll 1
        for (uint32_t m = __ballot_sync(0xffffffffu, bad); m; m &= m - 1) {
            const int x = x0 + __ffs((int)m) - 1;
            if (need && x >= lo && x <= hi) term(x - a.r.kv_base);
        }
        if (!__any_sync(0xffffffffu, need != 0)) break;
    }
    if (need && !is_main && (a.r.parts & BA_PART_BRANCH)) {
#pragma unroll 1
        for (uint64_t m = a.meta.br_mask[row]; m && need; m &= m - 1) term(n + a.meta.br_start[row] + __ffsll((long long)m) - 1);
    }
    return need != 0;
}
// The same for dV (want_dv) or dK of key `key`.
template <typename T, int D, int C>
__device__ __forceinline__ bool key_row_mixed(const RowArgs &a, bool is_main, int key, int g, bool want_dv, int col0, uint64_t need) {
    const int lane = threadIdx.x & 31;
    const int64_t n = a.meta.n_main;
    const int64_t off = ((is_main ? key - a.r.kv_base : n + key) * a.h_kv + g) * D;
    const T *k = (const T *)a.k + off, *v = (const T *)a.v + off;
    int m0 = INT_MAX, m1 = -1, b0 = INT_MAX, b1 = -1;
    if (need) {
        if (is_main && a.q_main) { m0 = max(key, (int)a.r.qm_begin); m1 = min(a.meta.key_qend[key], (int)a.r.qm_end); }
        b0 = max(is_main ? a.meta.key_bq_begin[key] : a.meta.br_start[key], (int)a.r.tok_begin);
        b1 = min(is_main ? a.meta.key_bq_end[key] : a.meta.br_end[key], (int)a.r.tok_end);
    }
#pragma unroll 1
    for (int h = g * a.group; h < (g + 1) * a.group; ++h) {
        // query rows [r0, r1) of this lane's key; rows of `src`, which is rows `base` .. of dO and the scalars
        auto scan = [&](int r0, int r1, const T *src, int64_t base, bool masked) {
            const int first = __reduce_min_sync(0xffffffffu, r0), last = __reduce_max_sync(0xffffffffu, r1) - 1;
#pragma unroll 1
            for (int x0 = first; x0 <= last; x0 += 32) {
                const int64_t x = x0 + lane, gx = base + x;
                bool bad = false;
                if (x <= last)
                    bad = a.delta_t[h * a.row_pitch + gx] * 0.f != 0.f || row_bad<T, D>(src + (x * a.h_q + h) * D) ||
                          row_bad<T, D>((const T *)a.d_o + (gx * a.h_q + h) * D);
#pragma unroll 1
                for (uint32_t m = __ballot_sync(0xffffffffu, bad); m; m &= m - 1) {
                    const int r = x0 + __ffs((int)m) - 1;
                    if (!need || r < r0 || r >= r1) continue;
                    if (masked && !((a.meta.br_mask[r] >> (key - a.meta.br_start[r])) & 1ull)) continue;
                    const int64_t gr = base + r;
                    const T *q = src + ((int64_t)r * a.h_q + h) * D, *go = (const T *)a.d_o + (gr * a.h_q + h) * D;
                    float w = exp2f(fmaf(row_dot<T, D>(q, k), a.scale_log2, a.nlse2_t[h * a.row_pitch + gr]));
                    if (!want_dv) w *= row_dot<T, D>(go, v) - a.delta_t[h * a.row_pitch + gr];
                    need = still_needed<T, C>(need, w, (want_dv ? go : q) + col0);
                }
                if (!__any_sync(0xffffffffu, need != 0)) break;
            }
        };
        scan(m0, m1, (const T *)a.q_main, 0, false);
        scan(b0, b1, (const T *)a.q_branch, n, !is_main);
    }
    return need != 0;
}
// Whole warp: x, four columns of a result (NaN columns: `nans`, 0 where nothing is asked), formed again if it is mixed.
template <typename T, int D, bool BWD>
__device__ __noinline__ float4 repair_query4(const RowArgs &a, bool is_main, int row, int h, int g, float neg2, int col0, uint64_t nans, float4 x) {
    if (query_row_mixed<T, D, BWD, 4>(a, is_main, row, h, g, neg2, col0, nans)) {
        const Cols<4> c = query_row_sum<T, D, BWD, 4>(a, is_main, row, h, neg2, col0);
        x = make_float4(c.v[0], c.v[1], c.v[2], c.v[3]);
    }
    __syncwarp();
    return x;
}
template <typename T, int D>
__device__ __noinline__ float4 repair_key4(const RowArgs &a, bool is_main, int key, int g, bool want_dv, int col0, uint64_t nans, float4 x) {
    if (key_row_mixed<T, D, 4>(a, is_main, key, g, want_dv, col0, nans)) {
        const Cols<4> c = key_row_sum<T, D, 4>(a, is_main, key, g, want_dv, col0);
        x = make_float4(c.v[0], c.v[1], c.v[2], c.v[3]);
    }
    __syncwarp();
    return x;
}

// head_dim 64, bf16.  Whole warp: `cols` columns from col0 of a row have been stored at `dst`, `nans` are the NaN ones
// among them; what is mixed is formed again, times `mul`, C columns at a time.  Inlined, and frugal with
// registers: as calls they cost a forward that makes none of them 6 % (169 -> 180 us at 4,096 tokens); this way the
// look at the sums and the code beside the key loop cost 3.5 % (175 us), and dQ with dK/dV nothing (526 us).
template <int C> __device__ __forceinline__ void store_cols(__nv_bfloat16 *dst, const Cols<C> &x, float mul) {
#pragma unroll
    for (int c = 0; c < C; c += 2) *reinterpret_cast<__nv_bfloat162 *>(dst + c) = __floats2bfloat162_rn(x.v[c] * mul, x.v[c + 1] * mul);
}
template <bool BWD, int C>
__device__ __forceinline__ void repair_query_row(const RowArgs &a, bool is_main, int row, int h, int g, float neg2, int col0, int cols,
                                                 uint64_t nans, float mul, __nv_bfloat16 *dst) {
#pragma unroll 1
    for (int c = 0; c < cols; c += C, nans >>= C) {
        const uint64_t need = nans & ((1ull << C) - 1);
        if (!__any_sync(0xffffffffu, need != 0)) continue;
        if (query_row_mixed<__nv_bfloat16, 64, BWD, C>(a, is_main, row, h, g, neg2, col0 + c, need))
            store_cols(dst + c, query_row_sum<__nv_bfloat16, 64, BWD, C>(a, is_main, row, h, neg2, col0 + c), mul);
        __syncwarp();
    }
}
template <int C>
__device__ __forceinline__ void repair_key_row(const RowArgs &a, bool is_main, int key, int g, bool want_dv, int col0, int cols,
                                               uint64_t nans, float mul, __nv_bfloat16 *dst) {
#pragma unroll 1
    for (int c = 0; c < cols; c += C, nans >>= C) {
        const uint64_t need = nans & ((1ull << C) - 1);
        if (!__any_sync(0xffffffffu, need != 0)) continue;
        if (key_row_mixed<__nv_bfloat16, 64, C>(a, is_main, key, g, want_dv, col0 + c, need))
            store_cols(dst + c, key_row_sum<__nv_bfloat16, 64, C>(a, is_main, key, g, want_dv, col0 + c), mul);
        __syncwarp();
    }
}

}  // namespace
