// Single result rows, summed over their visible pairs only.
//
// The kernels multiply whole tiles: a pair that a mask excludes enters with weight 0, and 0 x NaN (or infinity) is
// NaN.  So a row of a tile may come out as NaN although nothing that it sees is.  The kernels whose results must
// not mix rows that way (plain FMA, and head_dim 64 on the tensor cores) look at what they are about to store: a
// NaN that came by a weight of 0 cannot leave a sum any more, so finite results need no further look, and a row
// that is not finite is formed again here, pair by pair.  Inputs without NaN or infinity never get here.
#pragma once

#include "ba_common.cuh"

namespace {

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

template <int C> struct Cols {
    float v[C];
    __device__ __forceinline__ bool all_nan() const {      // no term can change the sums any more
        bool all = true;
#pragma unroll
        for (int c = 0; c < C; ++c) all = all && v[c] != v[c];
        return all;
    }
};

__device__ __forceinline__ float elem(const float *p, int i) { return p[i]; }
__device__ __forceinline__ float elem(const __nv_bfloat16 *p, int i) { return __bfloat162float(p[i]); }

template <typename T, int D> __device__ __forceinline__ float row_dot(const T *a, const T *b) {
    float s = 0.f;
#pragma unroll 8
    for (int i = 0; i < D; ++i) s = fmaf(elem(a, i), elem(b, i), s);
    return s;
}
template <typename T, int C> __device__ __forceinline__ void add_row(Cols<C> &out, float w, const T *x) {
#pragma unroll
    for (int c = 0; c < C; ++c) out.v[c] = fmaf(w, elem(x, c), out.v[c]);
}

// Columns [col0, col0 + C) of query row `row` (main row or branch token), head h:
//   forward   sum P v,  P = 2^(scale_log2 q.k + neg2) with neg2 = -maximum of the row
//   BWD       sum dS k, dS = P (dP - delta)           with neg2 = -LSE log2(e); without the factor `scale`
template <typename T, int D, bool BWD, int C>
__device__ __noinline__ Cols<C> exact_query_row(const RowArgs &a, bool is_main, int row, int h, float neg2, int col0) {
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
__device__ __noinline__ Cols<C> exact_key_row(const RowArgs &a, bool is_main, int key, int g, bool want_dv, int col0) {
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

}  // namespace
