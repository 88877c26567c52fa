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
    int depth, num_branches, branch_len, branch_tiles_per_depth;
    int *status;
    RowArgs rows;                     // head_dim 64: rows that are formed again one by one
};

// Branch tokens per branch key tile.  Branches of one length: a tile that starts and ends with a branch is seen
// by its own tokens only (chains of three: 126 keys and 128 query rows instead of 128 and up to 135, which
// costs a third 64-row step per head), unless more than an eighth of the lanes would stay empty.
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

}  // namespace
