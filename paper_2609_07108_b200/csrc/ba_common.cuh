// Shared declarations of the branch-attention CUDA library (internal).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "branch_attn.h"

// Device-side view of the metadata a plan holds (all pointers into plan_mem).
// Rows are numbered "main rows [0, N) then branch tokens [N, N + M)".
struct BaMeta {
    int64_t n_main, n_branch;
    const int32_t *row_lo;        // [N+M] first visible main key (start of the row's sequence)
    const int32_t *row_hi;        // [N+M] last visible main key (own index, or the anchor)
    const int32_t *br_start;      // [M] first token of the token's own branch
    const int32_t *br_end;        // [M] one past the last token of the token's own branch
    const uint64_t *br_mask;      // [M] bit u set: the token sees token br_start + u
    const int32_t *key_qend;      // [N] one past the last main query row that sees key x
    const int32_t *key_bq_begin;  // [N] first branch token whose anchor is >= x
    const int32_t *key_bq_end;    // [N] first branch token anchored beyond x's sequence
};

constexpr int kSms = 148;          // B200

// The order in which a kernel takes the tiles of a call over everything: heaviest first, over all sequences, so that
// the CTAs end together (the tiles' own numbering goes sequence by sequence).  Formed with the plan, handed to the
// kernels by value.  n = 0: the kernel's own rule.
constexpr int kMaxOrder = 1536;
struct BaOrder {
    int n;
    uint16_t tile[kMaxOrder];
};
// What an order was formed for: query row tiles or key tiles; numbers of tiles and rows per tile, main part and
// branch part; whether main rows are queries.
enum { BA_ORDER_ROWS, BA_ORDER_KEYS };
struct BaTiling {
    int kind, has_main;
    int64_t main_tiles, main_step, branch_tiles, branch_step;
};
constexpr int kMaxOrders = 8;
struct BaOrders {
    int count;
    BaTiling tiling[kMaxOrders];
    BaOrder order[kMaxOrders];
};

struct ba_plan {
    ba_problem_t prob;            // copy; the metadata pointers in it are NOT kept alive
    BaMeta meta;
    float scale;
    int impl;                     // BA_IMPL_SIMT or BA_IMPL_TC (resolved)
    int64_t pairs;
    int64_t row_pitch;            // rows per head of the head-major backward scratch (>= N + M + 128)
    int32_t *host_offsets;        // host copy of branch_offsets (NULL when uniform_len > 0)
    int32_t *dev_status;          // one int32 in plan_mem: device-side status word
    BaOrders *orders;             // or NULL
};

// Query / key selection of one call (monolithic = everything).
struct BaRange {
    int64_t qm_begin, qm_end;     // main query rows
    int64_t tok_begin, tok_end;   // branch tokens (query side and branch-key side)
    int64_t kv_begin, kv_end;     // main keys
    int64_t kv_base;              // first row that K, V (and dK, dV) hold: 0, or kv_begin on a received shard
    int parts;
};

// Backward preprocess of one call (ba_delta): inputs, head-major scratch, rows [a_begin, a_end) and [b_begin, b_end)
// (either may be empty)
struct BaDelta {
    const void *o, *d_o;
    const float *lse;
    float *delta_t, *nlse2_t;
    int64_t row_pitch, a_begin, a_end, b_begin, b_end;
    int h_q, d, dtype;
};

static inline bool ba_whole_call(const ba_plan *pl, const BaRange &r, bool has_main) {
    return (!has_main || (r.qm_begin == 0 && r.qm_end == pl->prob.n_main)) && r.tok_begin == 0 && r.tok_end == pl->prob.n_branch &&
           r.kv_begin == 0 && r.kv_end == pl->prob.n_main && r.kv_base == 0 && r.parts == (BA_PART_MAIN | BA_PART_BRANCH);
}
static inline BaRange ba_everything(const ba_plan *pl) {
    return {0, pl->prob.n_main, 0, pl->prob.n_branch, 0, pl->prob.n_main, 0, BA_PART_MAIN | BA_PART_BRANCH};
}
// ba_plan.cu: forms an order (`host`: problem with host arrays) and keeps it; finds it again (or an empty one)
void ba_add_order(ba_plan *pl, const ba_problem_t *host, const BaTiling &t);
const BaOrder &ba_find_order(const ba_plan *pl, const BaTiling &t);
// the tilings that the kernels use for calls over everything
void ba_tc_fwd_orders(ba_plan *pl, const ba_problem_t *host);
void ba_tc_bwd_orders(ba_plan *pl, const ba_problem_t *host);
void ba_simt_orders(ba_plan *pl, const ba_problem_t *host);
// the order that the launch of such a call finds (stage: 0 forward, BA_STAGE_DQ, BA_STAGE_DKDV), and the tiling
const BaOrder &ba_tc_fwd_order(const ba_plan *pl, bool has_main, BaTiling *t);
const BaOrder &ba_tc_bwd_order(const ba_plan *pl, int stage, bool has_main, BaTiling *t);
const BaOrder &ba_simt_order(const ba_plan *pl, int stage, bool has_main, BaTiling *t);

extern thread_local int g_ba_last_cuda_error;

#define BA_CUDA_CHECK(expr)                                  \
    do {                                                     \
        cudaError_t e__ = (expr);                            \
        if (e__ != cudaSuccess) {                            \
            g_ba_last_cuda_error = (int)e__;                 \
            return BA_ECUDA;                                 \
        }                                                    \
    } while (0)

static inline int ba_check_launch() {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_ba_last_cuda_error = (int)e;
        return BA_ECUDA;
    }
    return BA_OK;
}

// Launch that may come ahead of the end of the kernel before it in the stream (which the new kernel has to wait for
// itself, before it reads or writes anything)
static inline void dependent_launch(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, dim3 grid, unsigned threads, size_t smem, cudaStream_t st) {
    cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

// weights of Eq. (lse-merge) for merging (lse_p, O_p * inv) into the running pair with lse_a
__device__ __forceinline__ void merge_weights(float lse_a, float lse_p, float inv, float &lse_out, float &w_old, float &w_new) {
    const float mx = fmaxf(lse_a, lse_p);
    if (mx == -INFINITY) {
        lse_out = -INFINITY; w_new = 0.f; w_old = 0.f;
    } else {
        const float ea = expf(lse_a - mx), ep = expf(lse_p - mx), s = ea + ep;
        lse_out = mx + logf(s);
        w_old = ea / s;
        w_new = ep / s * inv;
    }
}

// --- kernels implemented in the other translation units -------------------
// Plain-FMA path (ba_simt.cu); partial_out as in ba_tc_fwd
int ba_simt_fwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                const void *k, const void *v, void *o, float *lse, int partial_out,
                cudaStream_t st);
int ba_simt_bwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                const void *k, const void *v, const float *lse, const float *delta,
                const void *d_o, int accumulate, void *dq_main, void *dq_branch, void *dk,
                void *dv, cudaStream_t st, int stages);
// Tensor-core path (ba_tc_fwd.cu / ba_tc_bwd.cu / ba_tc_dkdv.cu)
// partial_out: 0 = final layout in the input dtype, 1 = compact fp32, 2 = compact fp32 merged in place
// depth > 0: step-major call (queries = the depth-`depth` tokens of branches [r.tok_begin, r.tok_end),
// q_branch / o / lse indexed by branch, branch keys stored depth-major after the main rows).
// ba_tc_bwd runs BA_STAGE_PREP (`prep`) itself: whatever it refuses is refused before it launches anything.
int ba_tc_fwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
              const void *k, const void *v, void *o, float *lse, int partial_out,
              cudaStream_t st, int depth = 0);
int ba_tc_bwd(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
              const void *k, const void *v, const BaDelta &prep, int accumulate, void *dq_main,
              void *dq_branch, void *dk, void *dv, cudaStream_t st, int stages, int depth = 0);
// One-kernel backward (ba_tc_bwd_fused.cu): dq_* are fp32 accumulators (atomic adds) in either mode
int ba_tc_bwd_fused(const ba_plan *pl, const BaRange &r, const void *q_main, const void *q_branch,
                    const void *k, const void *v, const float *delta, const void *d_o,
                    int accumulate, void *dq_main, void *dq_branch, void *dk, void *dv,
                    cudaStream_t st);
bool ba_tc_supported(const ba_problem_t *p);
// Head_dim 64 with fp32 results (partial forwards, accumulated gradients) stays on the plain-FMA kernels: the
// tensor-core kernels carry P and dS as bf16 pairs (16 bits of mantissa), which bf16 results do not show and fp32
// results do.  Against fp64, 1,600 .. 3,000 tokens with chains, plain FMA / tensor cores, 2-norm: O 1e-7 .. 3e-7 /
// 2e-6, dQ 2e-7 .. 5e-7 / 3e-6, dK and dV 4e-7 .. 7e-7 / 4e-6 .. 1.4e-5.
// So do, as ever, tensors that are not 16-byte aligned (`addresses`: theirs, or-ed): tensor maps need that, the
// plain-FMA kernels 8 bytes.
static inline bool ba_use_tc(const ba_plan *pl, bool fp32_out, uintptr_t addresses) {
    return pl->impl == BA_IMPL_TC && !(pl->prob.head_dim == 64 && (fp32_out || (addresses & 15)));
}
// Elementwise (ba_elementwise.cu)
// Backward preprocess into head-major scratch [h_q, row_pitch]:
//   delta_t[h, r] = <dO[r, h], O[r, h]>,  nlse2_t[h, r] = -LSE[r, h] * log2(e)
// for the two row segments of `x`
int ba_delta(const BaDelta &x, cudaStream_t st);
// at most four CTAs to an SM
bool ba_delta_small(const BaDelta &x);
static inline int64_t ba_row_pitch(int64_t rows) { return (rows + 128 + 63) / 64 * 64; }
