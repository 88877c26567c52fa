// Metadata builder: varlen packing, anchors and branch masks -> per-row key
// bounds, per-token branch start / 64-bit visibility mask, per-key query ranges.
// (Paper Section 3.2: each branch query has two key sets -- the causal prefix of
// its packed main sequence up to its anchor, and its branch-local keys.)
//
// Every kernel here is safe on arbitrary (even invalid) metadata: searches are
// bounded, indices are clamped, the tree walk is capped at 64 steps.  Invalid
// metadata raises a flag that ba_plan_create reads before any data kernel can
// be launched with the plan.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "ba_common.cuh"

thread_local int g_ba_last_cuda_error = 0;

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct PlanLayout {
    size_t row_lo, row_hi, br_start, br_end, br_mask, key_qend, key_bq_begin, key_bq_end, status,
        pairs, total;
};

PlanLayout plan_layout(int64_t n, int64_t m) {
    PlanLayout l;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += align_up(bytes ? bytes : 1);
        return o;
    };
    l.row_lo = take((size_t)(n + m) * 4);
    l.row_hi = take((size_t)(n + m) * 4);
    l.br_start = take((size_t)m * 4);
    l.br_end = take((size_t)m * 4);
    l.br_mask = take((size_t)m * 8);
    l.key_qend = take((size_t)n * 4);
    l.key_bq_begin = take((size_t)n * 4);
    l.key_bq_end = take((size_t)n * 4);
    l.status = take(4);
    l.pairs = take(8);
    l.total = off;
    return l;
}

struct PlanArgs {
    int64_t n, m;
    int32_t b, a, kind, uniform_len;
    const int32_t *cu, *anchor, *offs, *parent;
    int32_t *row_lo, *row_hi, *br_start, *br_end, *key_qend, *key_bq_begin, *key_bq_end;
    uint64_t *br_mask;
    int32_t *status;
    unsigned long long *pairs;
};

// Token offset of branch b.  With no branches (A = 0) there is no offsets array
// to read -- the caller may have passed NULL -- and every offset is 0.
__device__ __forceinline__ int32_t branch_offset(const PlanArgs &p, int32_t b) {
    if (p.uniform_len > 0) return b * p.uniform_len;
    if (p.a == 0 || p.offs == nullptr) return 0;
    return p.offs[b];
}

// Largest s in [0, B) with cu[s] <= i and cu[s+1] > i (the non-empty sequence
// holding i); clamped to [0, B-1] on bad input.
__device__ __forceinline__ int32_t seq_of(const PlanArgs &p, int32_t i) {
    int32_t lo = 0, hi = p.b;  // first s with cu[s+1] > i
    while (lo < hi) {
        int32_t mid = (lo + hi) >> 1;
        if (p.cu[mid + 1] > i) hi = mid; else lo = mid + 1;
    }
    return min(lo, max(p.b - 1, 0));
}

// First branch whose anchor is >= x.
__device__ __forceinline__ int32_t first_anchor_ge(const PlanArgs &p, int32_t x) {
    int32_t lo = 0, hi = p.a;
    while (lo < hi) {
        int32_t mid = (lo + hi) >> 1;
        if (p.anchor[mid] >= x) hi = mid; else lo = mid + 1;
    }
    return lo;
}

__global__ void plan_validate_kernel(PlanArgs p) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (tid == 0) {
        if (p.cu[0] != 0 || (int64_t)p.cu[p.b] != p.n) bad = true;
        if (branch_offset(p, 0) != 0 || (int64_t)branch_offset(p, p.a) != p.m) bad = true;
    }
    for (int64_t s = tid; s < p.b; s += stride)
        if (p.cu[s + 1] < p.cu[s]) bad = true;
    for (int64_t b = tid; b < p.a; b += stride) {
        const int32_t a = p.anchor[b];
        if (a < 0 || (int64_t)a >= p.n) bad = true;
        if (b > 0 && p.anchor[b - 1] > a) bad = true;
        const int32_t len = branch_offset(p, (int32_t)b + 1) - branch_offset(p, (int32_t)b);
        if (len < 0 || len > 64) bad = true;
    }
    if (bad) atomicExch(p.status, 1);
}

__device__ __forceinline__ unsigned long long plan_main_rows(const PlanArgs &p, int64_t tid, int64_t stride) {
    unsigned long long local_pairs = 0;
    for (int64_t i = tid; i < p.n; i += stride) {
        const int32_t s = seq_of(p, (int32_t)i);
        const int32_t lo = p.cu[s], end = p.cu[s + 1];
        p.row_lo[i] = lo;
        p.row_hi[i] = (int32_t)i;
        p.key_qend[i] = end;
        p.key_bq_begin[i] = branch_offset(p, first_anchor_ge(p, (int32_t)i));
        p.key_bq_end[i] = branch_offset(p, first_anchor_ge(p, end));
        local_pairs += (unsigned long long)max((int32_t)i - lo + 1, 0);
    }
    return local_pairs;
}

__device__ __forceinline__ unsigned long long plan_branch_rows(const PlanArgs &p, int64_t tid, int64_t stride) {
    unsigned long long local_pairs = 0;
    bool bad = false;
    for (int64_t t = tid; t < p.m; t += stride) {
        // branch holding token t
        int32_t b;
        if (p.uniform_len > 0) {
            b = (int32_t)(t / p.uniform_len);
        } else {
            int32_t lo = 0, hi = p.a;  // first b with offs[b+1] > t
            while (lo < hi) {
                int32_t mid = (lo + hi) >> 1;
                if (p.offs[mid + 1] > t) hi = mid; else lo = mid + 1;
            }
            b = min(lo, p.a - 1);
        }
        const int32_t start = branch_offset(p, b), end = branch_offset(p, b + 1);
        const int32_t i = (int32_t)t - start;
        const int32_t len = end - start;
        int32_t a = p.anchor[b];
        a = max(0, min(a, (int32_t)p.n - 1));
        const int32_t s = seq_of(p, a);
        uint64_t mask = 0;
        if (i < 0 || i >= 64 || len > 64) {
            bad = true;
        } else if (p.kind == BA_MASK_CHAIN) {
            mask = (i == 63) ? ~0ull : ((2ull << i) - 1ull);
        } else if (p.kind == BA_MASK_BLOCK) {
            mask = (len >= 64) ? ~0ull : ((1ull << len) - 1ull);
        } else {
            int32_t node = i;
            for (int step = 0; step < 64 && node >= 0; ++step) {
                mask |= 1ull << node;
                const int32_t par = p.parent[start + node];
                if (par >= node || par < -1) { bad = true; break; }
                node = par;
            }
        }
        p.row_lo[p.n + t] = p.cu[s];
        p.row_hi[p.n + t] = a;
        p.br_start[t] = start;
        p.br_end[t] = end;
        p.br_mask[t] = mask;
        local_pairs += (unsigned long long)max(a - p.cu[s] + 1, 0) + (unsigned long long)__popcll(mask);
    }
    if (bad) atomicExch(p.status, 1);
    return local_pairs;
}

// Blocks [0, main_blocks) take the main rows, the others the branch rows.  p.pairs == NULL: the metadata was
// validated and counted on the host; the status word is then set here, and nothing else touches it.
__global__ void plan_rows_kernel(PlanArgs p, int main_blocks) {
    const bool main = (int)blockIdx.x < main_blocks;
    const int64_t block = main ? blockIdx.x : blockIdx.x - main_blocks;
    const int64_t tid = block * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)(main ? main_blocks : gridDim.x - main_blocks) * blockDim.x;
    unsigned long long local_pairs = main ? plan_main_rows(p, tid, stride) : plan_branch_rows(p, tid, stride);
    if (!p.pairs) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0;
        return;
    }
    for (int o = 16; o; o >>= 1) local_pairs += __shfl_xor_sync(0xffffffffu, local_pairs, o);
    if ((threadIdx.x & 31) == 0 && local_pairs) atomicAdd(p.pairs, local_pairs);
}


int grid_for(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > kSms * 16) g = kSms * 16;
    return (int)g;
}

}  // namespace

extern "C" const char *ba_status_string(int status) {
    switch (status) {
        case BA_OK: return "ok";
        case BA_EINVAL: return "invalid argument";
        case BA_EUNSUPPORTED: return "unsupported dtype, head_dim or branch length";
        case BA_EWORKSPACE: return "plan memory or workspace too small or misaligned";
        case BA_EMETA: return "metadata failed device-side validation";
        case BA_ECUDA: return "CUDA runtime error";
        case BA_ETIMEOUT: return "bounded device-side wait expired";
        default: return "unknown status";
    }
}

extern "C" int ba_last_cuda_error(void) { return g_ba_last_cuda_error; }

static int check_sizes(const ba_problem_t *p) {
    if (!p) return BA_EINVAL;
    if (p->n_main < 0 || p->n_branch < 0 || p->num_seqs < 0 || p->num_branches < 0) return BA_EINVAL;
    if (p->n_main + p->n_branch >= (int64_t)1 << 31) return BA_EUNSUPPORTED;
    if (p->h_q <= 0 || p->h_kv <= 0 || p->h_q % p->h_kv != 0) return BA_EINVAL;
    if (p->head_dim != 64 && p->head_dim != 128) return BA_EUNSUPPORTED;
    if (p->dtype != BA_BF16 && p->dtype != BA_FP32) return BA_EUNSUPPORTED;
    if (p->mask_kind < BA_MASK_CHAIN || p->mask_kind > BA_MASK_TREE) return BA_EINVAL;
    if (p->uniform_len < 0 || p->uniform_len > 64) return BA_EUNSUPPORTED;
    if (p->impl < BA_IMPL_AUTO || p->impl > BA_IMPL_TC) return BA_EINVAL;
    if (p->n_main > 0 && p->num_seqs == 0) return BA_EINVAL;
    if (p->n_branch > 0 && (p->num_branches == 0 || p->n_main == 0)) return BA_EINVAL;
    if (p->uniform_len > 0 && (int64_t)p->uniform_len * p->num_branches != p->n_branch) return BA_EINVAL;
    if (!(p->softmax_scale >= 0.0f) || isinf(p->softmax_scale)) return BA_EINVAL;
    return BA_OK;
}

extern "C" size_t ba_plan_bytes(const ba_problem_t *p) {
    if (check_sizes(p) != BA_OK) return 0;
    return plan_layout(p->n_main, p->n_branch).total;
}

// Device view of the caller's arrays and of plan_mem.  A = 0: the branch arrays are never read, whatever the
// caller passed for them.
static PlanArgs plan_args(const ba_problem_t *p, const PlanLayout &l, char *base) {
    PlanArgs a;
    a.n = p->n_main; a.m = p->n_branch; a.b = p->num_seqs; a.a = p->num_branches;
    a.kind = p->mask_kind; a.uniform_len = p->uniform_len;
    a.cu = p->cu_seqlens;
    a.anchor = p->num_branches > 0 ? p->anchor_idx : nullptr;
    a.offs = (p->num_branches > 0 && p->uniform_len == 0) ? p->branch_offsets : nullptr;
    a.parent = (p->mask_kind == BA_MASK_TREE && p->n_branch > 0) ? p->parent : nullptr;
    a.row_lo = (int32_t *)(base + l.row_lo); a.row_hi = (int32_t *)(base + l.row_hi);
    a.br_start = (int32_t *)(base + l.br_start); a.br_end = (int32_t *)(base + l.br_end);
    a.br_mask = (uint64_t *)(base + l.br_mask);
    a.key_qend = (int32_t *)(base + l.key_qend);
    a.key_bq_begin = (int32_t *)(base + l.key_bq_begin);
    a.key_bq_end = (int32_t *)(base + l.key_bq_end);
    a.status = (int32_t *)(base + l.status);
    a.pairs = (unsigned long long *)(base + l.pairs);
    return a;
}

static int launch_rows(const PlanArgs &a, cudaStream_t st) {
    const int mb = a.n > 0 ? grid_for(a.n, 256) : 0, bb = a.m > 0 ? grid_for(a.m, 256) : 0;
    if (mb + bb == 0) return BA_OK;
    plan_rows_kernel<<<mb + bb, 256, 0, st>>>(a, mb);
    return ba_check_launch();
}

// What ba_plan_create and ba_plan_create_host check before anything else.
static int check_create(const ba_problem_t *p, const void *plan_mem, size_t plan_bytes) {
    int rc = check_sizes(p);
    if (rc != BA_OK) return rc;
    if (p->num_seqs > 0 && !p->cu_seqlens) return BA_EINVAL;
    if (p->num_branches > 0 && (!p->anchor_idx || (p->uniform_len == 0 && !p->branch_offsets))) return BA_EINVAL;
    if (p->mask_kind == BA_MASK_TREE && p->n_branch > 0 && !p->parent) return BA_EINVAL;
    if (p->impl == BA_IMPL_TC && !ba_tc_supported(p)) return BA_EUNSUPPORTED;
    if (!plan_mem || plan_bytes < plan_layout(p->n_main, p->n_branch).total || ((uintptr_t)plan_mem & (kAlign - 1)))
        return BA_EWORKSPACE;
    return BA_OK;
}

// The host object; takes over `host_offsets`.
static ba_plan *new_plan(const ba_problem_t *p, const PlanArgs &a, int64_t pairs, int32_t *host_offsets) {
    ba_plan *pl = (ba_plan *)calloc(1, sizeof(ba_plan));
    if (!pl) { free(host_offsets); return nullptr; }
    pl->prob = *p;
    pl->prob.cu_seqlens = pl->prob.anchor_idx = pl->prob.branch_offsets = pl->prob.parent = nullptr;
    pl->meta.n_main = p->n_main; pl->meta.n_branch = p->n_branch;
    pl->meta.row_lo = a.row_lo; pl->meta.row_hi = a.row_hi;
    pl->meta.br_start = a.br_start; pl->meta.br_end = a.br_end; pl->meta.br_mask = a.br_mask;
    pl->meta.key_qend = a.key_qend; pl->meta.key_bq_begin = a.key_bq_begin;
    pl->meta.key_bq_end = a.key_bq_end;
    pl->scale = p->softmax_scale > 0.0f ? p->softmax_scale : 1.0f / sqrtf((float)p->head_dim);
    pl->impl = p->impl == BA_IMPL_AUTO ? (ba_tc_supported(p) ? BA_IMPL_TC : BA_IMPL_SIMT) : p->impl;
    pl->pairs = pairs;
    pl->row_pitch = ba_row_pitch(p->n_main + p->n_branch);
    pl->host_offsets = host_offsets;
    pl->dev_status = a.status;
    return pl;
}

// The checks of plan_validate_kernel and of the tree walk on host arrays, the pair count, and the branch length
// if all branches have the same (else 0).
static int check_metadata(const ba_problem_t *p, int64_t *pairs_out, int32_t *uniform_out) {
    const int32_t *cu = p->cu_seqlens, *anchor = p->anchor_idx, *offs = p->branch_offsets;
    const int32_t nb = p->num_branches, ns = p->num_seqs;
    *pairs_out = 0;
    *uniform_out = p->uniform_len;
    if (ns == 0) return BA_OK;
    if (cu[0] != 0 || (int64_t)cu[ns] != p->n_main) return BA_EMETA;
    int64_t pairs = 0;
    for (int32_t s = 0; s < ns; ++s) {
        const int64_t len = (int64_t)cu[s + 1] - cu[s];
        if (len < 0) return BA_EMETA;
        pairs += len * (len + 1) / 2;
    }
    int32_t uniform = p->uniform_len;
    if (nb == 0) {
        if (p->n_branch != 0) return BA_EMETA;
    } else if (uniform == 0) {
        if (offs[0] != 0 || (int64_t)offs[nb] != p->n_branch) return BA_EMETA;
        uniform = offs[1];
        for (int32_t b = 0; b < nb; ++b) {
            const int64_t len = (int64_t)offs[b + 1] - offs[b];
            if (len < 0 || len > 64) return BA_EMETA;
            if (len != uniform) uniform = 0;
        }
    }
    int32_t seq = 0;
    for (int32_t b = 0; b < nb; ++b) {
        const int32_t a = anchor[b];
        if (a < 0 || (int64_t)a >= p->n_main || (b > 0 && anchor[b - 1] > a)) return BA_EMETA;
        while (cu[seq + 1] <= a) ++seq;
        const int32_t start = uniform > 0 ? b * uniform : offs[b], len = uniform > 0 ? uniform : offs[b + 1] - offs[b];
        pairs += (int64_t)(a - cu[seq] + 1) * len;
        if (p->mask_kind == BA_MASK_CHAIN) pairs += (int64_t)len * (len + 1) / 2;
        else if (p->mask_kind == BA_MASK_BLOCK) pairs += (int64_t)len * len;
        else {
            int32_t depth[64];
            for (int32_t i = 0; i < len; ++i) {
                const int32_t par = p->parent[start + i];
                if (par >= i || par < -1) return BA_EMETA;
                depth[i] = par < 0 ? 1 : depth[par] + 1;
                pairs += depth[i];
            }
        }
    }
    *pairs_out = pairs;
    *uniform_out = uniform;
    return BA_OK;
}

constexpr int64_t kL2Bytes = 126 << 20;

// Number of keys that a query row tile walks, or of query rows that a key tile is walked by, per tile.
static void tile_weights(const ba_problem_t *host, int32_t uniform, const BaTiling &t, int64_t *w) {
    const int32_t *cu = host->cu_seqlens, *anchor = host->anchor_idx;
    const int32_t ns = host->num_seqs, nb = host->num_branches;
    const int64_t n = host->n_main, m = host->n_branch;
    auto seq = [&](int64_t i) { return (int32_t)(std::upper_bound(cu + 1, cu + ns, (int32_t)i) - (cu + 1)); };      // of main row i
    auto offset = [&](int64_t b) -> int64_t { return uniform > 0 ? b * uniform : host->branch_offsets[b]; };
    auto branch = [&](int64_t tok) -> int64_t {
        return uniform > 0 ? tok / uniform
                           : std::upper_bound(host->branch_offsets + 1, host->branch_offsets + nb, (int32_t)tok) - (host->branch_offsets + 1);
    };
    auto anchored = [&](int64_t key) { return nb > 0 ? offset(std::lower_bound(anchor, anchor + nb, (int32_t)key) - anchor) : 0; };
    for (int64_t i = 0; i < t.main_tiles; ++i) {
        const int64_t a = i * t.main_step, b = std::min(a + t.main_step, n) - 1;
        if (t.kind == BA_ORDER_ROWS) {
            w[i] = b - cu[seq(a)] + 1;
        } else {
            const int64_t end = cu[seq(b) + 1];
            w[i] = (t.has_main ? end - a : 0) + anchored(end) - anchored(a);
        }
    }
    for (int64_t i = 0; i < t.branch_tiles; ++i) {
        const int64_t a = i * t.branch_step, b = std::min(a + t.branch_step, m) - 1;
        w[t.main_tiles + i] = b - a + 1;      // own-branch keys / rows
        if (t.kind == BA_ORDER_ROWS) w[t.main_tiles + i] += anchor[branch(b)] - cu[seq(anchor[branch(a)])] + 1;
    }
}

void ba_add_order(ba_plan *pl, const ba_problem_t *host, const BaTiling &t) {
    const ba_problem_t &pr = pl->prob;
    const int64_t tiles = t.main_tiles + t.branch_tiles, items = tiles * pr.h_kv;
    if (tiles < 2 || tiles > kMaxOrder || ba_find_order(pl, t).n > 0) return;
    // Not where the streamed rows (K and V, or Q and dO) take more than twice the L2: tiles of one sequence have to be taken
    // together then, while that sequence's rows are there.  Time without an order against with one, chains, blocks and
    // trees, four and twelve sequences, 32/8, 16/4, 16/2 and 8/8 heads.  Forward and dQ: 0.98 to 1.16 at 50 to 175 MB, 0.99 to
    // 1.04 at 210 and 260 (one of 0.92), 0.95 to 1.04 at 330; 65,536 tokens with trees (403 MB) 0.94.  dK/dV at 32/8: 0.96 to
    // 1.19 up to 190 MB, 0.98 to 1.10 at 240, 0.95 to 1.07 at 300, 0.92 to 1.01 at 400; with fewer KV heads the gain lasts longer
    // (16/4: 1.01 to 1.12 at 300 MB, 0.97 to 1.06 at 400; 16/2: 0.96 to 1.11 at 550).  Nor for key tiles in more than 12 items
    // per SM, whose last ones are short enough as they are (8/8 heads: 0.97 to 1.03 up to 10 items, 0.94 to 1.03 from 13 on).
    const int64_t rows = (t.kind == BA_ORDER_ROWS || t.has_main ? pr.n_main : 0) + pr.n_branch;
    const int64_t streamed = 2 * rows * (t.kind == BA_ORDER_ROWS ? pr.h_kv : pr.h_q) * pr.head_dim * (pr.dtype == BA_FP32 ? 4 : 2);
    if (streamed > 2 * kL2Bytes || (t.kind == BA_ORDER_KEYS && items > 12 * kSms)) return;
    if (!pl->orders) pl->orders = (BaOrders *)calloc(1, sizeof(BaOrders));
    if (!pl->orders || pl->orders->count == kMaxOrders) return;
    int64_t w[kMaxOrder];
    tile_weights(host, pl->prob.uniform_len, t, w);
    BaOrder &o = pl->orders->order[pl->orders->count];
    // equal weights in the kernels' own order: later query rows, earlier keys first
    for (int64_t i = 0; i < tiles; ++i) o.tile[i] = (uint16_t)(t.kind == BA_ORDER_ROWS ? tiles - 1 - i : i);
    std::stable_sort(o.tile, o.tile + tiles, [&](uint16_t a, uint16_t b) { return w[a] > w[b]; });
    o.n = (int)tiles;
    pl->orders->tiling[pl->orders->count++] = t;
}

const BaOrder &ba_find_order(const ba_plan *pl, const BaTiling &t) {
    static const BaOrder none = {};
    for (int i = 0; pl->orders && i < pl->orders->count; ++i) {
        const BaTiling &x = pl->orders->tiling[i];
        if (x.kind == t.kind && x.has_main == t.has_main && x.main_tiles == t.main_tiles && x.main_step == t.main_step &&
            x.branch_tiles == t.branch_tiles && x.branch_step == t.branch_step)
            return pl->orders->order[i];
    }
    return none;
}

extern "C" int ba_plan_create(const ba_problem_t *p, void *plan_mem, size_t plan_bytes, void *stream,
                              ba_plan_t **out) {
    if (!out) return BA_EINVAL;
    *out = nullptr;
    int rc = check_create(p, plan_mem, plan_bytes);
    if (rc != BA_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const PlanArgs a = plan_args(p, plan_layout(p->n_main, p->n_branch), (char *)plan_mem);

    BA_CUDA_CHECK(cudaMemsetAsync(a.status, 0, 4, st));
    BA_CUDA_CHECK(cudaMemsetAsync(a.pairs, 0, 8, st));
    int32_t status_host = 0;
    unsigned long long pairs_host = 0;
    if (p->num_seqs > 0) {
        const int64_t work = p->num_seqs > p->num_branches ? p->num_seqs : p->num_branches;
        plan_validate_kernel<<<grid_for(work, 256), 256, 0, st>>>(a);
        if ((rc = ba_check_launch()) != BA_OK) return rc;
        // stop here on bad top-level metadata: the row kernels index with it
        BA_CUDA_CHECK(cudaMemcpyAsync(&status_host, a.status, 4, cudaMemcpyDeviceToHost, st));
        BA_CUDA_CHECK(cudaStreamSynchronize(st));
        if (status_host != 0) return BA_EMETA;
        if ((rc = launch_rows(a, st)) != BA_OK) return rc;
        BA_CUDA_CHECK(cudaMemcpyAsync(&status_host, a.status, 4, cudaMemcpyDeviceToHost, st));
        BA_CUDA_CHECK(cudaMemcpyAsync(&pairs_host, a.pairs, 8, cudaMemcpyDeviceToHost, st));
    }
    int32_t *host_offsets = nullptr;
    if (p->uniform_len == 0 && p->num_branches > 0) {
        host_offsets = (int32_t *)malloc(sizeof(int32_t) * ((size_t)p->num_branches + 1));
        if (!host_offsets) return BA_EINVAL;
        cudaError_t e = cudaMemcpyAsync(host_offsets, p->branch_offsets,
                                        sizeof(int32_t) * ((size_t)p->num_branches + 1),
                                        cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) { free(host_offsets); g_ba_last_cuda_error = (int)e; return BA_ECUDA; }
    }
    {
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { free(host_offsets); g_ba_last_cuda_error = (int)e; return BA_ECUDA; }
    }
    if (status_host != 0) { free(host_offsets); return BA_EMETA; }

    ba_plan *pl = new_plan(p, a, (int64_t)pairs_host, host_offsets);
    if (!pl) return BA_EINVAL;
    *out = pl;
    return BA_OK;
}

extern "C" int ba_plan_create_host(const ba_problem_t *host, const ba_problem_t *dev, void *plan_mem, size_t plan_bytes,
                                   void *stream, ba_plan_t **out) {
    if (!out) return BA_EINVAL;
    *out = nullptr;
    if (!host || !dev) return BA_EINVAL;
    int rc = check_create(host, plan_mem, plan_bytes);
    if (rc == BA_OK) rc = check_create(dev, plan_mem, plan_bytes);
    if (rc != BA_OK) return rc;
    if (host->n_main != dev->n_main || host->n_branch != dev->n_branch || host->num_seqs != dev->num_seqs ||
        host->num_branches != dev->num_branches || host->uniform_len != dev->uniform_len || host->mask_kind != dev->mask_kind)
        return BA_EINVAL;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    BA_CUDA_CHECK(cudaStreamIsCapturing((cudaStream_t)stream, &capture));
    if (capture != cudaStreamCaptureStatusNone) return BA_EINVAL;
    int64_t pairs = 0;
    ba_problem_t pr = *dev;
    if ((rc = check_metadata(host, &pairs, &pr.uniform_len)) != BA_OK) return rc;
    PlanArgs a = plan_args(&pr, plan_layout(pr.n_main, pr.n_branch), (char *)plan_mem);
    a.pairs = nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    if (pr.num_seqs > 0 && pr.n_main + pr.n_branch > 0) {
        if ((rc = launch_rows(a, st)) != BA_OK) return rc;
    } else {
        BA_CUDA_CHECK(cudaMemsetAsync(a.status, 0, 4, st));
    }
    int32_t *offsets = nullptr;
    if (pr.uniform_len == 0 && pr.num_branches > 0) {
        const size_t bytes = sizeof(int32_t) * ((size_t)pr.num_branches + 1);
        offsets = (int32_t *)malloc(bytes);
        if (!offsets) return BA_EINVAL;
        memcpy(offsets, host->branch_offsets, bytes);
    }
    ba_plan *pl = new_plan(&pr, a, pairs, offsets);
    if (!pl) return BA_EINVAL;
    if (pr.num_seqs > 1) {      // (one sequence: the tiles' own order is heaviest first)
        if (pl->impl == BA_IMPL_TC) {
            ba_tc_fwd_orders(pl, host);
            ba_tc_bwd_orders(pl, host);
        } else {
            ba_simt_orders(pl, host);
        }
    }
    *out = pl;
    return BA_OK;
}

extern "C" int ba_host_wait(void *event) {
    // relaxed: another stream of this thread may be capturing, and the event lies outside that capture
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    BA_CUDA_CHECK(cudaThreadExchangeStreamCaptureMode(&mode));
    const cudaError_t e = cudaEventSynchronize((cudaEvent_t)event);
    BA_CUDA_CHECK(cudaThreadExchangeStreamCaptureMode(&mode));
    BA_CUDA_CHECK(e);
    return BA_OK;
}

extern "C" int ba_plan_destroy(ba_plan_t *plan) {
    if (!plan) return BA_EINVAL;
    free(plan->host_offsets);
    free(plan->orders);
    free(plan);
    return BA_OK;
}

extern "C" int64_t ba_plan_pairs(const ba_plan_t *plan) { return plan ? plan->pairs : -1; }

extern "C" int ba_plan_tile_order(const ba_plan_t *plan, int stage, int has_main_q, int64_t *tiling, uint16_t *order, int capacity) {
    if (!plan || !tiling || (capacity > 0 && !order) || capacity < 0) return BA_EINVAL;
    if (stage != 0 && stage != BA_STAGE_DQ && stage != BA_STAGE_DKDV) return BA_EINVAL;
    BaTiling t;
    const BaOrder &o = plan->impl != BA_IMPL_TC ? ba_simt_order(plan, stage, has_main_q != 0, &t)
                       : stage == 0             ? ba_tc_fwd_order(plan, has_main_q != 0, &t)
                                                : ba_tc_bwd_order(plan, stage, has_main_q != 0, &t);
    tiling[0] = t.main_tiles; tiling[1] = t.main_step; tiling[2] = t.branch_tiles; tiling[3] = t.branch_step;
    for (int i = 0; i < o.n && i < capacity; ++i) order[i] = o.tile[i];
    return o.n;
}

extern "C" int ba_plan_impl(const ba_plan_t *plan) { return plan ? plan->impl : BA_EINVAL; }

extern "C" int ba_plan_check(ba_plan_t *plan, void *stream) {
    if (!plan) return BA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int32_t status = 0;
    BA_CUDA_CHECK(cudaMemcpyAsync(&status, plan->dev_status, 4, cudaMemcpyDeviceToHost, st));
    BA_CUDA_CHECK(cudaMemsetAsync(plan->dev_status, 0, 4, st));
    BA_CUDA_CHECK(cudaStreamSynchronize(st));
    return status == 0 ? BA_OK : BA_ETIMEOUT;
}
