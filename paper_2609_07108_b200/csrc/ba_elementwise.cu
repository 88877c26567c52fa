// HBM-bound elementwise kernels: Eq. (lse-merge), the backward preprocess
// delta = rowsum(dO * O), and the fp32 -> output-dtype conversion of gradient
// accumulators.  All are 16-byte vectorised, one pass over memory; merge and conversion
// are grid-stride, delta has one CTA per tile of rows and heads.
#include "ba_common.cuh"
#include "ba_sm100.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kBlocksPerSm = 8;

inline int stream_grid(int64_t work_items) {
    int64_t g = (work_items + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)kSms * kBlocksPerSm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

__device__ __forceinline__ uint2 pack_bf16x4(float4 x) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn(x.z, x.w);
    uint2 r;
    r.x = *reinterpret_cast<uint32_t *>(&lo);
    r.y = *reinterpret_cast<uint32_t *>(&hi);
    return r;
}

// Eq. (lse-merge) in max-subtracted form.  LPI = lanes per (row, head) item,
// each lane owning one float4 of the d-vector; all lanes of an item sit in one
// warp so that in-place updates (O_out == O_a, LSE_out == LSE_a) are safe.
template <int LPI, bool OUT_BF16>
__global__ void __launch_bounds__(kThreads)
lse_merge_kernel(int64_t items, const float4 *oa, const float *lse_a,   // may alias o_out / lse_out: no __restrict__
                 const float4 *__restrict__ ob, const float *__restrict__ lse_b,
                 void *o_out, float *lse_out) {
    constexpr int IPW = 32 / LPI;  // items per warp
    const int lane = threadIdx.x & 31;
    const int sub = lane % LPI;
    const int64_t warp = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    const int64_t warps = ((int64_t)gridDim.x * kThreads) >> 5;
    for (int64_t base = warp * IPW; base < items; base += warps * IPW) {
        const int64_t i = base + lane / LPI;
        const bool live = i < items;
        float la = -INFINITY, lb = -INFINITY;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (live) {
            la = lse_a[i];
            lb = lse_b[i];
            a = oa[i * LPI + sub];
            b = ob[i * LPI + sub];
        }
        __syncwarp();
        const float m = fmaxf(la, lb);
        float wa = 0.f, wb = 0.f, l = -INFINITY;
        if (m != -INFINITY) {
            const float ea = expf(la - m), eb = expf(lb - m);
            const float s = ea + eb;
            l = m + logf(s);
            const float inv = 1.0f / s;
            wa = ea * inv;
            wb = eb * inv;
        }
        if (live) {
            float4 r;
            r.x = wa * a.x + wb * b.x;
            r.y = wa * a.y + wb * b.y;
            r.z = wa * a.z + wb * b.z;
            r.w = wa * a.w + wb * b.w;
            if (OUT_BF16)
                reinterpret_cast<uint2 *>(o_out)[i * LPI + sub] = pack_bf16x4(r);
            else
                reinterpret_cast<float4 *>(o_out)[i * LPI + sub] = r;
            if (sub == 0 && lse_out) lse_out[i] = l;
        }
    }
}

template <bool OUT_BF16>
int launch_merge(int lpi, int64_t items, const float *oa, const float *la, const float *ob,
                 const float *lb, void *oo, float *lo, cudaStream_t st) {
    const int grid = stream_grid(items * lpi);
#define BA_MERGE_CASE(L)                                                                          \
    case L:                                                                                       \
        lse_merge_kernel<L, OUT_BF16><<<grid, kThreads, 0, st>>>(                                 \
            items, (const float4 *)oa, la, (const float4 *)ob, lb, oo, lo);                       \
        break;
    switch (lpi) {
        BA_MERGE_CASE(1) BA_MERGE_CASE(2) BA_MERGE_CASE(4) BA_MERGE_CASE(8) BA_MERGE_CASE(16)
        BA_MERGE_CASE(32)
        default: return BA_EUNSUPPORTED;
    }
#undef BA_MERGE_CASE
    return ba_check_launch();
}

// delta_t[h, r] = sum_d dO[r, h, d] * O[r, h, d] and nlse2_t[h, r] = -LSE[r, h] log2(e),
// both head-major with `pitch` rows per head; one 16-byte chunk per lane.  The rows are
// two segments handled by one launch: the main query rows and the branch rows of one call.
//
// Bound by the reads of O and dO.  A CTA works on 4 rows (aligned to 4) of up to 64 heads,
// which are consecutive in O and dO, with the loads of four passes in flight, keeps the
// results in shared memory and writes them head-major.  O and dO are read with an
// evict-first hint: what the caches still hold of them then is not pushed out by the rest.
// 288K rows of 32 heads x 128 (bf16) 1066 -> 720 us (6.6 TB/s), 40K rows 130 -> 97 us, 8K
// rows 28.8 -> 21.2 us; of fp32 5.7 -> 5.4 us at 3K rows of 8 heads.  Tiles of 8 or 16 rows take 28 / 27 us
// at 8K rows, plain loads 25, a batch of two passes the same, of eight 28 (fewer warps fit).
constexpr int kDeltaRows = 4, kDeltaHeads = 64;

struct DeltaSegment {
    int64_t begin, end, tiles;      // rows, tiles of kDeltaRows rows from begin rounded down
};

// 16 bytes with the evict-first hint; volatile, so that no read moves ahead of wait_prerequisites()
__device__ __forceinline__ uint4 load_once(const uint4 *p) {
    uint4 x;
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "l"(p));
    return x;
}

// (The kernel may be launched while the one that writes o and lse still runs: no pointer is __restrict__, which would let
// the compiler read through it before the wait.)
template <typename T, int LPI>
__global__ void __launch_bounds__(kThreads)
delta_kernel(const uint4 *o, const uint4 *d_o, const float *lse, float *delta_t, float *nlse2_t, DeltaSegment seg_a,
             DeltaSegment seg_b, int h_q, int64_t pitch) {
    sm100::wait_prerequisites();      // (ba_delta: the launch may come ahead of the end of the forward)
    sm100::launch_dependents();
    constexpr int kItems = kThreads / LPI;      // (row, head) items per pass
    __shared__ float s_delta[kDeltaHeads][kDeltaRows + 1], s_nlse2[kDeltaHeads][kDeltaRows + 1];
    const bool in_a = (int64_t)blockIdx.x < seg_a.tiles;
    const DeltaSegment &seg = in_a ? seg_a : seg_b;
    const int64_t tile0 = (seg.begin & ~(int64_t)(kDeltaRows - 1)) +
                          ((int64_t)blockIdx.x - (in_a ? 0 : seg_a.tiles)) * kDeltaRows;
    const int64_t r0 = max(tile0, seg.begin), r1 = min(tile0 + kDeltaRows, seg.end);
    const int rows = (int)(r1 - r0);
    const int h0 = (int)blockIdx.y * kDeltaHeads, heads = min(kDeltaHeads, h_q - h0);
    const int items = rows * heads;
    const int sub = threadIdx.x % LPI, lead = threadIdx.x / LPI;
    constexpr int kBatch = 4;                   // passes whose loads are in flight together
    for (int i0 = lead; i0 - lead < items; i0 += kBatch * kItems) {
        uint4 x[kBatch], y[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int i = min(i0 + b * kItems, items - 1);
            const int64_t e = ((r0 + i / heads) * h_q + h0 + i % heads) * LPI + sub;
            x[b] = load_once(o + e);
            y[b] = load_once(d_o + e);
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int i = i0 + b * kItems;
            float acc = 0.f;
            if (sizeof(T) == 4) {
                const float *xf = reinterpret_cast<const float *>(&x[b]);
                const float *yf = reinterpret_cast<const float *>(&y[b]);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc += xf[c] * yf[c];
            } else {
                const __nv_bfloat162 *xb = reinterpret_cast<const __nv_bfloat162 *>(&x[b]);
                const __nv_bfloat162 *yb = reinterpret_cast<const __nv_bfloat162 *>(&y[b]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float2 xf = __bfloat1622float2(xb[c]), yf = __bfloat1622float2(yb[c]);
                    acc += xf.x * yf.x + xf.y * yf.y;
                }
            }
#pragma unroll
            for (int off = LPI / 2; off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (i < items && sub == 0) s_delta[i % heads][i / heads] = acc;
        }
    }
    if ((int)threadIdx.x < items)      // kDeltaRows * kDeltaHeads == kThreads
        s_nlse2[threadIdx.x % heads][threadIdx.x / heads] =
            -lse[(r0 + threadIdx.x / heads) * h_q + h0 + threadIdx.x % heads] * 1.4426950408889634f;
    __syncthreads();
    const int r = threadIdx.x % kDeltaRows, h = threadIdx.x / kDeltaRows;
    if (r < rows && h < heads) {
        delta_t[(h0 + h) * pitch + r0 + r] = s_delta[h][r];
        nlse2_t[(h0 + h) * pitch + r0 + r] = s_nlse2[h][r];
    }
}
static_assert(kDeltaRows * kDeltaHeads == kThreads, "one thread per (row, head) of a tile");

// WIDE: src and dst on 16-byte boundaries; otherwise element by element (rows of LSE of an odd number of heads)
template <bool OUT_BF16, bool WIDE>
__global__ void __launch_bounds__(kThreads)
finalize_kernel(int64_t chunks, int64_t count, const float *__restrict__ src, void *dst) {
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x; c < chunks; c += stride) {
        const int64_t e = c * 4;
        if (WIDE && e + 4 <= count) {
            const float4 x = *reinterpret_cast<const float4 *>(src + e);
            if (OUT_BF16)
                *reinterpret_cast<uint2 *>((__nv_bfloat16 *)dst + e) = pack_bf16x4(x);
            else
                *reinterpret_cast<float4 *>((float *)dst + e) = x;
        } else {
            for (int64_t j = e; j < min(e + 4, count); ++j) {
                if (OUT_BF16) ((__nv_bfloat16 *)dst)[j] = __float2bfloat16_rn(src[j]);
                else ((float *)dst)[j] = src[j];
            }
        }
    }
}

}  // namespace

extern "C" int lse_merge(int64_t rows_heads, int d, const float *O_a, const float *LSE_a,
                         const float *O_b, const float *LSE_b, void *O_out, int out_dtype,
                         float *LSE_out, void *stream) {
    if (rows_heads < 0 || d <= 0) return BA_EINVAL;
    if (rows_heads == 0) return BA_OK;
    if (!O_a || !O_b || !LSE_a || !LSE_b || !O_out) return BA_EINVAL;
    if (d % 4 != 0 || 32 % (d / 4) != 0) return BA_EUNSUPPORTED;
    if (out_dtype != BA_FP32 && out_dtype != BA_BF16) return BA_EUNSUPPORTED;
    if (((uintptr_t)O_a | (uintptr_t)O_b | (uintptr_t)O_out) & 15) return BA_EINVAL;
    if (out_dtype == BA_BF16 && O_out == (const void *)O_a) return BA_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (out_dtype == BA_BF16)
        return launch_merge<true>(d / 4, rows_heads, O_a, LSE_a, O_b, LSE_b, O_out, LSE_out, st);
    return launch_merge<false>(d / 4, rows_heads, O_a, LSE_a, O_b, LSE_b, O_out, LSE_out, st);
}

namespace {
struct DeltaGrid {
    DeltaSegment a, b;
    dim3 grid;
    explicit DeltaGrid(const BaDelta &x) {
        auto segment = [](int64_t begin, int64_t end) {
            DeltaSegment g = {begin, end, 0};
            if (end > begin) g.tiles = (end - (begin & ~(int64_t)(kDeltaRows - 1)) + kDeltaRows - 1) / kDeltaRows;
            return g;
        };
        a = segment(x.a_begin, x.a_end);
        b = segment(x.b_begin, x.b_end);
        grid = dim3((unsigned)(a.tiles + b.tiles), (unsigned)((x.h_q + kDeltaHeads - 1) / kDeltaHeads));
    }
    bool small() const { return (int64_t)grid.x * grid.y <= 4 * kSms; }
};
}  // namespace

bool ba_delta_small(const BaDelta &x) { return DeltaGrid(x).small(); }

int ba_delta(const BaDelta &x, cudaStream_t st) {
    const DeltaGrid g(x);
    if (g.grid.x == 0) return BA_OK;
    const int lpi = x.d * (x.dtype == BA_FP32 ? 4 : 2) / 16;
    // Forward, delta and dQ follow one another in a step: each may be launched while the one before ends, and waits for
    // it at its head (640 tokens in fp32, whole step 65.5 -> 63.9 us, 4,096 in bf16 at head_dim 64 676 -> 660).  A larger
    // delta is launched as usual: its blocks would crowd the SMs that are free first (8,192 rows: 27 us instead of 24).
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    dependent_launch(cfg, attr, g.grid, kThreads, 0, st);
    if (!g.small()) cfg.numAttrs = 0;
#define BA_DELTA_LAUNCH(T, L) \
    BA_CUDA_CHECK(cudaLaunchKernelEx(&cfg, delta_kernel<T, L>, (const uint4 *)x.o, (const uint4 *)x.d_o, x.lse, x.delta_t, x.nlse2_t, g.a, g.b, x.h_q, \
                                     x.row_pitch))
    if (x.dtype == BA_FP32 && lpi == 16) BA_DELTA_LAUNCH(float, 16);
    else if (x.dtype == BA_FP32 && lpi == 32) BA_DELTA_LAUNCH(float, 32);
    else if (x.dtype == BA_BF16 && lpi == 8) BA_DELTA_LAUNCH(__nv_bfloat16, 8);
    else if (x.dtype == BA_BF16 && lpi == 16) BA_DELTA_LAUNCH(__nv_bfloat16, 16);
    else return BA_EUNSUPPORTED;
#undef BA_DELTA_LAUNCH
    return ba_check_launch();
}

extern "C" int ba_finalize_grads(const float *src, void *dst, int64_t count, int dst_dtype,
                                 void *stream) {
    if (count < 0) return BA_EINVAL;
    if (count == 0) return BA_OK;
    if (!src || !dst) return BA_EINVAL;
    if (dst_dtype != BA_FP32 && dst_dtype != BA_BF16) return BA_EUNSUPPORTED;
    if (((uintptr_t)src & 3) || ((uintptr_t)dst & (dst_dtype == BA_BF16 ? 1 : 3))) return BA_EINVAL;
    const bool wide = (((uintptr_t)src | (uintptr_t)dst) & 15) == 0;
    const int64_t chunks = (count + 3) / 4;
    const int grid = stream_grid(chunks);
    cudaStream_t st = (cudaStream_t)stream;
    auto kernel = dst_dtype == BA_BF16 ? (wide ? finalize_kernel<true, true> : finalize_kernel<true, false>)
                                       : (wide ? finalize_kernel<false, true> : finalize_kernel<false, false>);
    kernel<<<grid, kThreads, 0, st>>>(chunks, count, src, dst);
    return ba_check_launch();
}
