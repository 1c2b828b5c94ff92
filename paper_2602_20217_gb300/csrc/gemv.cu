// Skinny GEMM kernel for fp32 models (the tiny parity workload), plus the
// TMA descriptor helpers of the bf16 kernels.
//
// Y[r][n] = sum_k W[n][k] A[r][k] for R <= 16 rows: the per-token
// projections of the Attn and MLP sublayers and the LM head (Sec. 2 decoder;
// every pass of a1 / a2).  A CTA has 16 features, each of its eight warps two
// (with SwiGLU two gate and two up rows): the lanes stride over K, every row of
// the pass is accumulated from the same weights in registers, and a butterfly
// adds the lanes.  The weights of a 512-column chunk are loaded while its
// activations are staged, the first chunk's before the previous launch is done
// (programmatic dependent launch).  What bounds it is latency (the tiny workload's
// matrices are 0.3 to 1.4 MB in L2): one feature after the other per warp, 64 per
// CTA, with K slices and a last-CTA reduction took 23 to 39 us a launch; this
// takes 4 to 6.  Results depend only on K, never on R, so rows agree bit
// for bit between passes of any size.  The optional RMSNorm prologue builds
// each row's sum of squares from the per-16-feature partials that the
// residual's producer wrote, in group order.
#include "common.cuh"
#include "internal.h"
#include "tma.cuh"

#include <cudaTypedefs.h>

#include <climits>

namespace ks {

constexpr int kGemvWarps = 8;
constexpr int kGemvThreads = 32 * kGemvWarps;
constexpr int kFeatures = 2 * kGemvWarps;     // output features per CTA (one sum-of-squares group)
constexpr int kGemvChunk = 512;               // columns staged at a time
constexpr int kMaxRows = 16;
static_assert(kFeatures == kSsGroup, "a CTA writes one sum-of-squares group");

int gemv_groups(int N) { return (N + kFeatures - 1) / kFeatures; }

int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
    }
    return n;
}

// LM head, last CTA of the launch: per row, the best candidate over groups.
KS_DEV void final_argmax(const GemvArgs& a, int groups) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int r = warp; r < a.R; r += kGemvWarps) {
        float bv = -INFINITY;
        int bi = INT_MAX;
        for (int c = lane; c < groups; c += 32) {
            const float v = __ldcg(&a.amax_val[c * kMaxRows + r]);
            const int i = __ldcg(&a.amax_idx[c * kMaxRows + r]);
            if (better(v, i, bv, bi)) { bv = v; bi = i; }
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
        }
        if (lane == 0) a.tokens[r] = (bi == INT_MAX) ? 0 : bi;
    }
}

// RB: rows the registers have room for (a.R <= RB); a row's arithmetic is the
// same in each.
template <int RB, int EPI>
__global__ void __launch_bounds__(kGemvThreads) gemv_f32_kernel(const GemvArgs a) {
    if (a.stop && *a.stop) return;   // a draft pass after the dynamic exit
    constexpr int NW = EPI == EPI_SWIGLU ? 4 : 2;           // weight rows of a warp
    constexpr int IT = kGemvChunk / 128;                    // float4 steps of a chunk
    __shared__ __align__(16) float act[RB][kGemvChunk];
    __shared__ float inv[kMaxRows];
    __shared__ float val[kFeatures][kMaxRows];              // squares of the new residual, or logits
    __shared__ int is_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = a.R, n0 = blockIdx.x * kFeatures + 2 * warp;
    const float* W = reinterpret_cast<const float*>(a.W);
    const float* in = reinterpret_cast<const float*>(a.in);
    const float* gain = reinterpret_cast<const float*>(a.norm_gain);
    const float* row[NW];
#pragma unroll
    for (int f = 0; f < NW; ++f) {
        const int n = min(n0 + (f & 1), a.N - 1);            // a feature past N repeats the last one, unused
        row[f] = W + (size_t)(n + (f >= 2 ? a.N : 0)) * a.K;
    }
    grid_launch_dependents();   // the next launch may start: it waits for this one before it reads its input
    float4 w[IT][NW];
    auto load_weights = [&](int k0) {
        const int kq = min(kGemvChunk, a.K - k0) / 4;
#pragma unroll
        for (int t = 0; t < IT; ++t)
#pragma unroll
            for (int f = 0; f < NW; ++f)
                if (lane + 32 * t < kq) w[t][f] = *reinterpret_cast<const float4*>(row[f] + k0 + 4 * (lane + 32 * t));
    };
    load_weights(0);            // before the previous launch is done
    grid_dependency_wait();
    if (gain != nullptr && tid < R) {
        float s = 0.f;
#pragma unroll 8
        for (int g = 0; g < a.ss_groups; ++g) s += a.ss_in[g * kMaxRows + tid];
        inv[tid] = rsqrtf(s / (float)a.K + a.eps);
    }
    float acc[NW][RB];
#pragma unroll
    for (int f = 0; f < NW; ++f)
#pragma unroll
        for (int r = 0; r < RB; ++r) acc[f][r] = 0.f;
    for (int k0 = 0; k0 < a.K; k0 += kGemvChunk) {           // K is a multiple of 8
        const int kq = min(kGemvChunk, a.K - k0) / 4;
        if (k0 > 0) load_weights(k0);
        __syncthreads();   // inv is written; the previous chunk's rows are read
        for (int idx = tid; idx < R * kq; idx += kGemvThreads) {
            const int r = idx / kq, k = 4 * (idx - r * kq);
            float4 x = *reinterpret_cast<const float4*>(in + (size_t)r * a.in_ld + k0 + k);
            if (gain != nullptr) {
                const float4 g = *reinterpret_cast<const float4*>(gain + k0 + k);
                const float s = inv[r];
                x = make_float4((x.x * s) * g.x, (x.y * s) * g.y, (x.z * s) * g.z, (x.w * s) * g.w);
            }
            *reinterpret_cast<float4*>(&act[r][k]) = x;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < IT; ++t) {
            if (lane + 32 * t >= kq) continue;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                if (r >= R) continue;
                const float4 x = *reinterpret_cast<const float4*>(&act[r][4 * (lane + 32 * t)]);
#pragma unroll
                for (int f = 0; f < NW; ++f)
                    acc[f][r] = fmaf(w[t][f].w, x.w,
                                     fmaf(w[t][f].z, x.z, fmaf(w[t][f].y, x.y, fmaf(w[t][f].x, x.x, acc[f][r]))));
            }
        }
    }
    // lane r takes row r's sums
    float v[NW];
#pragma unroll
    for (int f = 0; f < NW; ++f) v[f] = 0.f;
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        if (r >= R) continue;
#pragma unroll
        for (int f = 0; f < NW; ++f) {
            const float s = warp_sum(acc[f][r]);
            if (lane == r) v[f] = s;
        }
    }
    if (lane < R) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const int n = n0 + f, r = lane;
            const bool ok = n < a.N;
            if constexpr (EPI == EPI_STORE) {
                if (ok) a.out[(size_t)r * a.out_ld + n] = v[f];
            } else if constexpr (EPI == EPI_SWIGLU) {
                if (ok) reinterpret_cast<float*>(a.act)[(size_t)r * a.act_ld + n] = silu(v[f]) * v[f + 2];
            } else if constexpr (EPI == EPI_RESID) {
                float nx = 0.f;
                if (ok) {
                    float* x = a.resid + (size_t)r * a.resid_ld + n;
                    nx = *x + v[f];
                    *x = nx;
                    if (a.capture) a.capture[(size_t)r * a.capture_ld + n] = nx;
                }
                val[2 * warp + f][r] = nx * nx;
            } else {
                if (ok) a.logits[(size_t)r * a.logits_ld + n] = v[f];
                val[2 * warp + f][r] = ok ? v[f] : -INFINITY;
            }
        }
    }
    if constexpr (EPI == EPI_RESID) {
        // the sum of squares of these 16 features, in feature order
        __syncthreads();
        if (tid < R) {
            float s = 0.f;
#pragma unroll
            for (int f = 0; f < kFeatures; ++f) s += val[f][tid];
            a.ss_out[blockIdx.x * kMaxRows + tid] = s;
        }
    }
    if constexpr (EPI == EPI_LMHEAD) {
        __syncthreads();
        if (tid < R) {
            float bv = -INFINITY;
            int bi = INT_MAX;
#pragma unroll
            for (int f = 0; f < kFeatures; ++f) {
                const int n = blockIdx.x * kFeatures + f;
                if (n < a.N && better(val[f][tid], n, bv, bi)) {
                    bv = val[f][tid];
                    bi = n;
                }
            }
            a.amax_val[blockIdx.x * kMaxRows + tid] = bv;
            a.amax_idx[blockIdx.x * kMaxRows + tid] = bi;
            __threadfence();
        }
        __syncthreads();
        if (tid == 0) is_last = (atomicAdd(&a.counters[0], 1) == (int)gridDim.x - 1);
        __syncthreads();
        if (!is_last) return;
        __threadfence();
        final_argmax(a, gridDim.x);
        if (tid == 0) a.counters[0] = 0;
    }
}

// ---------------------------------------------------------------- launcher
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (encode == nullptr) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || fn == nullptr)
            return nullptr;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    return encode;
}

bool make_chunk_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t K, uint32_t box_rows,
                    uint32_t chunks) {
    auto encode = tensor_map_encoder();
    if (!encode || K % 8 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
    const cuuint32_t estr[3] = {1, 1, 1};
    if (K % 64 == 0) {
        // {64 columns, rows, K / 64 chunks}: a box is `chunks` chunks of box_rows rows
        const cuuint64_t dims[3] = {64, rows, K / 64};
        const cuuint64_t strides[2] = {K * 2, 128};
        const cuuint32_t box[3] = {64, box_rows, chunks};
        return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    const cuuint64_t dims[2] = {K, rows};
    const cuuint64_t strides[1] = {K * 2};
    const cuuint32_t box[2] = {64, box_rows};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_wide_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t K) {
    auto encode = tensor_map_encoder();
    if (!encode || K % 8 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
    const cuuint64_t dims[2] = {K, rows};
    const cuuint64_t strides[1] = {K * 2};
    const cuuint32_t box[2] = {64, 128};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_wide_kv_map(CUtensorMap* map, const void* base, uint64_t rows, uint32_t hd) {
    auto encode = tensor_map_encoder();
    if (!encode || hd % 64 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
    const cuuint64_t dims[3] = {64, rows, hd / 64};
    const cuuint64_t strides[2] = {(cuuint64_t)hd * 2, 128};
    const cuuint32_t box[3] = {64, 128, hd / 64};
    const cuuint32_t estr[3] = {1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int EPI>
static cudaError_t launch_f32(const GemvArgs& a, cudaStream_t s) {
    const int grid = gemv_groups(a.N);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGemvThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.R == 1) return cudaLaunchKernelEx(&cfg, gemv_f32_kernel<1, EPI>, a);
    if (a.R <= 8) return cudaLaunchKernelEx(&cfg, gemv_f32_kernel<8, EPI>, a);
    return cudaLaunchKernelEx(&cfg, gemv_f32_kernel<16, EPI>, a);
}

cudaError_t launch_gemv(int epi, const GemvArgs& a, cudaStream_t s) {
    // fp32 models only; bf16 projections run in the chain kernel
    if (a.R < 1 || a.R > kMaxRows) return cudaErrorInvalidValue;
    switch (epi) {
        case EPI_STORE: return launch_f32<EPI_STORE>(a, s);
        case EPI_RESID: return launch_f32<EPI_RESID>(a, s);
        case EPI_SWIGLU: return launch_f32<EPI_SWIGLU>(a, s);
        default: return launch_f32<EPI_LMHEAD>(a, s);
    }
}

}  // namespace ks
