// The hidden-state dynamic program of Alg. 1 (Sec. 3.4) on the device: the
// per-sublayer bookkeeping kernels.  The sublayer evaluations themselves are
// ordinary decoder passes (model.cu) over one state's history rows.
//
// State j (skipped weight j = 0 .. J-1) holds r rows of d floats.  For
// sublayer i:
//   dp_cos_kernel     sigma of every execute candidate E[j] and of every
//                     state G[j] against the target's X^(i) rows;
//   dp_select_kernel  the pull form: g[i, j] = E[j] when its cosine is >= the
//                     skip candidate G[j - w_i]'s (ties execute), valid when
//                     its source is valid and its cosine >= tau; column 0 is
//                     X^(i); records the choice and the validity word that
//                     gates the next evaluations;
//   dp_gather_kernel  copies the chosen rows into the next state buffer.
// dp_backtrack_kernel rebuilds each terminal state's layer set from the
// choices (at j = 0 every remaining sublayer is executed).
#include "common.cuh"
#include "internal.h"

#include <cfloat>

namespace ks {

namespace {

constexpr int kCosThreads = 1024;

// mean over the r rows of cos(A_r, B_r); A: a state's contiguous rows, B: the
// history plane's rows hidx[0..r).  blockIdx.y picks the execute candidates
// (0) or the previous states (1).  One CTA per state, a row per warp (32 rows
// in flight; with a whole CTA and three block sums per row this took 177 us
// for 13 states of 28 rows of 4096), the row terms added in row order.
__global__ void __launch_bounds__(kCosThreads) dp_cos_kernel(const float* A0, const float* A1, long long a_stride,
                                                             const float* B, const int32_t* hidx, int r, int d,
                                                             float* sig0, float* sig1) {
    const float* a = (blockIdx.y ? A1 : A0) + (size_t)blockIdx.x * a_stride;
    float* sig = blockIdx.y ? sig1 : sig0;
    __shared__ float term[kCosThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float acc = 0.f;
    for (int r0 = 0; r0 < r; r0 += kCosThreads / 32) {
        const int row = r0 + warp;
        if (row < r) {
            const float4* x = reinterpret_cast<const float4*>(a + (size_t)row * d);
            const float4* y = reinterpret_cast<const float4*>(B + (size_t)hidx[row] * d);
            float xy = 0.f, xx = 0.f, yy = 0.f;
#pragma unroll 4
            for (int k = lane; k < d / 4; k += 32) {   // d is a multiple of 8
                const float4 u = x[k], v = y[k];
                xy = fmaf(u.x, v.x, fmaf(u.y, v.y, fmaf(u.z, v.z, fmaf(u.w, v.w, xy))));
                xx = fmaf(u.x, u.x, fmaf(u.y, u.y, fmaf(u.z, u.z, fmaf(u.w, u.w, xx))));
                yy = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, yy))));
            }
            xy = warp_sum(xy);
            xx = warp_sum(xx);
            yy = warp_sum(yy);
            if (lane == 0) term[warp] = xy / (sqrtf(xx) * sqrtf(yy));
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int i = 0; i < min(kCosThreads / 32, r - r0); ++i) acc += term[i];
        __syncthreads();
    }
    if (threadIdx.x == 0) sig[blockIdx.x] = acc / (float)r;
}

// Input of a wide pass: row q of `rows`, features 256 y .. (blockIdx.y).
KS_DEV void wide_row(float v, int q, int k, int d, const __nv_bfloat16* gain, __nv_bfloat16* xg, float* ss, int ss_ld) {
    __shared__ float red[9];
    if (k < d) xg[(size_t)q * d + k] = __float2bfloat16_rn(v * __bfloat162float(gain[k]));
    const float s = block_sum<8>(v * v, red);
    if (threadIdx.x == 0) ss[(size_t)blockIdx.y * ss_ld + q] = s;
}

// grid (n r, ceil(d / 256)): row q belongs to state j0 + q / r.  Invalid
// states become zeros: their values are never used, but what lies there could
// send the attention's check of its key tiles down its slow path.
__global__ void __launch_bounds__(256) dp_prep_kernel(const float* G, int j0, const int* valid, int r, int d,
                                                      const __nv_bfloat16* gain, float* E, __nv_bfloat16* xg,
                                                      float* ss, int ss_ld) {
    const int q = blockIdx.x, k = blockIdx.y * 256 + threadIdx.x;
    const size_t at = ((size_t)j0 * r + q) * d + k;
    const bool ok = valid[j0 + q / r] == 0;
    float v = 0.f;
    if (k < d) {
        if (ok) v = G[at];
        E[at] = v;
    }
    wide_row(v, q, k, d, gain, xg, ss, ss_ld);
}

__global__ void __launch_bounds__(256) dp_head_kernel(const float* G, const int* js, int n_cand, int row0, int r,
                                                      int d, const __nv_bfloat16* gain, __nv_bfloat16* xg, float* ss,
                                                      int ss_ld) {
    const int q = blockIdx.x, k = blockIdx.y * 256 + threadIdx.x;
    const int c = (row0 + q) / r, i = row0 + q - c * r;
    const int j = c < n_cand ? js[c] : 0;
    const float v = k < d ? G[((size_t)j * r + i) * d + k] : 0.f;
    wide_row(v, q, k, d, gain, xg, ss, ss_ld);
}

// One thread per skipped weight j.  valid_*: 0 valid, 1 invalid (the value
// the decoder kernels read as their stop word).  choice: 0 execute, 1 skip,
// 2 invalid.  src: the row source of the new state (-1: X^(i), else 2 j' for
// E[j'], 2 j' + 1 for G[j']).
__global__ void dp_select_kernel(int J, int w, float tau, const int* valid_prev, const float* sig_e,
                                 const float* sig_s, int* valid_cur, float* sig_cur, uint8_t* choice, int* src) {
    const int j = threadIdx.x;
    if (j >= J) return;
    const bool e_ok = valid_prev[j] == 0;
    const bool s_ok = j >= w && valid_prev[j - w] == 0;
    const float se = j == 0 ? 1.f : sig_e[j];
    const float ss = s_ok ? sig_s[j - w] : -FLT_MAX;
    int c = 2, s = 0;
    float sg = 0.f;
    if (e_ok && (!s_ok || se >= ss)) {
        c = 0;
        sg = se;
        s = j == 0 ? -1 : 2 * j;
    } else if (s_ok) {
        c = 1;
        sg = ss;
        s = 2 * (j - w) + 1;
    }
    if (c != 2 && !(sg >= tau)) c = 2;
    valid_cur[j] = c == 2 ? 1 : 0;
    sig_cur[j] = sg;
    choice[j] = (uint8_t)c;
    src[j] = s;
}

// grid (J, r): one row of state j from its source
__global__ void __launch_bounds__(256) dp_gather_kernel(const int* src, const int* valid_cur, const float* E,
                                                        const float* G_prev, long long stride, const float* X,
                                                        const int32_t* hidx, int r, int d, float* G_cur) {
    const int j = blockIdx.x;
    if (valid_cur[j]) return;
    const int row = blockIdx.y;
    const int s = src[j];
    const float* in = s < 0 ? X + (size_t)hidx[row] * d
                            : (s & 1 ? G_prev : E) + (size_t)(s >> 1) * stride + (size_t)row * d;
    const float4* from = reinterpret_cast<const float4*>(in);
    float4* out = reinterpret_cast<float4*>(G_cur + (size_t)j * stride + (size_t)row * d);
    for (int k = threadIdx.x; k < d / 4; k += 256) out[k] = from[k];   // d is a multiple of 8
}

// one thread per candidate: candidate c is terminal state js[c]
__global__ void dp_backtrack_kernel(int n_cand, const int* js, int n_items, int J, const uint8_t* choices,
                                    const int* w, uint8_t* masks) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_cand) return;
    int j = js[c];
    uint8_t* m = masks + (size_t)c * n_items;
    for (int i = n_items; i >= 1; --i) {
        const uint8_t ch = choices[(size_t)(i - 1) * J + j];
        if (j == 0 || ch == 0) {
            m[i - 1] = 1;
        } else {
            m[i - 1] = 0;
            j -= w[i - 1];
        }
    }
}

// the terminal candidates in executed-weight order (j descending) and their count
__global__ void dp_candidates_kernel(int J, const int* valid, int* js, int* n_cand) {
    if (threadIdx.x != 0) return;
    int n = 0;
    for (int j = J - 1; j >= 0; --j)
        if (valid[j] == 0) js[n++] = j;
    *n_cand = n;
}

}  // namespace

cudaError_t launch_dp_cos(const float* A0, const float* A1, long long stride, int n, const float* B,
                          const int32_t* hidx, int r, int d, float* sig0, float* sig1, cudaStream_t s) {
    if (n < 1) return cudaSuccess;
    dp_cos_kernel<<<dim3(n, 2), kCosThreads, 0, s>>>(A0, A1, stride, B, hidx, r, d, sig0, sig1);
    return cudaGetLastError();
}

cudaError_t launch_dp_prep(const float* G, int j0, int n, const int* valid, int r, int d, const __nv_bfloat16* gain,
                           float* E, __nv_bfloat16* xg, float* ss, int ss_ld, cudaStream_t s) {
    dp_prep_kernel<<<dim3(n * r, (d + 255) / 256), 256, 0, s>>>(G, j0, valid, r, d, gain, E, xg, ss, ss_ld);
    return cudaGetLastError();
}

cudaError_t launch_dp_head(const float* G, const int* js, int n_cand, int row0, int rows, int r, int d,
                           const __nv_bfloat16* gain, __nv_bfloat16* xg, float* ss, int ss_ld, cudaStream_t s) {
    dp_head_kernel<<<dim3(rows, (d + 255) / 256), 256, 0, s>>>(G, js, n_cand, row0, r, d, gain, xg, ss, ss_ld);
    return cudaGetLastError();
}

cudaError_t launch_dp_select(int J, int w, float tau, const int* valid_prev, const float* sig_e, const float* sig_s,
                             int* valid_cur, float* sig_cur, uint8_t* choice, int* src, cudaStream_t s) {
    if (J < 1 || J > 1024) return cudaErrorInvalidValue;
    dp_select_kernel<<<1, J, 0, s>>>(J, w, tau, valid_prev, sig_e, sig_s, valid_cur, sig_cur, choice, src);
    return cudaGetLastError();
}

cudaError_t launch_dp_gather(int J, const int* src, const int* valid_cur, const float* E, const float* G_prev,
                             long long stride, const float* X, const int32_t* hidx, int r, int d, float* G_cur,
                             cudaStream_t s) {
    dp_gather_kernel<<<dim3(J, r), 256, 0, s>>>(src, valid_cur, E, G_prev, stride, X, hidx, r, d,
                                                              G_cur);
    return cudaGetLastError();
}

cudaError_t launch_dp_backtrack(const int* js, int n_cand, int n_items, int J, const uint8_t* choices, const int* w,
                                uint8_t* masks, cudaStream_t s) {
    if (n_cand < 1) return cudaSuccess;
    dp_backtrack_kernel<<<(n_cand + 127) / 128, 128, 0, s>>>(n_cand, js, n_items, J, choices, w, masks);
    return cudaGetLastError();
}

cudaError_t launch_dp_candidates(int J, const int* valid, int* js, int* n_cand, cudaStream_t s) {
    dp_candidates_kernel<<<1, 32, 0, s>>>(J, valid, js, n_cand);
    return cudaGetLastError();
}

}  // namespace ks
