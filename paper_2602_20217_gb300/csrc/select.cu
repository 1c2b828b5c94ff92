// a4 and a5 of the hot path: history cosines and knapsack mask selection.
//
// ks_cosine  - Sec. 2's matrix cosine, a cluster of CTAs per pair; each warp
//              takes rows in turn, one thread sums the row terms in row order.
// ks_select_mask - Sec. 3.4 integer weight normalisation (App. C latency
//              model) and the exact 0/1 knapsack of Sec. 3.3 over the 2L
//              sublayers: items processed in order 1..2L, all capacities of
//              an item in parallel across the CTA, int64 fixed-point values,
//              an item taken only on strict improvement, then a backtrack
//              from item 2L that returns the optimal mask with the smallest
//              bitmask value.  One CTA: the table is 2L x (B + 1) with B a few
//              hundred units, so the solve is a few microseconds.
#include "../../include/knapspec.h"
#include "common.cuh"
#include "internal.h"
#include "umma.cuh"

#include <algorithm>
#include <climits>
#include <cmath>

namespace ks {

// A cluster of kCosCtas CTAs per pair, a row per warp at a time: one CTA per
// pair left most of the chip idle (64 pairs on 152 SMs, a load in flight per
// lane; 64 pairs of 25 rows of 4096 fp32: 35.8 us, now 12.2 us with 16-byte
// loads, eight of each side in flight).  The warps' row terms meet in the
// first CTA's shared memory and one thread adds them in row order.
constexpr int kCosCtas = 4;
constexpr int kCosThreads = 256;

// VEC: elements per load, 16 bytes' worth or 1 (rows that are not 16-byte
// aligned).  CTAS: kCosCtas, or 1 for pairs of little work, which a cluster's
// launch and barriers would only slow down.
template <typename T, int VEC, int CTAS>
KS_DEV void cosine_pair(const T* X, const T* Y, int rows, int d, int64_t pair_stride, const int32_t* row_index,
                        float* out) {
    extern __shared__ float rowcos[];
    if (CTAS > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // this CTA's shared memory may be written
    const int64_t p = blockIdx.x / CTAS;
    const uint32_t rank = CTAS > 1 ? cluster_rank() : 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T* Xp = X + p * pair_stride;
    const T* Yp = Y + p * pair_stride;
    bool waited = CTAS == 1;
    for (int i = (int)rank + CTAS * warp; i < rows; i += CTAS * (kCosThreads / 32)) {
        const int64_t ri = row_index ? row_index[i] : i;
        const T* x = Xp + ri * d;
        const T* y = Yp + ri * d;
        float xy = 0.f, xx = 0.f, yy = 0.f;
        auto add = [&](float a, float b) {
            xy = fmaf(a, b, xy);
            xx = fmaf(a, a, xx);
            yy = fmaf(b, b, yy);
        };
        if constexpr (VEC == 1) {
#pragma unroll 8
            for (int k = lane; k < d; k += 32) add(to_float(x[k]), to_float(y[k]));
        } else {
            const uint4* xv = reinterpret_cast<const uint4*>(x);
            const uint4* yv = reinterpret_cast<const uint4*>(y);
#pragma unroll 8
            for (int k = lane; k < d / VEC; k += 32) {
                const uint4 u = xv[k], v = yv[k];
                const uint32_t a[4] = {u.x, u.y, u.z, u.w}, b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if constexpr (VEC == 4) {
                        add(__uint_as_float(a[e]), __uint_as_float(b[e]));
                    } else {
                        add(bf16_lo(a[e]), bf16_lo(b[e]));
                        add(bf16_hi(a[e]), bf16_hi(b[e]));
                    }
                }
            }
        }
        xy = warp_sum(xy);
        xx = warp_sum(xx);
        yy = warp_sum(yy);
        if (!waited) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        waited = true;
        if (lane == 0) {
            const float c = xy / (sqrtf(xx) * sqrtf(yy));
            if (CTAS == 1) rowcos[i] = c;
            else asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(&rowcos[i], 0)), "f"(c) : "memory");
        }
    }
    if (!waited) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (CTAS > 1) cluster_sync();   // the row terms are in the first CTA
    else __syncthreads();
    if (rank == 0 && threadIdx.x == 0) {
        float s = 0.f;
        for (int i = 0; i < rows; ++i) s += rowcos[i];
        out[p] = s / (float)rows;
    }
}

template <typename T, int VEC>
__global__ void __cluster_dims__(kCosCtas, 1, 1) __launch_bounds__(kCosThreads)
    cosine_kernel(const T* X, const T* Y, int rows, int d, int64_t pair_stride, const int32_t* row_index, float* out) {
    cosine_pair<T, VEC, kCosCtas>(X, Y, rows, d, pair_stride, row_index, out);
}
template <typename T, int VEC>
__global__ void __launch_bounds__(kCosThreads) cosine_small_kernel(const T* X, const T* Y, int rows, int d,
                                                                   int64_t pair_stride, const int32_t* row_index,
                                                                   float* out) {
    cosine_pair<T, VEC, 1>(X, Y, rows, d, pair_stride, row_index, out);
}

// Bytes of a pair's rows up to which one CTA takes the pair.  A loop of calls
// on 64 pairs took, in us per call with one CTA / with a cluster: 9.0 / 9.5 at
// 32 KB, 8.4 / 9.5 at 160 KB, 8.7 / 9.6 at 256 KB (16 pairs), 10.3 / 9.5 at
// 300 KB, 10.2 / 9.9 at 320 KB, 20.5 / 12.0 at 1000 KB (128 pairs).
constexpr int64_t kCosSmall = 256 * 1024;

cudaError_t launch_cosine(const void* X, const void* Y, int dtype, int64_t n_pairs, int rows, int d,
                          int64_t pair_stride, const int32_t* row_index, float* out, cudaStream_t s) {
    const size_t smem = sizeof(float) * (size_t)rows;
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    const int vec = dtype == KS_DTYPE_BF16 ? 8 : 4;   // elements of 16 bytes
    // every row of every pair starts on a 16-byte boundary
    const bool aligned = d % vec == 0 && pair_stride % vec == 0 &&
                         ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
    constexpr int64_t kMost = 1 << 28;   // pairs of a launch: the grid's limit
    const bool small = 2 * (int64_t)rows * d * (16 / vec) <= kCosSmall;
    auto run = [&](auto kern, auto kern_small, auto x, auto y) {
        for (int64_t p = 0; p < n_pairs; p += kMost) {
            const unsigned n = (unsigned)(n_pairs - p < kMost ? n_pairs - p : kMost);
            if (small)
                kern_small<<<n, kCosThreads, smem, s>>>(x + p * pair_stride, y + p * pair_stride, rows, d, pair_stride,
                                                        row_index, out + p);
            else
                kern<<<n * kCosCtas, kCosThreads, smem, s>>>(x + p * pair_stride, y + p * pair_stride, rows, d,
                                                             pair_stride, row_index, out + p);
        }
        return cudaGetLastError();
    };
    if (dtype == KS_DTYPE_BF16) {
        auto x = reinterpret_cast<const __nv_bfloat16*>(X), y = reinterpret_cast<const __nv_bfloat16*>(Y);
        return aligned ? run(cosine_kernel<__nv_bfloat16, 8>, cosine_small_kernel<__nv_bfloat16, 8>, x, y)
                       : run(cosine_kernel<__nv_bfloat16, 1>, cosine_small_kernel<__nv_bfloat16, 1>, x, y);
    }
    auto x = reinterpret_cast<const float*>(X), y = reinterpret_cast<const float*>(Y);
    return aligned ? run(cosine_kernel<float, 4>, cosine_small_kernel<float, 4>, x, y)
                   : run(cosine_kernel<float, 1>, cosine_small_kernel<float, 1>, x, y);
}

// ----------------------------------------------------------------- knapsack
constexpr int kMaxItems = 256;
constexpr int kMaxTpt = 128;   // ks_select_tpt passes at most KS_TPT_MAX_CANDIDATES; the DP stage more
constexpr int kKnapMaxThreads = 1024;

struct KnapArgs {
    int kind;                 // 0 latency model, 1 explicit units
    double c1, c2, c3;
    long long n;              // context length
    int n_items;
    int budget;               // used when budget_frac < 0
    double budget_frac;       // >= 0: budget = floor(frac * sum w)
    int units[kMaxItems];
    const float* sims;
    uint8_t* mask;
    double* objective;
    int32_t* weights_out;
    int32_t* budget_out;      // optional: the budget used
    long long* best;          // scratch [2][cap + 1]
    uint32_t* take;           // scratch: choice bits, [n_items][words of cap + 1]
    int cap;                  // capacity of the scratch tables
    int shared_cap;           // capacity of the tables in shared memory
    int n_frontier;           // > 0: also backtrack the optima of budgets floor(sum w (j + 1) / n_frontier)
    uint8_t* frontier;        // [n_frontier][n_items] masks of those budgets
};

// The tables of a budget up to `cap`: two rows of int64 values and a choice
// bit per (item, capacity).
__host__ __device__ constexpr int knap_words(int cap) { return (cap + 32) / 32; }
__host__ __device__ constexpr size_t knap_table_bytes(int n_items, int cap) {
    return sizeof(long long) * 2 * ((size_t)cap + 1) + sizeof(uint32_t) * (size_t)n_items * knap_words(cap);
}

// Items N - 1 .. 0 from capacity c; two items' words are read together (the
// second at both capacities that the first may leave).
KS_DEV void knap_backtrack(const uint32_t* take, int W, const int* w, int N, int c, uint8_t* mask) {
    int i = N - 1;
    for (; i >= 1; i -= 2) {
        const int w1 = w[i], c1 = max(c - w1, 0);
        const uint32_t t1 = (take[(size_t)i * W + (c >> 5)] >> (c & 31)) & 1u;
        const uint32_t skip = (take[(size_t)(i - 1) * W + (c >> 5)] >> (c & 31)) & 1u;
        const uint32_t took = (take[(size_t)(i - 1) * W + (c1 >> 5)] >> (c1 & 31)) & 1u;
        const uint32_t t0 = t1 ? took : skip;
        c -= (t1 ? w1 : 0) + (t0 ? w[i - 1] : 0);
        mask[i] = (uint8_t)t1;
        mask[i - 1] = (uint8_t)t0;
    }
    if (i == 0) mask[0] = (uint8_t)((take[c >> 5] >> (c & 31)) & 1u);
}

// The dynamic program over items 0 .. N - 1, two items a step: v1 is the value
// with item i decided, at c and at c - w(i + 1), and v2 the value with item
// i + 1 decided on top; each is taken only on strict improvement, exactly as
// one item at a time.  Two table reads more per capacity, half the barriers.
// Returns the row that holds the final values.
KS_DEV const long long* knap_solve(long long* cur, long long* nxt, uint32_t* take, int W, const int* w,
                                   const long long* q, int N, int cap1) {
    const int tid = threadIdx.x, T = blockDim.x;
    const int rounds = (cap1 + T - 1) / T;   // every warp does each round: the ballots are whole
    int w0 = w[0], w1 = N > 1 ? w[1] : 0;
    long long q0 = q[0], q1 = N > 1 ? q[1] : 0;
    for (int i = 0; i < N; i += 2) {
        const bool two = i + 1 < N;
        // the next pair's, while this one is worked on
        const int w2 = i + 2 < N ? w[i + 2] : 0, w3 = i + 3 < N ? w[i + 3] : 0;
        const long long q2 = i + 2 < N ? q[i + 2] : 0, q3 = i + 3 < N ? q[i + 3] : 0;
#pragma unroll 1
        for (int k = 0; k < rounds; ++k) {
            const int c = tid + k * T;
            const bool in = c < cap1;
            auto at = [&](int x) { return in && x >= 0 ? cur[x] : 0; };
            const long long a0 = at(c), a1 = at(c - w0) + q0, b0 = at(c - w1), b1 = at(c - w1 - w0) + q0;
            const bool t0 = in && c >= w0 && a1 > a0;
            const long long v1 = t0 ? a1 : a0;
            const bool s0 = c >= w1 + w0 && b1 > b0;
            const long long with1 = (s0 ? b1 : b0) + q1;
            const bool t1 = in && two && c >= w1 && with1 > v1;
            if (in) nxt[c] = t1 ? with1 : v1;
            const uint32_t m0 = __ballot_sync(0xffffffffu, t0), m1 = __ballot_sync(0xffffffffu, t1);
            if ((tid & 31) == 0 && in) {
                take[(size_t)i * W + (c >> 5)] = m0;
                if (two) take[(size_t)(i + 1) * W + (c >> 5)] = m1;
            }
        }
        __syncthreads();
        long long* tmp = cur;
        cur = nxt;
        nxt = tmp;
        w0 = w2;
        w1 = w3;
        q0 = q2;
        q1 = q3;
    }
    return cur;
}

// One CTA.  The tables are in shared memory whenever the budget fits (with
// them in global memory and a barrier per item, a 64-layer model's 128 items
// at 153 units took 50 us, most of it round trips; now 18); larger budgets
// use the caller's scratch (256 items at 16000 units: 1941 -> 880 us).
__global__ void __launch_bounds__(kKnapMaxThreads) knapsack_kernel(const KnapArgs a) {
    extern __shared__ __align__(16) unsigned char tables[];
    __shared__ int w[kMaxItems];
    __shared__ long long q[kMaxItems];
    __shared__ long long part[kKnapMaxThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = a.n_items;
    int wa = 1, wm = 1;
    if (a.kind == 0) {
        // Sec. 3.4: Delta = min(t_Attn(n), t_MLP), w = round(t / Delta), >= 1
        // explicit _rn intrinsics: no FMA contraction, the same two
        // roundings as c2 * n + c3 evaluated left to right
        const double ta = __dadd_rn(__dmul_rn(a.c2, (double)a.n), a.c3);
        const double tm = a.c1;
        const double delta = fmin(ta, tm);
        wa = max(1, (int)llround(__ddiv_rn(ta, delta)));
        wm = max(1, (int)llround(__ddiv_rn(tm, delta)));
    }
    long long sum = 0;
    for (int i = tid; i < N; i += blockDim.x) {
        // 0-based item i is sublayer i + 1: even i -> Attn, odd i -> MLP
        const int wi = (a.kind == 0) ? ((i % 2 == 0) ? wa : wm) : a.units[i];
        w[i] = wi;
        sum += wi;
        // q_i = round((1 - sigma_i) * 2^30), half away from zero, in double
        q[i] = llround(__dmul_rn(__dsub_rn(1.0, (double)a.sims[i]), 1073741824.0));
        if (a.weights_out) a.weights_out[i] = wi;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) part[warp] = sum;
    __syncthreads();
    long long SW = 0;
    for (int i = 0; i < (int)blockDim.x / 32; ++i) SW += part[i];
    long long b = a.budget;
    if (a.budget_frac >= 0.0) b = (long long)floor(__dmul_rn(a.budget_frac, (double)SW));
    if (b > a.cap) b = a.cap;
    if (b < 0) b = 0;
    const int B = (int)b, cap1 = B + 1;
    if (tid == 0 && a.budget_out) *a.budget_out = B;
    // frontier and mask backtracks: one thread each from the shared tables' bits
    auto finish = [&](const long long* values, const uint32_t* take, int W) {
        if (tid == 0) {
            knap_backtrack(take, W, w, N, B, a.mask);
            if (a.objective) *a.objective = (double)values[B] / 1073741824.0;
        }
        // The TPT stage's candidate set: the optimum of each frontier budget,
        // backtracked from the same table (the DP up to capacity c does not
        // depend on larger capacities).  One candidate per warp.
        for (int j = warp; j < a.n_frontier; j += (int)blockDim.x / 32) {
            if (lane != 0) continue;
            int c = (int)((SW * (long long)(j + 1)) / a.n_frontier);
            if (c > B) c = B;
            knap_backtrack(take, W, w, N, c, a.frontier + (size_t)j * N);
        }
    };
    if (B <= a.shared_cap) {
        long long* row = reinterpret_cast<long long*>(tables);
        uint32_t* take = reinterpret_cast<uint32_t*>(row + 2 * cap1);
        for (int c = tid; c < cap1; c += blockDim.x) row[c] = 0;
        __syncthreads();
        finish(knap_solve(row, row + cap1, take, knap_words(B), w, q, N, cap1), take, knap_words(B));
    } else {
        for (int c = tid; c < cap1; c += blockDim.x) a.best[c] = 0;
        __syncthreads();
        finish(knap_solve(a.best, a.best + (a.cap + 1), a.take, knap_words(B), w, q, N, cap1), a.take, knap_words(B));
    }
}

size_t select_scratch_bytes(int n_items, int cap) {
    const size_t best = sizeof(long long) * 2 * ((size_t)cap + 1);
    const size_t take = (size_t)n_items * ((size_t)cap + 1);
    return ((best + take + 255) / 256) * 256;
}

cudaError_t launch_select(const ks_latency* lat, const float* sims, int64_t n, int n_items, int budget,
                          double budget_frac, uint8_t* mask, double* objective, int32_t* weights,
                          int32_t* budget_out, void* scratch, int cap, cudaStream_t s, int n_frontier,
                          uint8_t* frontier) {
    KnapArgs a{};
    a.kind = lat->kind;
    a.c1 = lat->c1;
    a.c2 = lat->c2;
    a.c3 = lat->c3;
    a.n = n;
    a.n_items = n_items;
    a.budget = budget;
    a.budget_frac = budget_frac;
    if (lat->kind == 1)
        for (int i = 0; i < n_items; ++i) a.units[i] = lat->units[i];
    a.sims = sims;
    a.mask = mask;
    a.objective = objective;
    a.weights_out = weights;
    a.budget_out = budget_out;
    a.cap = cap;
    a.best = reinterpret_cast<long long*>(scratch);
    a.take = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(scratch) + sizeof(long long) * 2 * ((size_t)cap + 1));
    a.n_frontier = n_frontier;
    a.frontier = frontier;
    // The budget as the kernel computes it (its weights' sum; one more unit in
    // case a rounding differs here), for the launch only: the kernel checks
    // what fits.
    long long b = budget;
    if (budget_frac >= 0.0) {
        double sum = 0.0;
        if (lat->kind == 1) {
            for (int i = 0; i < n_items; ++i) sum += lat->units[i];
        } else {
            const double ta = lat->c2 * (double)n + lat->c3, tm = lat->c1, dl = std::fmin(ta, tm);
            sum = 0.5 * n_items * (std::fmax(1.0, std::round(ta / dl)) + std::fmax(1.0, std::round(tm / dl)));
        }
        b = (long long)std::fmin(std::floor(budget_frac * sum) + 1.0, 65536.0);
    }
    const int want = (int)std::max<long long>(0, std::min<long long>(b, cap));
    size_t smem = 0;
    a.shared_cap = -1;
    if (knap_table_bytes(n_items, want) <= 200 * 1024) {
        a.shared_cap = want;
        smem = knap_table_bytes(n_items, want);
    }
    // a capacity per thread below 512 (128 items at 153 units: 18.4 us, with
    // two per thread 22.5), above that two (64 items at 1000: 20.5 against 23.6)
    const int threads = std::min(kKnapMaxThreads, (want / (want < 512 ? 1 : 2) + 32) / 32 * 32);
    if (smem > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(knapsack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   200 * 1024);
        if (e != cudaSuccess) return e;
    }
    knapsack_kernel<<<1, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- TPT stage
// Alg. 2 after the frontier: Eq. 4's acceptance of each candidate on the
// history rows (its predicted tokens against the full layer set's), then the
// grid search of Eq. 3 over candidates (in order) x gamma = 1..D, a pair
// replacing the best only when its TPT is strictly larger.  Double
// arithmetic with explicit round-to-nearest operations in a fixed order.
struct TptArgs {
    int kind;                 // 0 latency model, 1 explicit units
    double c1, c2, c3;
    long long n;
    int units[kMaxItems];
    int n_items, n_layers;
    int K, r, D;
    const uint8_t* frontier;  // [K][n_items]
    const int32_t* tokens;    // [(K + 1) r]: candidate j's rows at j r, the full set's at K r
    uint8_t* mask_out;        // [n_items] the chosen candidate
    int32_t* info;            // [0] chosen candidate, [1] gamma
    double* out;              // [0] TPT, [1 + j] alpha of candidate j
};

// One CTA: a warp per candidate counts its matches and its sublayers, then a
// thread per (candidate, gamma) evaluates Eq. 3 with the grid search's order
// kept by the tie rule (the first of the largest values in candidate order,
// gamma ascending, which is what replacing on strictly larger finds).  One
// thread doing all of it in sequence took 50 us for 8 candidates at D = 10,
// 90 for 13 of the hidden-state DP; now 9.
__global__ void __launch_bounds__(256) tpt_kernel(const TptArgs a) {
    __shared__ double alpha[kMaxTpt], draft[kMaxTpt];
    __shared__ double best_v[8];
    __shared__ int best_i[8];
    __shared__ int sel;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double ta = 0.0, tm = 0.0;
    if (a.kind == 0) {
        ta = __dadd_rn(__dmul_rn(a.c2, (double)a.n), a.c3);
        tm = a.c1;
    }
    const int32_t* full = a.tokens + (size_t)a.K * a.r;
    for (int j = warp; j < a.K; j += 8) {
        int cnt = 0, na = 0, nm = 0;
        long long units = 0;   // whole numbers below 2^53: exact as the double sum is
        for (int i = lane; i < a.r; i += 32) cnt += a.tokens[(size_t)j * a.r + i] == full[i];
        const uint8_t* m = a.frontier + (size_t)j * a.n_items;
        for (int i = lane; i < a.n_items; i += 32)
            if (m[i]) {
                (i % 2 == 0 ? na : nm)++;
                if (a.kind == 1) units += a.units[i];
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            na += __shfl_xor_sync(0xffffffffu, na, o);
            nm += __shfl_xor_sync(0xffffffffu, nm, o);
            units += __shfl_xor_sync(0xffffffffu, units, o);
        }
        if (lane == 0) {
            alpha[j] = __ddiv_rn((double)cnt, (double)a.r);
            a.out[1 + j] = alpha[j];
            draft[j] = a.kind == 0 ? __dadd_rn(__dmul_rn((double)na, ta), __dmul_rn((double)nm, tm)) : (double)units;
        }
    }
    long long all = 0;
    if (a.kind == 1)
        for (int i = lane; i < a.n_items; i += 32) all += a.units[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    const double tt = a.kind == 0 ? __dmul_rn((double)a.n_layers, __dadd_rn(ta, tm)) : (double)all;
    __syncthreads();
    double bv = 0.0;
    int bi = INT_MAX;
    auto take = [&](double v, int i) {
        if (v > bv || (v == bv && i < bi && bi != INT_MAX)) {
            bv = v;
            bi = i;
        }
    };
    for (int q = tid; q < a.K * a.D; q += 256) {
        const int j = q / a.D, gamma = q - j * a.D + 1;
        double e = 1.0, p = 1.0;
        for (int g = 1; g <= gamma; ++g) {
            p = __dmul_rn(p, alpha[j]);
            e = __dadd_rn(e, p);   // Eq. 1 summed term by term
        }
        take(__ddiv_rn(e, __dadd_rn(__dmul_rn((double)gamma, draft[j]), tt)), q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        take(ov, oi);
    }
    if (lane == 0) {
        best_v[warp] = bv;
        best_i[warp] = bi;
    }
    __syncthreads();
    if (tid == 0) {
        for (int k = 1; k < 8; ++k) take(best_v[k], best_i[k]);
        const bool found = bi != INT_MAX;   // false only where the times overflow
        a.info[0] = found ? bi / a.D : -1;
        a.info[1] = found ? bi % a.D + 1 : 0;
        a.out[0] = bv;
        sel = found ? bi / a.D : 0;
    }
    __syncthreads();
    for (int i = tid; i < a.n_items; i += blockDim.x) a.mask_out[i] = a.frontier[(size_t)sel * a.n_items + i];
}

cudaError_t launch_tpt(const ks_latency* lat, int64_t n, int n_items, int n_layers, int K, int r, int D,
                       const uint8_t* frontier, const int32_t* tokens, uint8_t* mask_out, int32_t* info,
                       double* out, cudaStream_t s) {
    if (K < 1 || K > kMaxTpt || r < 1 || D < 1 || n_items > kMaxItems) return cudaErrorInvalidValue;
    TptArgs a{};
    a.kind = lat->kind;
    a.c1 = lat->c1;
    a.c2 = lat->c2;
    a.c3 = lat->c3;
    a.n = n;
    if (lat->kind == 1)
        for (int i = 0; i < n_items; ++i) a.units[i] = lat->units[i];
    a.n_items = n_items;
    a.n_layers = n_layers;
    a.K = K;
    a.r = r;
    a.D = D;
    a.frontier = frontier;
    a.tokens = tokens;
    a.mask_out = mask_out;
    a.info = info;
    a.out = out;
    tpt_kernel<<<1, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ks

// Sec. 3.4 / App. C: the integer weights are round(t / Delta) with Delta =
// min(t_Attn(n), t_MLP), t_Attn(n) = c2 n + c3, t_MLP = c1.  Both times must
// be positive, and the larger may be at most 65535 times the smaller (the
// limit of explicit units), or the quotient would not be a valid weight.
bool ks::latency_valid(const ks_latency* lat, int32_t n_sublayers, int64_t context_len) {
    if (!lat) return false;
    if (lat->kind == 0) {
        if (!(lat->c1 > 0.0) || !(lat->c2 >= 0.0) || !(lat->c3 >= 0.0) || !std::isfinite(lat->c1) ||
            !std::isfinite(lat->c2) || !std::isfinite(lat->c3) || context_len < 0)
            return false;
        const double ta = lat->c2 * (double)context_len + lat->c3;
        if (!(ta > 0.0) || !std::isfinite(ta)) return false;
        const double hi = std::fmax(ta, lat->c1), lo = std::fmin(ta, lat->c1);
        return hi / lo <= 65535.0;
    }
    if (lat->kind == 1) {
        if (!lat->units) return false;
        for (int i = 0; i < n_sublayers; ++i)
            if (lat->units[i] < 1 || lat->units[i] > 65535) return false;
        return true;
    }
    return false;
}

namespace ks {

// ------------------------------------------------ allocation-free variant
// Work tables of ks_select_mask_static: one array for the whole process on
// every device that loads the library, sized for KS_SELECT_STATIC_MAX_BUDGET
// units and kMaxItems sublayers (about 1.1 MB).  Host code may not use the
// symbol as an address; the device address comes from cudaGetSymbolAddress.
constexpr int kStaticCap = KS_SELECT_STATIC_MAX_BUDGET;
constexpr size_t kStaticScratchBytes =
    ((sizeof(long long) * 2 * ((size_t)kStaticCap + 1) + (size_t)kMaxItems * ((size_t)kStaticCap + 1)) + 255) / 256 *
    256;
static __device__ __align__(256) unsigned char g_select_scratch[kStaticScratchBytes];

// Device address of g_select_scratch on the current device.  Looked up on
// every call (cheap once the module is loaded), so a new primary context
// after cudaDeviceReset gets the address of its own copy of the array.
static cudaError_t static_scratch(void** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_select_scratch);
    if (e != cudaSuccess) return e;
    *out = p;
    return cudaSuccess;
}

}  // namespace ks

// ------------------------------------------------------------------- C ABI
using namespace ks;

extern "C" ks_status ks_select_mask_static(const ks_latency* lat, const float* sims, int64_t context_len,
                                           int32_t n_sublayers, int32_t budget_units, uint8_t* mask_out,
                                           double* objective_out, int32_t* weights_out, void* stream) {
    if (!sims || !mask_out) {
        set_error("ks_select_mask_static: null pointer");
        return KS_ERR_INVALID_ARG;
    }
    if (n_sublayers < 2 || n_sublayers > kMaxItems || (n_sublayers & 1) || context_len < 0) {
        set_error("ks_select_mask_static: bad n_sublayers / context_len");
        return KS_ERR_INVALID_ARG;
    }
    if (budget_units < 0 || budget_units > kStaticCap) {
        set_error("ks_select_mask_static: budget_units %d outside 0..%d (the size of the built-in tables)",
                  budget_units, kStaticCap);
        return KS_ERR_INVALID_ARG;
    }
    if (!latency_valid(lat, n_sublayers, context_len)) {
        set_error("ks_select_mask_static: bad latency model (times must be positive, ratio at most 65535)");
        return KS_ERR_INVALID_ARG;
    }
    void* scratch = nullptr;
    cudaError_t e = static_scratch(&scratch);
    if (e != cudaSuccess) {
        set_error("ks_select_mask_static: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        return KS_ERR_CUDA;
    }
    e = launch_select(lat, sims, context_len, n_sublayers, budget_units, -1.0, mask_out, objective_out, weights_out,
                      nullptr, scratch, budget_units, reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        set_error("ks_select_mask_static: %s", cudaGetErrorString(e));
        return KS_ERR_CUDA;
    }
    return KS_OK;
}

extern "C" ks_status ks_cosine(const void* X, const void* Y, int32_t dtype, int64_t n_pairs, int32_t rows,
                               int32_t d, int64_t pair_stride, const int32_t* row_index, float* out,
                               void* stream) {
    if (!X || !Y || !out) {
        set_error("ks_cosine: null pointer");
        return KS_ERR_INVALID_ARG;
    }
    if (n_pairs < 1 || n_pairs > (1 << 30) || rows < 1 || rows > 8192 || d < 1 || pair_stride < 0 ||
        (dtype != KS_DTYPE_F32 && dtype != KS_DTYPE_BF16)) {
        set_error("ks_cosine: bad size or dtype");
        return KS_ERR_INVALID_ARG;
    }
    cudaError_t e = launch_cosine(X, Y, dtype, n_pairs, rows, d, pair_stride, row_index, out,
                                  reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        set_error("ks_cosine: %s", cudaGetErrorString(e));
        return KS_ERR_CUDA;
    }
    return KS_OK;
}

extern "C" ks_status ks_fit_latency(const double* n, const double* t_attn, int32_t count, const double* t_mlp,
                                    int32_t count_mlp, ks_latency* out) {
    if (!n || !t_attn || !t_mlp || !out || count < 2 || count_mlp < 1) {
        set_error("ks_fit_latency: need at least two attention points and one MLP time");
        return KS_ERR_INVALID_ARG;
    }
    // App. C: t_Attn(n) = c2 n + c3 by least squares, t_MLP = c1 (the mean)
    double sn = 0.0, st = 0.0, c1 = 0.0;
    for (int k = 0; k < count; ++k) {
        if (!std::isfinite(n[k]) || !std::isfinite(t_attn[k]) || n[k] < 0.0) {
            set_error("ks_fit_latency: bad sample %d", k);
            return KS_ERR_INVALID_ARG;
        }
        sn += n[k];
        st += t_attn[k];
    }
    for (int k = 0; k < count_mlp; ++k) c1 += t_mlp[k];
    c1 /= count_mlp;
    const double nb = sn / count, tb = st / count;
    double sxx = 0.0, sxy = 0.0;
    for (int k = 0; k < count; ++k) {
        sxx += (n[k] - nb) * (n[k] - nb);
        sxy += (n[k] - nb) * (t_attn[k] - tb);
    }
    if (!(sxx > 0.0)) {
        set_error("ks_fit_latency: the context lengths must not all be equal");
        return KS_ERR_INVALID_ARG;
    }
    double c2 = sxy / sxx, c3 = tb - c2 * nb;
    // the model's coefficients are non-negative: a negative intercept refits
    // through the origin, a negative slope leaves the mean as the intercept
    if (c3 < 0.0) {
        double snn = 0.0, snt = 0.0;
        for (int k = 0; k < count; ++k) {
            snn += n[k] * n[k];
            snt += n[k] * t_attn[k];
        }
        c2 = snt / snn;
        c3 = 0.0;
    }
    if (c2 < 0.0) {
        c2 = 0.0;
        c3 = tb;
    }
    if (!(c1 > 0.0) || !std::isfinite(c1) || !std::isfinite(c2) || !std::isfinite(c3)) {
        set_error("ks_fit_latency: the fitted model is not valid (t_MLP must be positive)");
        return KS_ERR_INVALID_ARG;
    }
    out->kind = 0;
    out->c1 = c1;
    out->c2 = c2;
    out->c3 = c3;
    out->units = nullptr;
    return KS_OK;
}

extern "C" size_t ks_select_scratch_bytes(int32_t n_sublayers, int32_t budget_units) {
    if (n_sublayers < 2 || n_sublayers > kMaxItems || budget_units < 0 || budget_units > 65535) return 0;
    return select_scratch_bytes(n_sublayers, budget_units);
}


extern "C" ks_status ks_select_mask(const ks_latency* lat, const float* sims, int64_t context_len,
                                    int32_t n_sublayers, int32_t budget_units, uint8_t* mask_out,
                                    double* objective_out, int32_t* weights_out, void* scratch,
                                    size_t scratch_bytes, void* stream) {
    if (!sims || !mask_out || !scratch) {
        set_error("ks_select_mask: null pointer");
        return KS_ERR_INVALID_ARG;
    }
    if (n_sublayers < 2 || n_sublayers > kMaxItems || (n_sublayers & 1) || budget_units < 0 ||
        budget_units > 65535 || context_len < 0) {
        set_error("ks_select_mask: bad n_sublayers / budget / context_len");
        return KS_ERR_INVALID_ARG;
    }
    if (!latency_valid(lat, n_sublayers, context_len)) {
        set_error("ks_select_mask: bad latency model (times must be positive, ratio at most 65535)");
        return KS_ERR_INVALID_ARG;
    }
    if ((reinterpret_cast<uintptr_t>(scratch) & 15) != 0) {
        set_error("ks_select_mask: scratch must be 16-byte aligned");
        return KS_ERR_INVALID_ARG;
    }
    if (scratch_bytes < select_scratch_bytes(n_sublayers, budget_units)) {
        set_error("ks_select_mask: scratch too small");
        return KS_ERR_WORKSPACE;
    }
    cudaError_t e = launch_select(lat, sims, context_len, n_sublayers, budget_units, -1.0, mask_out,
                                  objective_out, weights_out, nullptr, scratch, budget_units,
                                  reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        set_error("ks_select_mask: %s", cudaGetErrorString(e));
        return KS_ERR_CUDA;
    }
    return KS_OK;
}
