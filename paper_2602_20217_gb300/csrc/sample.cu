// Sampling-mode speculative decoding on the device (Sec. 2.1, sampling
// branch; nucleus sampling of the Sec. 4 experiments).
//
// filter_kernel: per row of logits, the distribution a token is drawn from:
// logits / T, the top_k largest (ties: lower id first), softmax over them,
// then the shortest prefix in descending probability whose cumulative
// probability reaches top_p, renormalised.
// In a draft pass the same kernel draws the draft token with its uniform and
// keeps the support as the draft distribution q of that position.
//
// spec_accept_kernel: the acceptance of Sec. 2.1 over the drafts in order:
// draft t is accepted when u <= min(1, p_t(x) / q_t(x)); at the first
// rejection the token is drawn from norm(max(0, p_t - q_t)) over p_t's
// support (from p_t if that has no mass); after gamma acceptances one more
// token is drawn from p_gamma.
//
// Uniforms: Philox4x64 with 10 rounds (Salmon, Moraes, Dror, Shaw, SC 2011),
// key (seed, 0), counter (step, row, purpose, 0); u = the top 24 bits of the
// first output word / 2^24.  Purposes: 0 draft sample of position t, 1
// acceptance test of draft t, 2 the step's residual or bonus sample.
#include "common.cuh"
#include "internal.h"
#include "umma.cuh"

namespace ks {

namespace {

constexpr unsigned long long kPhiloxM0 = 0xD2E7470EE14C6C93ull;
constexpr unsigned long long kPhiloxM1 = 0xCA5A826395121157ull;
constexpr unsigned long long kPhiloxW0 = 0x9E3779B97F4A7C15ull;
constexpr unsigned long long kPhiloxW1 = 0xBB67AE8584CAA73Bull;
constexpr int kFilterCtas = 8;
constexpr int kFilterThreads = 1024;
constexpr int kFilterPer = 16;   // logits per thread and round: 128 K of a row at a time

KS_DEV unsigned long long philox_word0(unsigned long long c0, unsigned long long c1, unsigned long long c2,
                                       unsigned long long c3, unsigned long long k0, unsigned long long k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += kPhiloxW0;
            k1 += kPhiloxW1;
        }
        const unsigned long long hi0 = __umul64hi(kPhiloxM0, c0), lo0 = kPhiloxM0 * c0;
        const unsigned long long hi1 = __umul64hi(kPhiloxM1, c2), lo1 = kPhiloxM1 * c2;
        const unsigned long long n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    return c0;
}

KS_DEV float uniform(unsigned long long seed, unsigned long long step, int row, int purpose) {
    const unsigned long long x = philox_word0(step, (unsigned long long)row, (unsigned long long)purpose, 0ull,
                                              seed, 0ull);
    return (float)(unsigned)(x >> 40) * (1.0f / 16777216.0f);
}

// larger float -> larger key (no NaNs in logits)
KS_DEV unsigned order_key(float v) {
    const unsigned b = __float_as_uint(v);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

KS_DEV float prob_in(const int* ids, const float* probs, int n, int tok) {
    for (int j = 0; j < n; ++j)
        if (ids[j] == tok) return probs[j];
    return 0.f;
}

// inverse CDF over an ordered support: the first entry whose cumulative
// probability exceeds u (the last one if rounding leaves u above the total)
KS_DEV int draw(const int* ids, const float* probs, int n, float u) {
    float c = 0.f;
    for (int j = 0; j < n; ++j) {
        c += probs[j];
        if (u < c) return ids[j];
    }
    return ids[n - 1];
}

// Larger first, then the lower id: one 64-bit order for (logit, id).  0 is no entry.
KS_DEV unsigned long long filter_key(float v, int id) {
    return ((unsigned long long)order_key(v) << 32) | (0xFFFFFFFFu - (unsigned)id);
}
KS_DEV int filter_id(unsigned long long key) { return (int)(0xFFFFFFFFu - (unsigned)(key & 0xFFFFFFFFull)); }

// A cluster of kFilterCtas CTAs per row.  With one CTA per row, seven passes
// over the vocabulary and single-thread scans of its histograms, a row of
// 128256 logits took 212 us on one SM; now 23 us.
//   1. Each CTA takes a slice of the row, kFilterPer logits per thread in
//      registers, and finds its K best by a binary search on the bits of the
//      K-th best (key, id) pair: a count over the CTA per bit, ended as soon
//      as exactly K pairs lie at or above the bound.  All pairs differ, so
//      ties between logits need no care of their own.  Slices longer than a
//      CTA's registers go in rounds; the best so far join each round.
//   2. The CTAs' survivors meet in the first CTA's shared memory, where each
//      is ranked against all of them.
//   3. Softmax, top-p and renormalisation: exponentials and quotients one per
//      thread, the sums by one thread in support order (at most 64 terms), so
//      the arithmetic has one fixed order.
__global__ void __cluster_dims__(kFilterCtas, 1, 1) __launch_bounds__(kFilterThreads) filter_kernel(const FilterArgs a) {
    const int row = blockIdx.x / kFilterCtas;
    const int rank = (int)cluster_rank();
    const float* l = a.logits + (size_t)row * a.ld;
    const int V = a.vocab, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = min(a.top_k, min(V, kSampleMaxK));
    __shared__ __align__(16) unsigned long long cand[kFilterCtas][kSampleMaxK];   // the first CTA: everybody's survivors
    __shared__ unsigned long long kept[kSampleMaxK];                // this CTA's best so far
    __shared__ unsigned long long order[kSampleMaxK];
    __shared__ int counts[2][kFilterThreads / 32];
    __shared__ int n_kept;
    __shared__ float pr[kSampleMaxK];
    __shared__ int s_keep;
    __shared__ float s_max, s_sum, s_sum2;
    if (tid < kSampleMaxK) kept[tid] = 0ull;
    cluster_sync();   // every CTA runs: the first one's shared memory may be written

    const int slice = (V + kFilterCtas - 1) / kFilterCtas;
    const int lo = rank * slice, hi = min(V, lo + slice);
    for (int base = lo; base < hi; base += kFilterThreads * kFilterPer) {
        unsigned long long key[kFilterPer];
#pragma unroll
        for (int i = 0; i < kFilterPer; ++i) {
            const int id = base + i * kFilterThreads + tid;
            key[i] = id < hi ? filter_key(l[id], id) : 0ull;
        }
        const unsigned long long old = tid < kSampleMaxK ? kept[tid] : 0ull;
        // bound: the largest value with at least K pairs at or above it (0: all of fewer than K)
        unsigned long long bound = 0ull;
        for (int bit = 63, turn = 0; bit >= 0; --bit, turn ^= 1) {
            const unsigned long long t = bound | (1ull << bit);
            int c = old >= t;
#pragma unroll
            for (int i = 0; i < kFilterPer; ++i) c += key[i] >= t;
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) counts[turn][warp] = c;
            __syncthreads();   // two turns' counters: the next turn writes the other one
            c = __reduce_add_sync(0xffffffffu, counts[turn][lane]);
            if (c >= K) bound = t;
            if (c == K) break;
        }
        if (tid == 0) n_kept = 0;
        __syncthreads();
        auto keep = [&](unsigned long long k) {
            if (k != 0ull && k >= bound) kept[atomicAdd(&n_kept, 1)] = k;   // at most K
        };
        keep(old);
#pragma unroll
        for (int i = 0; i < kFilterPer; ++i) keep(key[i]);
        __syncthreads();
        if (tid >= n_kept && tid < kSampleMaxK) kept[tid] = 0ull;
        __syncthreads();
    }
    if (tid < kSampleMaxK)
        asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_addr(&cand[rank][tid], 0)), "l"(kept[tid])
                     : "memory");
    cluster_sync();
    if (rank != 0) return;
    // 2. ranks among all survivors
    constexpr int kAll = kFilterCtas * kSampleMaxK;
    const ulonglong2* all = reinterpret_cast<const ulonglong2*>(&cand[0][0]);
    const unsigned long long mine = tid < kAll ? (&cand[0][0])[tid] : 0ull;
    if (mine != 0ull) {
        int r = 0;
#pragma unroll 8
        for (int i = 0; i < kAll / 2; ++i) {
            const ulonglong2 v = all[i];
            r += (v.x > mine) + (v.y > mine);
        }
        if (r < K) order[r] = mine;
        if (r == 0) s_max = l[filter_id(mine)] * a.inv_t;
    }
    __syncthreads();
    // 3. softmax of l / T over the K candidates, then top-p, in support order
    if (tid < K) pr[tid] = expf(l[filter_id(order[tid])] * a.inv_t - s_max);
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        for (int j = 0; j < K; ++j) s += pr[j];
        s_sum = s;
    }
    __syncthreads();
    if (tid < K) pr[tid] = pr[tid] / s_sum;
    __syncthreads();
    if (tid == 0) {
        int keep = K;
        float c = 0.f;
        for (int j = 0; j < K; ++j) {
            c += pr[j];
            if (c >= a.top_p) {
                keep = j + 1;
                break;
            }
        }
        float s2 = 0.f;
        for (int j = 0; j < keep; ++j) s2 += pr[j];
        s_keep = keep;
        s_sum2 = s2;
        a.n[a.slot0 + row] = keep;
    }
    __syncthreads();
    int* ids = a.ids + (size_t)(a.slot0 + row) * kSampleMaxK;
    float* probs = a.probs + (size_t)(a.slot0 + row) * kSampleMaxK;
    if (tid < s_keep) {
        pr[tid] = pr[tid] / s_sum2;
        ids[tid] = filter_id(order[tid]);
        probs[tid] = pr[tid];
    }
    __syncthreads();
    if (tid == 0 && a.token_out) {
        // inverse CDF over the ordered support, as draw() does from memory
        const float u = uniform(a.seed, a.step, a.slot0 + row, 0);
        float c = 0.f;
        int j = 0;
        for (; j < s_keep - 1; ++j) {
            c += pr[j];
            if (u < c) break;
        }
        *a.token_out = filter_id(order[j]);
    }
}

__global__ void spec_accept_kernel(const AcceptSampleArgs a) {
    if (threadIdx.x != 0) return;
    const int g = a.gamma;
    const float u_last = uniform(a.seed, a.step, 0, 2);
    int acc = g, rep = -1;
    for (int t = 0; t < g; ++t) {
        const int* pi = a.p_ids + (size_t)t * kSampleMaxK;
        const float* pp = a.p_probs + (size_t)t * kSampleMaxK;
        const int* qi = a.q_ids + (size_t)t * kSampleMaxK;
        const float* qp = a.q_probs + (size_t)t * kSampleMaxK;
        const int pn = a.p_n[t], qn = a.q_n[t];
        const int x = a.rows[1 + t];
        const float px = prob_in(pi, pp, pn, x), qx = prob_in(qi, qp, qn, x);
        if (qx > 0.f && uniform(a.seed, a.step, t, 1) <= fminf(1.f, px / qx)) continue;
        // rejected: draw from norm(max(0, p - q)) over p's support, else from p
        float r[kSampleMaxK];
        float s = 0.f;
        for (int j = 0; j < pn; ++j) {
            r[j] = fmaxf(0.f, pp[j] - prob_in(qi, qp, qn, pi[j]));
            s += r[j];
        }
        if (s > 0.f) {
            for (int j = 0; j < pn; ++j) r[j] = r[j] / s;
            rep = draw(pi, r, pn, u_last);
        } else {
            rep = draw(pi, pp, pn, u_last);
        }
        acc = t;
        break;
    }
    if (rep < 0) {
        rep = draw(a.p_ids + (size_t)g * kSampleMaxK, a.p_probs + (size_t)g * kSampleMaxK, a.p_n[g], u_last);
    }
    a.result[0] = acc;
    a.result[1] = g;
    for (int i = 0; i < acc; ++i) a.result[2 + i] = a.rows[1 + i];
    a.result[2 + acc] = rep;
    a.rows[0] = rep;
}

}  // namespace

cudaError_t launch_filter(const FilterArgs& a, int rows, cudaStream_t s) {
    if (rows < 1 || a.top_k < 1 || !(a.inv_t > 0.f) || !(a.top_p > 0.f) || a.vocab < 1)
        return cudaErrorInvalidValue;
    filter_kernel<<<rows * kFilterCtas, kFilterThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_spec_accept(const AcceptSampleArgs& a, cudaStream_t s) {
    if (a.gamma < 0) return cudaErrorInvalidValue;
    spec_accept_kernel<<<1, 32, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ks
