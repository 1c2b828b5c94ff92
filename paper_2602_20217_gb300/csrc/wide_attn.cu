// Causal GQA attention for many query rows of one sequence (prompt
// processing, bf16 models) on the tensor cores.
//
// The decode kernel (attn.cu) reads the whole cache once per 16 rows; here a
// CTA keeps 256 query rows of one head (two tiles of 128) and walks the keys
// 128 at a time, so K and V tiles are read from L2 once per 256 rows.  Per key
// tile and query tile:
//   S = Q K^T          tcgen05.mma, both operands in shared memory, S in TMEM
//   softmax            one thread per query row: running maximum, P = 2^(S - m)
//                      in bf16 back into the TMEM columns of S
//   O += P V           tcgen05.mma with P as the TMEM operand, V as it lies in
//                      the cache (keys x head_dim: an MN-major operand)
// The two query tiles alternate: while one is in its softmax, the tensor core
// works on the other (Shah et al., FlashAttention-3, 2024).  O is rescaled only
// when a row's maximum grew by more than 2^8 (the conditional rescaling known
// from FlashAttention-4): the factor 2^(m - m_ref) of the rest stays exact in
// fp32 and bf16 alike (a power of two apart, the relative precision is the same).
// STATES: the rows are several states of r rows (the hidden-state DP's); all
// see the cache's keys below p0, and each row its own state's rows up to
// itself, so the key tiles are the cache's and then those of the block's own
// K/V rows under a band mask.
// A masked key has P = 0, but 0 times an infinity or a NaN in its V row would
// still be NaN, for rows that do not see that key: in the tiles that some row
// does not see whole (the last two or three of a CTA), a warp of its own clears
// V rows that are not finite before they are used and notes their keys, and the
// rows that do see such a key get NaN.  It works under the softmax of the tile's
// scores: the DP over 16 sublayers (eight launches of 276 rows) takes 2713 us with
// it, 2731 with the check in the MMA warp, 2700 without; prompts of 4096 and 9001
// tokens differ by less than their runs.
// Queries come prepared (QK-norm, RoPE, log2(e) / sqrt(hd)), the keys and
// values of these rows are already in the cache.
//
// Bound by the softmax warps (TMEM reads, maxima, exponentials, conversion:
// the tensor pipe waits for P), not by the MMAs or memory: 2048
// rows of 32 heads at p0 = 0 take 44 us (770 TFLOP/s, tensor pipe 41 % active,
// 25 MB from HBM), a 9001-token prompt of 64 heads runs at about 1.2 PFLOP/s.
// The decode kernel read the cache once per 16 rows for the same work.
//
// Warps: 0-3 and 4-7 the softmax of query tile 0 and 1, 8 the MMAs, 9 the
// loads, 10 the check of the masked tiles.  TMEM: S0, S1 (128 columns each), O0,
// O1 (hd columns each).  Longest query blocks first.  Every wait is bounded.
#include "common.cuh"
#include "internal.h"
#include "umma.cuh"

#include <algorithm>

namespace ks {

namespace {

constexpr int kQ = 128;                      // rows of a query tile, keys of a key tile
constexpr int kChunk = kQ * 128;             // bytes of 128 rows x 64 columns
constexpr int kRing = 4;                     // K and V tiles in flight
constexpr int kThreads = 352;
constexpr float kRescale = 8.f;              // log2 of the growth of a maximum that O is rescaled for
constexpr int kMaskedTiles = 16;             // tiles with masked keys: at most 3, states up to kMaxStateRows: 14
constexpr int kMaxStateRows = 1280;
template <int HD>
constexpr size_t wide_attn_smem() { return 1024 + (size_t)(2 + kRing) * (HD / 64) * kChunk; }

KS_DEV float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One warp: the rows (keys) of a V tile that hold an infinity or a NaN are cleared
// and recorded in bad[4] (a bit per key); false if there are none.
template <int HD>
KS_DEV bool clear_bad_keys(unsigned char* tile, uint32_t* bad) {
    constexpr int CH = HD / 64;
    const int lane = threadIdx.x & 31;
    // lane l: 16 bytes of row 4 it + l / 8 in every chunk (the swizzle stays within a row)
    auto at = [&](int it, int c) { return reinterpret_cast<uint4*>(tile + c * kChunk + it * 512 + lane * 16); };
    // 0 * x is NaN exactly where x is not finite
    auto probe = [](uint4 v, __nv_bfloat162 (&s)[4]) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            s[e] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]), __float2bfloat162_rn(0.f), s[e]);
    };
    auto found = [](const __nv_bfloat162 (&s)[4]) {
        uint32_t any = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) any |= *reinterpret_cast<const uint32_t*>(&s[e]);
        return (any & 0x7fff7fffu) != 0;
    };
    __nv_bfloat162 s[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] = __float2bfloat162_rn(0.f);
#pragma unroll 8
    for (int it = 0; it < kQ / 4; ++it)
#pragma unroll
        for (int c = 0; c < CH; ++c) probe(*at(it, c), s);
    if (!__any_sync(0xffffffffu, found(s))) return false;
#pragma unroll 1
    for (int it = 0; it < kQ / 4; ++it) {
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = __float2bfloat162_rn(0.f);
#pragma unroll
        for (int c = 0; c < CH; ++c) probe(*at(it, c), s);
        const uint32_t hit = __ballot_sync(0xffffffffu, found(s));
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if ((hit >> (8 * q) & 0xffu) == 0) continue;
            if (lane == 0) bad[it / 8] |= 1u << (4 * (it % 8) + q);
            if (lane / 8 == q)
#pragma unroll
                for (int c = 0; c < CH; ++c) *at(it, c) = make_uint4(0, 0, 0, 0);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read the cleared rows
    __syncwarp();
    return true;
}

template <int HD, bool STATES>
__global__ void __launch_bounds__(kThreads, 1) wide_attn_kernel(const __grid_constant__ WideAttnArgs a) {
    constexpr int CH = HD / 64;              // 64-column chunks of a tile
    constexpr uint32_t TB = CH * kChunk;     // bytes of one 128-row tile
    constexpr uint32_t kIdescS = umma_idesc(128, 128, false);
    constexpr uint32_t kIdescO = umma_idesc(128, HD, true);
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char* qs = smem;
    unsigned char* ring = smem + 2 * TB;
    __shared__ __align__(8) uint64_t q_full, kv_full[kRing], kv_free[kRing], s_full[2], p_full[2], o_full[2], v_ok[2], check;
    __shared__ uint32_t tmem_slot;
    __shared__ int void_job;
    __shared__ uint32_t bad[kMaskedTiles][4];   // keys of the masked tiles whose V row is not finite
    __shared__ int any_bad;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h = (int)blockIdx.x % a.hq, kvh = h / (a.hq / a.hk);
    const int q0 = (a.blocks - 1 - (int)blockIdx.x / a.hq) * (2 * kQ);   // first row of this CTA
    // key tiles of each query tile (a tile without rows has none)
    int nt[2];
    const int n_cache = STATES ? (a.p0 + kQ - 1) / kQ : 1 << 30;                // key tiles from the cache
    const int own0 = STATES ? (q0 - q0 % a.state_rows) / kQ : 0;                // first tile of own rows
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int first = q0 + i * kQ, last = min(a.M, first + kQ) - 1;
        nt[i] = first >= a.M ? 0 : STATES ? n_cache + last / kQ - own0 + 1 : (a.p0 + last) / kQ + 1;
    }
    const int n = max(nt[0], nt[1]);
    // the first key tile that some row does not see whole
    const int m0 = STATES ? a.p0 / kQ : (a.p0 + q0 + 1) / kQ;

    if (tid < kMaskedTiles * 4) (&bad[0][0])[tid] = 0u;
    if (warp == 8) tmem_alloc<1>(&tmem_slot, 512);
    if (tid == 0) {
        void_job = __ldcg(a.err) != 0;
        any_bad = 0;
        mbar_init(&q_full, 1);
        mbar_init(&check, 1);
        for (int i = 0; i < kRing; ++i) {
            mbar_init(&kv_full[i], 1);
            mbar_init(&kv_free[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_full[i], 1);
            mbar_init(&p_full[i], 4);
            mbar_init(&o_full[i], 2);   // the MMAs' commit, and an arrival that orders `bad` before it
            mbar_init(&v_ok[i], 1);     // masked tiles m0 + i, m0 + i + 2, ..
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    umma_fence_before();
    __syncthreads();
    umma_fence_after();
    const uint32_t tmem = tmem_slot;

    if (!void_job) {
        if (warp == 9) {
            // ---------------------------------------------------------- loads
            if (lane == 0) {
                bool ok = true;
                mbar_expect_tx(&q_full, 2 * TB);
                for (int i = 0; i < 2; ++i)
                    for (int c = 0; c < CH; ++c)
                        tma_2d(qs + i * TB + c * kChunk, &a.qmap, h * HD + 64 * c, q0 + i * kQ, &q_full);
                int t = 0;
                for (; t < 2 * n; ++t) {     // K 0, V 0, K 1, V 1, ..
                    const int st = t % kRing;
                    if (t >= kRing && !mbar_wait(&kv_free[st], (uint32_t)((t / kRing - 1) & 1), kWaitLimitNs)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&kv_full[st], TB);
                    if (STATES && (t >> 1) >= n_cache)
                        tma_3d(ring + (size_t)st * TB, (t & 1) ? &a.vxmap : &a.kxmap, 0,
                               kvh * a.own_ld + (own0 + (t >> 1) - n_cache) * kQ, 0, &kv_full[st]);
                    else tma_3d(ring + (size_t)st * TB, &a.kvmap, 0,
                           ((t & 1) ? a.kv_row_v : a.kv_row_k) + kvh * a.max_seq + (t >> 1) * kQ, 0, &kv_full[st]);
                }
                if (!ok) {   // the copies in flight land before the CTA leaves
                    atomicCAS(a.err, 0, 1);
                    mbar_wait(&q_full, 0, kWaitLimitNs);
                    for (int q = max(0, t - kRing); q < t; ++q)
                        mbar_wait(&kv_full[q % kRing], (uint32_t)((q / kRing) & 1), kWaitLimitNs);
                }
            }
        } else if (warp == 8) {
            // ----------------------------------------------------------- MMAs
            if (lane == 0) {
                bool ok = mbar_wait(&q_full, 0, kWaitLimitNs);
                auto wait_tile = [&](int t) {
                    ok = ok && mbar_wait(&kv_full[t % kRing], (uint32_t)((t / kRing) & 1), kWaitLimitNs);
                    umma_fence_after();
                };
                auto scores = [&](int i, int j) {   // S_i = Q_i K_j^T
                    const uint32_t sa = smem_u32(qs + i * TB), sb = smem_u32(ring + (size_t)((2 * j) % kRing) * TB);
#pragma unroll
                    for (int k = 0; k < HD / 16; ++k) {
                        const uint32_t off = (uint32_t)(k / 4) * kChunk + 32 * (k % 4);
                        umma_ss<1>(tmem + 128 * i, umma_desc(sa + off, 16, 1024), umma_desc(sb + off, 16, 1024),
                                   kIdescS, k > 0);
                    }
                    umma_commit(&s_full[i]);
                };
                wait_tile(0);
                if (m0 == 0) mbar_arrive(&check);
                if (ok) {
                    for (int i = 0; i < 2; ++i)
                        if (nt[i] > 0) scores(i, 0);
                    umma_commit(&kv_free[0]);
                }
                for (int j = 0; j < n && ok; ++j) {
                    wait_tile(2 * j + 1);
                    if (j + 1 == m0) mbar_arrive(&check);
                    if (j + 1 < n) wait_tile(2 * j + 2);
                    if (j >= m0) ok = ok && mbar_wait(&v_ok[(j - m0) & 1], (uint32_t)((j - m0) >> 1 & 1), kWaitLimitNs);
                    if (!ok) break;
                    const uint32_t sv = smem_u32(ring + (size_t)((2 * j + 1) % kRing) * TB);
                    for (int i = 0; i < 2; ++i) {
                        if (j >= nt[i]) continue;
                        ok = ok && mbar_wait(&p_full[i], (uint32_t)(j & 1), kWaitLimitNs);
                        if (!ok) break;
                        umma_fence_after();
#pragma unroll
                        for (int k = 0; k < kQ / 16; ++k)   // 16 keys: 8 P columns, 2 KB of V rows
                            umma_ts(tmem + 256 + HD * i, tmem + 128 * i + 8 * k,
                                    umma_desc(sv + 2048 * k, kChunk, 1024), kIdescO, j > 0 || k > 0);
                        if (j + 1 < nt[i]) {
                            scores(i, j + 1);
                        } else {
                            umma_commit(&o_full[i]);
                            mbar_arrive(&o_full[i]);
                        }
                    }
                    if (!ok) break;
                    umma_commit(&kv_free[(2 * j + 1) % kRing]);
                    if (j + 1 < n) umma_commit(&kv_free[(2 * j + 2) % kRing]);
                }
                if (!ok) atomicCAS(a.err, 0, 1);
            }
        } else if (warp == 10) {
            // ------------------------------------------- check of the masked tiles
            // It starts once the V tiles before m0 have landed: a ring slot's parity tells a tile's copy only
            // from the slot's last one.  From tile m0 on the MMAs wait for it.
            bool ok = m0 >= n || __all_sync(0xffffffffu, mbar_wait(&check, 0, kWaitLimitNs));
            for (int j = m0; j < n && ok; ++j) {
                // every lane reads the tile, so each waits for it itself
                const int t = 2 * j + 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&kv_full[t % kRing], (uint32_t)((t / kRing) & 1), kWaitLimitNs));
                if (!ok) break;
                if (clear_bad_keys<HD>(ring + (size_t)(t % kRing) * TB, bad[j - m0]) && lane == 0) any_bad = 1;
                __syncwarp();
                if (lane == 0) mbar_arrive(&v_ok[(j - m0) & 1]);
            }
            if (!ok && lane == 0) atomicCAS(a.err, 0, 1);
        } else {
            // -------------------------------------------------------- softmax
            const int i = warp >> 2, quad = warp & 3;
            const int row = q0 + i * kQ + 32 * quad + lane;
            const int pos = a.p0 + row;
            const uint32_t lanes = tmem + ((uint32_t)(32 * quad) << 16);
            const uint32_t s_at = lanes + 128 * i, o_at = lanes + 256 + HD * i;
            float m = -INFINITY, l = 0.f;
            bool ok = true;
            // this row sees the keys lo .. hi of key tile j
            auto seen = [&](int j, int& lo, int& hi) {
                lo = 0;
                hi = pos - kQ * j;
                if (STATES) {
                    const int base = (own0 + j - n_cache) * kQ;
                    lo = j < n_cache ? 0 : row - row % a.state_rows - base;
                    hi = j < n_cache ? a.p0 - 1 - kQ * j : row - base;
                }
            };
            for (int j = 0; j < nt[i]; ++j) {
                ok = mbar_wait(&s_full[i], (uint32_t)(j & 1), kWaitLimitNs);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                umma_fence_after();
                uint32_t s[4][32];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32(s[c], s_at + 32 * c);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_pin(s[c]);
                // tiles that every row sees whole need no mask
                int lo, hi;
                seen(j, lo, hi);
                const bool masked = STATES ? j >= n_cache || kQ * (j + 1) > a.p0 : kQ * (j + 1) > a.p0 + q0 + i * kQ + 1;
                if (masked) {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int q = 0; q < 32; ++q)
                            if (32 * c + q > hi || (STATES && 32 * c + q < lo)) s[c][q] = 0xff800000u;   // -inf
                }
                float mx[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    mx[c] = __uint_as_float(s[c][0]);
#pragma unroll
                    for (int q = 1; q < 32; ++q) mx[c] = fmaxf(mx[c], __uint_as_float(s[c][q]));
                }
                const float mnew = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                if (j == 0) {
                    m = mnew;
                } else if (__any_sync(0xffffffffu, mnew > m + kRescale)) {
                    // only rows that grew change: a row never depends on its neighbours
                    // (one that has still seen no key has neither sum nor O: its factor must not be 2^(-inf + inf))
                    const float mm = mnew > m + kRescale ? mnew : m;
                    const float alpha = mm == -INFINITY ? 1.f : fast_exp2(m - mm);
                    m = mm;
                    l *= alpha;
#pragma unroll 1
                    for (int c = 0; c < HD; c += 32) {
                        uint32_t o[32];
                        tmem_ld32(o, o_at + c);
                        tmem_wait_ld();
                        tmem_pin(o);
#pragma unroll
                        for (int q = 0; q < 32; ++q) o[q] = __float_as_uint(__uint_as_float(o[q]) * alpha);
                        tmem_st32(o_at + c, o);
                    }
                }
                // no key seen yet (a state's row before its state's tile): P is then 0
                const float ref = m == -INFINITY ? 0.f : m;
                float sum[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sum[c] = 0.f;
#pragma unroll
                    for (int q = 0; q < 32; ++q) {
                        const float p = fast_exp2(__uint_as_float(s[c][q]) - ref);
                        sum[c] += p;
                        s[c][q] = __float_as_uint(p);
                    }
                }
                l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
#pragma unroll
                for (int c = 0; c < 2; ++c) {   // bf16 pairs: P columns 32 c .. 32 c + 31
                    uint32_t pk[32];
#pragma unroll
                    for (int q = 0; q < 32; ++q)
                        pk[q] = pack_bf16(__uint_as_float(s[2 * c + q / 16][2 * (q % 16)]),
                                          __uint_as_float(s[2 * c + q / 16][2 * (q % 16) + 1]));
                    tmem_st32(s_at + 32 * c, pk);
                }
                tmem_wait_st();
                umma_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&p_full[i]);
            }
            if (ok && nt[i] > 0) {
                ok = mbar_wait(&o_full[i], 0, kWaitLimitNs);
                ok = __all_sync(0xffffffffu, ok);
                if (ok) {
                    umma_fence_after();
                    float inv = 1.f / l;
                    for (int j = any_bad ? m0 : nt[i]; j < nt[i]; ++j) {   // a key with a V row that is not finite: NaN
                        int lo, hi;
                        seen(j, lo, hi);
                        for (int w = 0; w < 4; ++w)
                            for (uint32_t b = bad[j - m0][w]; b != 0; b &= b - 1) {
                                const int key = 32 * w + __ffs(b) - 1;
                                if (key >= lo && key <= hi) inv = __int_as_float(0x7fffffff);
                            }
                    }
                    __nv_bfloat16* dst = a.out + (size_t)row * a.hq * HD + h * HD;
#pragma unroll 1
                    for (int c = 0; c < HD; c += 32) {
                        uint32_t o[32];
                        tmem_ld32(o, o_at + c);
                        tmem_wait_ld();
                        tmem_pin(o);
                        if (row < a.M) {
#pragma unroll
                            for (int q = 0; q < 32; q += 8) {
                                uint32_t w[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    w[e] = pack_bf16(__uint_as_float(o[q + 2 * e]) * inv,
                                                     __uint_as_float(o[q + 2 * e + 1]) * inv);
                                *reinterpret_cast<uint4*>(dst + c + q) = make_uint4(w[0], w[1], w[2], w[3]);
                            }
                        }
                        __syncwarp();
                    }
                }
            }
            if (!ok && lane == 0) atomicCAS(a.err, 0, 1);
        }
    }
    umma_fence_before();
    __syncthreads();
    if (warp == 8) tmem_free<1>(tmem, 512);
}

}  // namespace

cudaError_t launch_wide_attention(int hd, const WideAttnArgs& args, cudaStream_t s) {
    if (args.M < 1 || args.p0 < 0 || args.err == nullptr || args.hq % args.hk || args.state_rows > kMaxStateRows)
        return cudaErrorInvalidValue;
    WideAttnArgs a = args;
    a.blocks = (a.M + 2 * kQ - 1) / (2 * kQ);
    auto run = [&](auto kern, size_t smem) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<a.hq * a.blocks, kThreads, smem, s>>>(a);
        return cudaGetLastError();
    };
    const bool st = a.state_rows > 0;
    if (hd == 128)
        return st ? run(wide_attn_kernel<128, true>, wide_attn_smem<128>())
                  : run(wide_attn_kernel<128, false>, wide_attn_smem<128>());
    if (hd == 64)
        return st ? run(wide_attn_kernel<64, true>, wide_attn_smem<64>())
                  : run(wide_attn_kernel<64, false>, wide_attn_smem<64>());
    return cudaErrorInvalidValue;
}

}  // namespace ks
