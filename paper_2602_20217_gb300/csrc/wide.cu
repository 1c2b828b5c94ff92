// Projections over many rows (prompt processing) for bf16 models: the same
// projections as the chain kernel's, as tensor-core GEMMs.
//
// Y[m][n] = sum_k A[m][k] W[n][k], M rows at a time (up to the caller's chunk).
// Streaming the weights once per 16 rows, as the decode path does, left the
// tensor cores idle: a 4096-token prompt read every weight 256 times.  Two
// layers of the Llama-3-8B shape over 4096 tokens: 90.5 -> 2.74 ms for the whole
// prefill; two of the Qwen3-32B shape over 9001: 391 -> 14.3 ms.  What bounds it
// is the tensor pipe: at 2048 rows the gate/up GEMM of the 8B shape takes 264 us
// (1821 TFLOP/s, pipe 84 % active), W_down 154, QKV 76 and W_o 55 (128 tiles of
// W_down and W_o, 192 of QKV are 1.7 and 2.5 rounds of the 76 pairs, so the last
// round and the epilogues show).
//
// One CTA pair (cta_group::2) works on a 256 x 256 tile: each CTA stages its
// 128 rows of A and its half of the tile's 256 weight rows (K-major, 64-column
// stages, 128-byte swizzle) by TMA, so per SM and stage 32 KB feed 256 x 256 x
// 64 multiply-adds: 64 bytes per clock at the full tensor rate, where a
// single CTA's 128 x 256 tile would need 96, more than L2 delivers.  The
// accumulators (128 lanes x 256 columns per CTA) are double buffered in TMEM,
// so a tile's epilogue runs under the next tile's MMAs.  Grid: one pair per
// two SMs, persistent; consecutive tiles share the weight rows (rows fastest),
// so the weights come from HBM once and the activations stay in L2.
//
// Per CTA: warp 0 loads, warp 1 issues the MMAs (the pair's first CTA only),
// warps 2-9 run the epilogue of the kind (32 rows x 128 columns each: with
// half as many warps their loads' latency showed at the end of a launch):
//   WK_QKV     1/rms, QK-RMSNorm, RoPE; prepared queries to q, keys and values
//              to the cache (a thread holds one row, so a head's norm and
//              rotation stay in its registers);
//   WK_RESID   residual add, the next RMSNorm's input x * gain and the sums of
//              squares of the tile's columns (via shared memory, so that the
//              global accesses are whole lines);
//   WK_SWIGLU  silu(gate) * up: the pair's first CTA stages gate rows, the
//              second the up rows of the same features;
//   WK_ARGMAX  the row's best (logit, id) as a 64-bit key, merged by atomicMax
//              (any order gives the same argmax): the LM head of the layer
//              selection's candidate states, whose logits nobody reads.
// The tiles that do not fill a last round of all pairs (all of them, for a few
// hundred rows) are cut along K where K is long (more than 7680 inputs) and the
// tiles are few: their stages are dealt out to the pairs in equal contiguous
// shares.  Every part of a cut tile leaves its sums
// in global memory, and per group of 32 rows the part that arrives last (a
// ticket) adds them in K order, puts the total back into its TMEM columns and
// runs the epilogue.  No pair waits for another.
// Every wait is bounded; a wait that gives up sets the status word and the
// CTA leaves after its copies have landed.
#include "common.cuh"
#include "internal.h"
#include "umma.cuh"

#include <algorithm>
#include <climits>

namespace ks {

namespace {

constexpr int kStages = 5;
constexpr int kTileM = 256, kTileN = 256, kTileK = 64;
constexpr uint32_t kHalf = 128 * kTileK * 2;               // 128 rows of one operand: 16 KB
constexpr uint32_t kStageBytes = 2 * kHalf;                // A half, then W half
constexpr uint32_t kPairBytes = 2 * kStageBytes;           // both CTAs' bytes of a stage
constexpr int kEpiWarps = 8;                               // two per 32 rows: columns 0-127 and 128-255
constexpr int kWideThreads = 64 + 32 * kEpiWarps;
constexpr int kEpiPitch = 36;                              // floats per row of the staging area
constexpr size_t kEpiBytes = kEpiWarps * 32 * kEpiPitch * sizeof(float);
constexpr size_t kWideSmem = 1024 + (size_t)kStages * kStageBytes + kEpiBytes;
constexpr int kMinShare = 8;                               // stages of a cut tile a pair takes at least
constexpr int kMergeStages = 112;                          // what merging a cut tile costs, in stages (below)
constexpr uint32_t kIdesc = umma_idesc(256, 256, false);
constexpr uint32_t kSbo = 1024;                            // 8 rows of 128 bytes

// 1 / rms of row m from the per-tile sums of squares, in tile order.
KS_DEV float row_scale(const WideArgs& a, int m) {
    float s = 0.f;
#pragma unroll 8
    for (int q = 0; q < a.ss_n; ++q) s += a.ss_in[(size_t)q * a.ss_ld + m];
    return rsqrtf(s / (float)a.d + a.eps);
}

KS_DEV unsigned long long argmax_key(float v, int i) {
    const uint32_t b = __float_as_uint(v);
    const uint32_t ord = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return ((unsigned long long)ord << 32) | (0xFFFFFFFFu - (uint32_t)i);
}

KS_DEV void load_chunk(uint32_t (&r)[32], uint32_t addr) {
    tmem_ld32(r, addr);
    tmem_wait_ld();
    tmem_pin(r);
}

// A pair's work: the whole tiles pair, pair + pairs, .. below a.full, then its
// share of the cut tiles' stages.  The parts of a cut tile belong to the
// consecutive pairs first .. last.
struct Work {
    int tile, k0, k1, first, last;
};
struct WorkList {
    int next_full, pos, end;
    KS_DEV WorkList(const WideArgs& a, int pair, int kblocks)
        : next_full(pair), pos(pair * a.share), end(min(a.tail * kblocks, (pair + 1) * a.share)) {}
    KS_DEV bool next(const WideArgs& a, int pair, int pairs, int kblocks, Work& w) {
        if (next_full < a.full) {
            w = Work{next_full, 0, kblocks, pair, pair};
            next_full += pairs;
            return true;
        }
        if (pos >= end) return false;
        const int t = pos / kblocks, k0 = pos - t * kblocks, k1 = min(kblocks, k0 + end - pos);
        w = Work{a.full + t, k0, k1, t * kblocks / a.share, ((t + 1) * kblocks - 1) / a.share};
        pos += k1 - k0;
        return true;
    }
};

// Cut tile: this warp's 32 rows x 128 columns go to the slab of (pair, tile);
// true for the part that arrives last, whose TMEM columns then hold the sum
// of all parts in K order.  Along the parts pair + tile grows by one, so it
// numbers the slabs.  Slab: [column / 4][row] float4, so that a warp's
// accesses are whole lines.
template <int KIND>
KS_DEV bool merge_parts(const WideArgs& a, uint32_t acc, int half, const Work& w, int pair, int group) {
    // the columns this warp's epilogue reads (SwiGLU: 64 gate features and their up features)
    auto column = [&](int c) { return KIND == WK_SWIGLU ? 64 * half + (c & 32) + 2 * (c & 64) : 128 * half + c; };
    const int lane = threadIdx.x & 31;
    constexpr size_t slab = 32 * 128 / 4, step = 2 * kEpiWarps * slab;   // float4s of a slab, of a (pair, tile)
    const int t = w.tile - a.full;
    float4* base = reinterpret_cast<float4*>(a.part) + (size_t)t * step + group * slab + lane;
    float4* mine = base + (size_t)pair * step;
#pragma unroll 1
    for (int c = 0; c < 128; c += 32) {
        uint32_t r[32];
        load_chunk(r, acc + column(c));
#pragma unroll
        for (int i = 0; i < 32; i += 4)
            __stcg(&mine[(c + i) / 4 * 32], make_float4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]),
                                                        __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])));
    }
    __threadfence();
    __syncwarp();
    int last = 0;
    if (lane == 0) {
        int* tk = a.ticket + t * 2 * kEpiWarps + group;
        last = atomicAdd(tk, 1) == w.last - w.first;
        if (last) *tk = 0;   // every part has arrived: zero for the next launch
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return false;
    __threadfence();
#pragma unroll 1
    for (int c = 0; c < 128; c += 32) {
        float4 t4[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int q = w.first; q <= w.last; ++q) {
            const float4* src = base + (size_t)q * step + c / 4 * 32;
            float4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldcg(&src[i * 32]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                t4[i].x += v[i].x;
                t4[i].y += v[i].y;
                t4[i].z += v[i].z;
                t4[i].w += v[i].w;
            }
        }
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            r[4 * i] = __float_as_uint(t4[i].x);
            r[4 * i + 1] = __float_as_uint(t4[i].y);
            r[4 * i + 2] = __float_as_uint(t4[i].z);
            r[4 * i + 3] = __float_as_uint(t4[i].w);
        }
        tmem_st32(acc + column(c), r);
    }
    tmem_wait_st();
    return true;
}

// The heads in this warp's 128 columns (n: the first one's feature), one row
// per thread: 1/rms, QK-RMSNorm, RoPE, bf16.  The rotation's (cos, sin) rows
// pass through shared memory 16 pairs at a time, so that they are read as
// whole lines.
template <int HD>
KS_DEV void qkv_heads(const WideArgs& a, uint32_t acc, int m0, int n, float scale, float* stg) {
    constexpr int NH = 128 / HD;
    const int lane = threadIdx.x & 31, m = m0 + lane, head0 = n / HD, heads = a.N / HD;
    const bool live = m < a.M;
    auto position = [&](int row) { return a.p0 + (a.state_rows > 0 ? row % a.state_rows : row); };
    const int pos = position(live ? m : 0);
    const int kv_row = a.state_rows > 0 ? m : pos;
    const __nv_bfloat16* gain[NH];
    float f[NH];                  // 1/rms of the row, times the head's own
    __nv_bfloat16* dst[NH];
    bool rotated = false;         // some head here is a query or key head
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const int head = head0 + h;
        gain[h] = head < a.hq ? a.q_norm : head < a.hq + a.hk ? a.k_norm : nullptr;
        dst[h] = head < a.hq ? a.q + ((size_t)m * a.hq + head) * HD
                 : head < a.hq + a.hk ? a.kcache + ((size_t)(head - a.hq) * a.max_seq + kv_row) * HD
                                      : a.vcache + ((size_t)(head - a.hq - a.hk) * a.max_seq + kv_row) * HD;
        rotated |= head < a.hq + a.hk;
        f[h] = 1.f;
        if (gain[h] != nullptr) {
            float ss = 0.f;
#pragma unroll 1
            for (int c = 0; c < HD; c += 32) {
                uint32_t r[32];
                load_chunk(r, acc + h * HD + c);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float v = __uint_as_float(r[i]) * scale;
                    ss = fmaf(v, v, ss);
                }
            }
            f[h] = rsqrtf(ss / (float)HD + a.eps);
        }
    }
    const float qs = 1.4426950408889634f * rsqrtf((float)HD);
    const int sub = lane >> 3, c4 = (lane & 7) * 4;
#pragma unroll 1
    for (int j = 0; j < HD / 2; j += 16) {   // pairs j .. j + 15: features j + i and j + i + HD / 2
        if (rotated) {
            float4 t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                t[i] = *reinterpret_cast<const float4*>(
                    a.rope + (size_t)position(min(m0 + 4 * i + sub, a.M - 1)) * HD + 2 * j + c4);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(stg + (4 * i + sub) * kEpiPitch + c4) = t[i];
            __syncwarp();
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            uint32_t ra[16], rb[16];
            tmem_ld16(ra, acc + h * HD + j);
            tmem_ld16(rb, acc + h * HD + HD / 2 + j);
            tmem_wait_ld();
            tmem_pin(ra);
            tmem_pin(rb);
            const int head = head0 + h;
            if (live && head < heads) {
                uint32_t wa[8], wb[8];
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    float x0 = __uint_as_float(ra[i]) * scale, x1 = __uint_as_float(ra[i + 1]) * scale;
                    float y0 = __uint_as_float(rb[i]) * scale, y1 = __uint_as_float(rb[i + 1]) * scale;
                    if (gain[h] != nullptr) {
                        const uint32_t gx = *reinterpret_cast<const uint32_t*>(gain[h] + j + i);
                        const uint32_t gy = *reinterpret_cast<const uint32_t*>(gain[h] + HD / 2 + j + i);
                        x0 = (x0 * f[h]) * bf16_lo(gx);
                        x1 = (x1 * f[h]) * bf16_hi(gx);
                        y0 = (y0 * f[h]) * bf16_lo(gy);
                        y1 = (y1 * f[h]) * bf16_hi(gy);
                    }
                    if (head < a.hq + a.hk) {
                        const float4 cs = *reinterpret_cast<const float4*>(stg + lane * kEpiPitch + 2 * i);
                        const float u0 = x0, u1 = x1;
                        x0 = u0 * cs.x - y0 * cs.y;
                        y0 = y0 * cs.x + u0 * cs.y;
                        x1 = u1 * cs.z - y1 * cs.w;
                        y1 = y1 * cs.z + u1 * cs.w;
                    }
                    if (head < a.hq) {
                        x0 *= qs;
                        x1 *= qs;
                        y0 *= qs;
                        y1 *= qs;
                    }
                    wa[i / 2] = pack_bf16(x0, x1);
                    wb[i / 2] = pack_bf16(y0, y1);
                }
                uint4* pa = reinterpret_cast<uint4*>(dst[h] + j);
                uint4* pb = reinterpret_cast<uint4*>(dst[h] + HD / 2 + j);
                pa[0] = make_uint4(wa[0], wa[1], wa[2], wa[3]);
                pa[1] = make_uint4(wa[4], wa[5], wa[6], wa[7]);
                pb[0] = make_uint4(wb[0], wb[1], wb[2], wb[3]);
                pb[1] = make_uint4(wb[4], wb[5], wb[6], wb[7]);
            }
            __syncwarp();   // every lane takes part in the next TMEM loads
        }
    }
}

// Epilogue of one tile by one warp: rows m0 .. m0 + 31 (this thread: m0 +
// lane), half `half` of its columns, TMEM address `acc` (this warp's lanes,
// first column of the buffer).
template <int KIND, int HD>
KS_DEV void wide_epilogue(const WideArgs& a, uint32_t acc, int m0, int tn, int half, float scale, float* stg) {
    const int lane = threadIdx.x & 31;
    const int m = m0 + lane;
    const bool live = m < a.M;
    if constexpr (KIND == WK_QKV) {
        const int n = tn * kTileN + 128 * half;
        if (n < a.N) qkv_heads<HD>(a, acc + 128 * half, m0, n, scale, stg);
    } else if constexpr (KIND == WK_SWIGLU) {
        const int n0 = tn * 128 + 64 * half;   // gate features; the up features lie 128 columns on
        acc += 64 * half;
#pragma unroll 1
        for (int c = 0; c < 64; c += 32) {
            uint32_t g[32], u[32];
            tmem_ld32(g, acc + c);
            tmem_ld32(u, acc + 128 + c);
            tmem_wait_ld();
            tmem_pin(g);
            tmem_pin(u);
            __nv_bfloat16* dst = a.act + (size_t)m * a.N + n0 + c;
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float g0 = __uint_as_float(g[i + 2 * j]) * scale, g1 = __uint_as_float(g[i + 2 * j + 1]) * scale;
                    const float u0 = __uint_as_float(u[i + 2 * j]) * scale, u1 = __uint_as_float(u[i + 2 * j + 1]) * scale;
                    w[j] = pack_bf16(silu(g0) * u0, silu(g1) * u1);
                }
                if (live && n0 + c + i < a.N) *reinterpret_cast<uint4*>(dst + i) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            __syncwarp();
        }
    } else if constexpr (KIND == WK_ARGMAX) {
        float bv = -INFINITY;
        int bi = INT_MAX;
#pragma unroll 1
        for (int c = 0; c < 128; c += 32) {
            uint32_t r[32];
            load_chunk(r, acc + 128 * half + c);
            const int n = tn * kTileN + 128 * half + c;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float v = __uint_as_float(r[i]) * scale;
                if (n + i < a.N && better(v, n + i, bv, bi)) {
                    bv = v;
                    bi = n + i;
                }
            }
        }
        if (live && bi != INT_MAX) atomicMax(&a.best[m], argmax_key(bv, bi));
    } else {
        // 32 columns at a time through shared memory: written one row per
        // thread, read back as whole row pieces of 32 columns
        float ssq[8];
        float4 xv[2][8];   // this chunk's and the next one's residual
        uint2 gw[2];
#pragma unroll
        for (int i = 0; i < 8; ++i) ssq[i] = 0.f;
        const int sub = lane >> 3, c4 = (lane & 7) * 4, n0 = tn * kTileN + 128 * half;
        // The residual is loaded a chunk ahead, eight rows at a time: loaded
        // where it is added to, each row's round trip waited behind the store
        // of the row before (60 us a tile instead of about 10).
        auto fetch = [&](int c, int slot) {
            const int n = n0 + c + c4;
            if (n < a.N) {   // N is a multiple of 8
                gw[slot] = *reinterpret_cast<const uint2*>(a.gain + n);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (m0 + 4 * i + sub < a.M)
                        xv[slot][i] = *reinterpret_cast<const float4*>(a.x + (size_t)(m0 + 4 * i + sub) * a.N + n);
            }
        };
        fetch(0, 0);
#pragma unroll 2
        for (int c = 0; c < 128; c += 32) {
            const int slot = (c / 32) & 1;
            uint32_t r[32];
            if (c + 32 < 128) fetch(c + 32, slot ^ 1);
            __syncwarp();
            load_chunk(r, acc + 128 * half + c);
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<uint4*>(stg + lane * kEpiPitch + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
            __syncwarp();
            const int n = n0 + c + c4;
            if (n < a.N) {
                const float g0 = bf16_lo(gw[slot].x), g1 = bf16_hi(gw[slot].x);
                const float g2 = bf16_lo(gw[slot].y), g3 = bf16_hi(gw[slot].y);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int mr = m0 + 4 * i + sub;
                    if (mr >= a.M) continue;
                    const float4 v = *reinterpret_cast<const float4*>(stg + (4 * i + sub) * kEpiPitch + c4);
                    float4 x = xv[slot][i];
                    x.x += v.x;
                    x.y += v.y;
                    x.z += v.z;
                    x.w += v.w;
                    *reinterpret_cast<float4*>(a.x + (size_t)mr * a.N + n) = x;
                    if (a.capture != nullptr && mr >= a.capture_from)
                        *reinterpret_cast<float4*>(a.capture + (size_t)(mr - a.capture_from) * a.N + n) = x;
                    *reinterpret_cast<uint2*>(a.xg + (size_t)mr * a.N + n) =
                        make_uint2(pack_bf16(x.x * g0, x.y * g1), pack_bf16(x.z * g2, x.w * g3));
                    ssq[i] = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, ssq[i]))));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) ssq[i] += __shfl_xor_sync(0xffffffffu, ssq[i], o);
            const int mr = m0 + 4 * i + sub;
            if ((lane & 7) == 0 && mr < a.M && a.ss_out != nullptr)
                a.ss_out[(size_t)(2 * tn + half) * a.ss_ld + mr] = ssq[i];
        }
    }
}

template <int KIND, int HD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kWideThreads, 1)
    wide_kernel(const __grid_constant__ WideArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    float* staging = reinterpret_cast<float*>(smem + (size_t)kStages * kStageBytes);
    __shared__ __align__(8) uint64_t full[kStages];     // the pair's first CTA: both CTAs' copies have landed
    __shared__ __align__(8) uint64_t empty[kStages];    // each CTA: the pair's MMAs have read the stage
    __shared__ __align__(8) uint64_t acc_full[2];       // each CTA: the buffer's accumulators are complete
    __shared__ __align__(8) uint64_t acc_free[2];       // the pair's first CTA: every epilogue warp has read it
    __shared__ uint32_t tmem_slot;
    __shared__ uint32_t skip;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
    const int kblocks = (a.K + kTileK - 1) / kTileK;
    WorkList list(a, pair, kblocks);
    Work w;

    if (warp == 1) tmem_alloc<2>(&tmem_slot, 512);
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_free[i], 2 * kEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // a job whose status word holds an error is void: the pair's first
        // CTA decides for both (the word can change during the launch)
        skip = __ldcg(a.err) != 0;
    }
    __syncthreads();
    umma_fence_before();
    cluster_sync();
    umma_fence_after();
    const uint32_t tmem = tmem_slot;
    if (cluster_load(cluster_addr(&skip, 0)) == 0) {
        if (warp == 0) {
            // ------------------------------------------------------ loader
            if (lane == 0) {
                bool ok = true;
                int t = 0;
                while (ok && list.next(a, pair, pairs, kblocks, w)) {
                    const int tm = w.tile % a.tiles_m, tn = w.tile / a.tiles_m;
                    const int ra = tm * kTileM + (int)rank * 128;
                    const int rw = KIND == WK_SWIGLU ? tn * 128 + (int)rank * a.N : tn * kTileN + (int)rank * 128;
                    for (int kb = w.k0; kb < w.k1; ++kb, ++t) {
                        const int st = t % kStages;
                        if (t >= kStages && !mbar_wait(&empty[st], (uint32_t)((t / kStages - 1) & 1), kWaitLimitNs)) {
                            ok = false;
                            break;
                        }
                        if (rank == 0) mbar_expect_tx(&full[st], kPairBytes);
                        const uint32_t bar = cluster_addr(&full[st], 0);
                        unsigned char* dst = smem + (size_t)st * kStageBytes;
                        tma_2d_pair(dst, &a.amap, kb * kTileK, ra, bar);
                        tma_2d_pair(dst + kHalf, &a.wmap, kb * kTileK, rw, bar);
                    }
                }
                if (!ok) {
                    atomicCAS(a.err, 0, 1);
                    // copies still in flight land before the pair leaves
                    if (rank == 0)
                        for (int q = max(0, t - kStages); q < t; ++q)
                            mbar_wait(&full[q % kStages], (uint32_t)((q / kStages) & 1), kWaitLimitNs);
                }
            }
        } else if (warp == 1) {
            // --------------------------------------------------------- MMA
            if (rank == 0 && lane == 0) {
                bool ok = true;
                int t = 0, n = 0;
                for (; ok && list.next(a, pair, pairs, kblocks, w); ++n) {
                    const int b = n & 1;
                    if (n >= 2 && !mbar_wait(&acc_free[b], (uint32_t)((n / 2 - 1) & 1), kWaitLimitNs)) {
                        ok = false;
                        break;
                    }
                    umma_fence_after();
                    const uint32_t acc = tmem + (uint32_t)(b * kTileN);
                    for (int kb = w.k0; kb < w.k1; ++kb, ++t) {
                        const int st = t % kStages;
                        if (!mbar_wait(&full[st], (uint32_t)((t / kStages) & 1), kWaitLimitNs)) {
                            ok = false;
                            break;
                        }
                        umma_fence_after();
                        const uint32_t sa = smem_u32(smem + (size_t)st * kStageBytes);
#pragma unroll
                        for (int k = 0; k < kTileK / 16; ++k)
                            umma_ss<2>(acc, umma_desc(sa + 32 * k, 16, kSbo), umma_desc(sa + kHalf + 32 * k, 16, kSbo),
                                       kIdesc, kb > w.k0 || k > 0);
                        umma_commit_pair(&empty[st]);
                    }
                    if (ok) umma_commit_pair(&acc_full[b]);
                }
                if (!ok) atomicCAS(a.err, 0, 1);
            }
        } else {
            // ---------------------------------------------------- epilogue
            const int quad = warp & 3, half = (warp - 2) >> 2;   // the TMEM lanes this warp may read, its columns
            float* stg = staging + (warp - 2) * 32 * kEpiPitch;
            bool ok = true;
            int n = 0;
            for (; list.next(a, pair, pairs, kblocks, w); ++n) {
                const int b = n & 1;
                const int tm = w.tile % a.tiles_m, tn = w.tile / a.tiles_m;
                const int m0 = tm * kTileM + (int)rank * 128 + 32 * quad;
                // the row's 1/rms, while the tile's MMAs run
                const float scale = KIND == WK_RESID ? 0.f : row_scale(a, min(m0 + lane, a.M - 1));
                ok = mbar_wait(&acc_full[b], (uint32_t)((n / 2) & 1), kWaitLimitNs);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                umma_fence_after();
                const uint32_t acc = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(b * kTileN);
                if (w.first == w.last || merge_parts<KIND>(a, acc, half, w, pair, (int)rank * kEpiWarps + 4 * half + quad))
                    wide_epilogue<KIND, HD>(a, acc, m0, tn, half, scale, stg);
                umma_fence_before();
                __syncwarp();
                if (lane == 0) cluster_arrive(cluster_addr(&acc_free[b], 0));
            }
            if (!ok && lane == 0) atomicCAS(a.err, 0, 1);
        }
    }
    __syncthreads();
    umma_fence_before();
    cluster_sync();   // neither CTA leaves while the other may still signal it
    if (warp == 1) tmem_free<2>(tmem, 512);
}

// Rows of the embedding table as the residual, the first projection's input
// and the rows' sums of squares (slot 0; the other tiles' slots are zero).
__global__ void __launch_bounds__(256) wide_embed_kernel(const __nv_bfloat16* embed, const int32_t* tok, int d,
                                                         int vocab, float* x, __nv_bfloat16* xg,
                                                         const __nv_bfloat16* gain, float* ss, int ss_n, int ss_ld,
                                                         float* capture, int capture_from) {
    __shared__ float red[9];
    const int m = blockIdx.x;
    int t = tok[m];
    if (t < 0 || t >= vocab) t = 0;
    const __nv_bfloat16* e = embed + (size_t)t * d;
    float s = 0.f;
    for (int k = (int)threadIdx.x * 8; k < d; k += 256 * 8) {   // d is a multiple of 8
        const uint4 w = *reinterpret_cast<const uint4*>(e + k), g = *reinterpret_cast<const uint4*>(gain + k);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w}, gs[4] = {g.x, g.y, g.z, g.w};
        float v[8];
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = bf16_lo(ws[i]);
            v[2 * i + 1] = bf16_hi(ws[i]);
            o[i] = pack_bf16(v[2 * i] * bf16_lo(gs[i]), v[2 * i + 1] * bf16_hi(gs[i]));
            s = fmaf(v[2 * i], v[2 * i], s);
            s = fmaf(v[2 * i + 1], v[2 * i + 1], s);
        }
        float4* xp = reinterpret_cast<float4*>(x + (size_t)m * d + k);
        xp[0] = make_float4(v[0], v[1], v[2], v[3]);
        xp[1] = make_float4(v[4], v[5], v[6], v[7]);
        if (capture != nullptr && m >= capture_from) {
            float4* cp = reinterpret_cast<float4*>(capture + (size_t)(m - capture_from) * d + k);
            cp[0] = make_float4(v[0], v[1], v[2], v[3]);
            cp[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
        *reinterpret_cast<uint4*>(xg + (size_t)m * d + k) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    s = block_sum<8>(s, red);
    if ((int)threadIdx.x < ss_n) ss[(size_t)threadIdx.x * ss_ld + m] = threadIdx.x == 0 ? s : 0.f;
}

__global__ void __launch_bounds__(256) wide_tokens_kernel(const unsigned long long* best, int M, int32_t* tokens) {
    const int m = blockIdx.x * 256 + threadIdx.x;
    if (m >= M) return;
    const unsigned long long key = best[m];
    tokens[m] = key == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
}

}  // namespace

cudaError_t launch_wide_tokens(const unsigned long long* best, int M, int32_t* tokens, cudaStream_t s) {
    wide_tokens_kernel<<<(M + 255) / 256, 256, 0, s>>>(best, M, tokens);
    return cudaGetLastError();
}

// launch_wide's rule below for the smallest share it deals out
bool wide_cuts(int K) { return kMinShare + kMergeStages < (K + kTileK - 1) / kTileK; }

int wide_tiles_n(int kind, int N) { return kind == WK_SWIGLU ? (N + 127) / 128 : (N + kTileN - 1) / kTileN; }

cudaError_t launch_wide_embed(const __nv_bfloat16* embed, const int32_t* tok, int M, int d, int vocab, float* x,
                              __nv_bfloat16* xg, const __nv_bfloat16* gain, float* ss, int ss_n, int ss_ld,
                              float* capture, int capture_from, cudaStream_t s) {
    if (M < 1 || ss_n > 256) return cudaErrorInvalidValue;
    wide_embed_kernel<<<M, 256, 0, s>>>(embed, tok, d, vocab, x, xg, gain, ss, ss_n, ss_ld, capture,
                                      capture_from);
    return cudaGetLastError();
}

cudaError_t launch_wide(int kind, int hd, const WideArgs& args, cudaStream_t s) {
    if (args.M < 1 || args.N < 1 || args.K < 8 || args.err == nullptr) return cudaErrorInvalidValue;
    WideArgs a = args;
    a.tiles_m = (a.M + kTileM - 1) / kTileM;
    a.tiles_n = wide_tiles_n(kind, a.N);
    // The tiles past the last full round of all pairs are cut along K where
    // that is shorter: their stages dealt out evenly, plus the partial sums'
    // round trip (kMergeStages), against a round of whole tiles.  In the
    // configured shapes that is W_down at most sizes (Llama-3-8B: up to 512 and
    // 1280 to 1792 rows, not 768, 1024 or 2048) and W_o of the Qwen3-32B shape at
    // 1024 and 2048.  Whole prefills of four Llama-3-8B layers with kMergeStages at 16, 48, 112 and
    // never cutting: 882, 850, 827, 943 us at 256 tokens (W_down: 16 tiles of
    // 224 stages), 2700, 2635, 2547, 2529 us at 2048 (128 tiles).
    const int tiles = a.tiles_m * a.tiles_n, kblocks = (a.K + kTileK - 1) / kTileK;
    const int pairs_max = std::min(sm_count() / 2, kWidePairs);
    const int rest = tiles % pairs_max, share = std::max((rest * kblocks + pairs_max - 1) / pairs_max, kMinShare);
    a.full = tiles;
    a.tail = 0;
    a.share = 1;
    int pairs = std::min(pairs_max, tiles);
    if (rest > 0 && share + kMergeStages < kblocks) {
        a.full = tiles - rest;
        a.tail = rest;
        a.share = share;
        if (a.full == 0) pairs = (rest * kblocks + share - 1) / share;
        else pairs = pairs_max;
    }
    auto run = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem);
        if (e != cudaSuccess) return e;
        kern<<<2 * pairs, kWideThreads, kWideSmem, s>>>(a);
        return cudaGetLastError();
    };
    switch (kind) {
        case WK_QKV:
            if (hd == 128) return run(wide_kernel<WK_QKV, 128>);
            if (hd == 64) return run(wide_kernel<WK_QKV, 64>);
            return cudaErrorInvalidValue;
        case WK_RESID: return run(wide_kernel<WK_RESID, 0>);
        case WK_SWIGLU: return run(wide_kernel<WK_SWIGLU, 0>);
        case WK_ARGMAX: return run(wide_kernel<WK_ARGMAX, 0>);
    }
    return cudaErrorInvalidValue;
}

}  // namespace ks
