// Chained projections for bf16 models: one persistent launch runs a sequence
// of decoder projections ("phases": QKV, O + residual, gate/up + SwiGLU,
// down + residual, LM head + argmax) of the Sec. 2 sublayers that a pass
// executes back to back, i.e. everything between two attention cores.
//
// Why: at R <= 16 rows each projection is a pure stream over its weights.
// Launched one by one, every projection pays a ramp (first tiles in flight),
// a tail (the last items on a few SMs) and a launch gap, which cost small
// matrices (W_o: 33.6 MB, 5 us at HBM speed) two thirds of their time.  Here
// the weight stream never stops at a phase boundary: weights do not depend on
// the activations, so each CTA's producer keeps loading the next phase's
// weight tiles while the previous phase is still finishing anywhere on the
// GPU.  Only the small activation tiles wait for the previous phase.
//
// Per CTA (two per SM for up to 8 rows, else one; 7 warps):
//  * warp 4 (weights): claims work units phase by phase from per-phase
//    atomic queues (16 output features over the full K) and issues their
//    2-D TMA weight boxes into a ring of shared-memory stages;
//  * warp 5 (activations): follows the same stage sequence; before a stage
//    it waits until the block of the previous phase's output that the stage
//    reads is complete (its lanes look at all blocks at once: one block and one
//    round trip per stage held a phase's first item up by 1.4 us a stage), then
//    issues the stage's activation boxes;
//  * warps 0-3 (consumers): mma.sync m16n8k16 with weights as A and the R
//    activation rows as B (columns independent: batch invariant), each warp
//    a quarter of every stage's columns and at its own pace,
//    then hand each item's per-warp sums to
//  * warp 6 (epilogue): adds them in warp order (fixed), computes the rows'
//    1/rms at its first item of a normed phase (normalised inputs), runs the
//    fused epilogue, and publishes the row group to the next phase.  LM head:
//    each CTA keeps its best (logit, id) per row and, after its last item,
//    merges it into a 64-bit key with atomicMax (value first, then the lower
//    id: any merge order gives the same argmax) and counts its items; the CTA
//    whose count completes the phase reads the keys.
//    Partials are double buffered, so consumers never wait for an epilogue.
// A stage is full when both loaders have arrived and all bytes have landed.
// A CTA's first unit of each phase is fixed by its index; further units are
// claimed from per-phase atomic queues.  Deadlock-free: every CTA of the grid
// becomes resident once the kernels before it finish (the grid is sized to
// fit), a CTA works its units in phase order, and the lowest unfinished phase
// always has all its inputs.  Every wait is bounded (2 s): on expiry the
// status word is set and the CTA leaves.
#include "common.cuh"
#include "internal.h"
#include "tma.cuh"

#include <algorithm>
#include <climits>

namespace ks {

namespace {

constexpr int kThreads = 224;
constexpr int kWarpW = 4;      // weight loader
constexpr int kWarpA = 5;      // activation loader
constexpr int kWarpE = 6;      // epilogue
constexpr int kMaxStages = 8;
constexpr int kBoxElems = 256 * 16;                  // 256 columns x 16 rows of a stage
constexpr int kChunkBytes = 64 * 16 * 2;             // weight chunk: 64 columns x 16 rows, 128-byte swizzled
constexpr uint32_t kWBytes = 4u * kBoxElems * 2u;    // weight bytes per stage (4 boxes)
// Ring per CTA: up to 8 rows run two CTAs per SM (two independent pipelines
// per SM measured 21 % faster than one with twice the ring); more rows need
// the room of one CTA per SM.
constexpr size_t kRingBudget1 = 196u * 1024u;        // one CTA per SM
constexpr size_t kRingBudget2 = 104u * 1024u;        // two CTAs per SM
constexpr int kMaxRows = 16;

// Status word codes (the first one recorded stays): a bounded wait ran out,
// or a self-check found a stage or item record out of range (the access it
// guards is skipped).
constexpr int kErrWait = 1;
constexpr int kErrCheckW = 2, kErrCheckA = 3, kErrCheckC = 4, kErrCheckE = 5;
KS_DEV void set_err(int* e, int code) { atomicCAS(e, 0, code); }

struct Phase {
    int kind, layer, N, K, n_items, tpi;   // items of 16 output features, stages per item
};

// W_o and W_down have only d / 16 row groups, fewer than the CTAs or little
// more, and an item still takes its whole K: cut into two K-slices whose
// partial sums met in global memory, a layer took 95.2 us (Llama-3-8B shape, 4k
// context) against 89.9, with more slices up to 123: the partial sums, the
// ticket and the other slices' read-back all sit on the one epilogue warp.  Other
// shapes, 16 decode steps of four layers before (slices) and since (without,
// and with the query prep's and the residual's loads ahead), ms: width 512 2.13,
// 2.06; 1024 2.43, 2.36; 2048 3.35, 3.25; 3072 4.31, 3.95; 8B 6.25, 5.84; 32B
// 11.19, 10.97; two of width 8192 8.77, 8.39.
KS_DEV Phase decode(const ChainArgs& a, int k) {
    const int code = a.code[k];
    Phase p;
    if (code >= 4 * a.n_layers) {
        p.kind = CH_LM; p.layer = 0; p.N = a.vocab; p.K = a.d;
    } else {
        p.kind = code & 3;
        p.layer = code >> 2;
        switch (p.kind) {
            case CH_QKV: p.N = a.nqkv; p.K = a.d; break;
            case CH_O: p.N = a.d; p.K = a.hqd; break;
            case CH_GU: p.N = a.F; p.K = a.d; break;
            default: p.N = a.d; p.K = a.F; break;
        }
    }
    p.n_items = (p.N + 15) >> 4;
    const int shift = p.kind == CH_GU ? 9 : 10;      // k columns per stage: 512 or 1024
    p.tpi = (p.K + (1 << shift) - 1) >> shift;
    return p;
}
KS_DEV bool normed_input(int kind) { return kind == CH_QKV || kind == CH_GU || kind == CH_LM; }
KS_DEV int stage_cols(int kind) { return kind == CH_GU ? 512 : 1024; }

// Wavefront between phases: a stage of phase k reads columns kt * cols ..
// of phase k - 1's output, so it waits only for the row groups that produce
// them (block kt of phase k - 1), not for the whole phase.  Each finished row
// group of phase k - 1 adds 1 to its block's counter.
constexpr int kMaxBlocks = 64;
KS_DEV int block_rowgroups(int n_out, int cols, int b) {   // row groups of block b
    const int first = b * (cols / 16);
    const int last = min((n_out + 15) / 16, (b + 1) * (cols / 16));
    return last - first;
}
KS_DEV const CUtensorMap* amap_of(const ChainArgs& a, int kind) {
    return &a.amap[kind == CH_GU ? 1 : kind == CH_O ? 2 : kind == CH_DOWN ? 3 : 0];
}
// K % 64 == 0: the maps are 3-D and a stage's weights or activations one copy
KS_DEV bool maps_3d(const Phase& P) { return (P.K & 63) == 0; }

// Independent accumulator chains per consumer warp: the MMAs of a stage go
// round-robin to kChains accumulators, so consecutive MMAs do not wait on each
// other's results (one dependent chain made the loop latency-bound).  The
// chains are added in chain order at the end of an item: a fixed order that
// depends on neither R nor the CTA.
constexpr int kChains = 2;

// One stage of one consumer warp: its quarter of the stage's columns.
// Weights and activations lie in 64-column chunks (16 and R rows of 128 bytes)
// under the 128-byte swizzle, which goes by shared-memory address: 16-byte unit
// u of the row at byte offset o (from a multiple of 1024) is at unit
// u ^ ((o >> 7) & 7).  ldmatrix reads eight rows of one unit at a time, eight
// different bank groups; 16-byte loads per lane in the MMA's row order met two
// rows in the same banks, and with a barrier of the four warps per stage a
// stage took 1.3 us from shared memory: no catching up after a wait at HBM's
// pace of 1.47 us.  A decode layer (Llama-3-8B shape, 4k context) went from
// 100.5 to 95.2 us, a verify layer of 5 rows from 119 to 108, of 11 from 175 to 133.
template <int NT, bool PAIR>
KS_DEV void mma_stage(uint32_t st, int R, int warp, int lane, float (&acc)[kChains][NT][4],
                      float (&accu)[kChains][NT][4]) {
    constexpr int kWarpCols = PAIR ? 128 : 256;
    // weights: matrix l >> 3 of a 16 x 16 step is rows (l >> 3 & 1) * 8 .., unit l >> 4
    const int wrow = (lane & 7) + ((lane >> 3) & 1) * 8;
    const uint32_t wbase = st + wrow * 128;
    const int wkey = lane & 7, wunit = lane >> 4;
    // activations: matrix l >> 3 of a 32-column step is its unit; rows past R repeat row 0 (their
    // columns of the product are not used)
    const int aunit = lane >> 3;
    int arow[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int r = nt * 8 + (lane & 7);
        arow[nt] = r < R ? r : 0;
    }
    const uint32_t abase = st + kWBytes;
#pragma unroll
    for (int ks = 0; ks < kWarpCols / 32; ++ks) {
        const int j0 = warp * kWarpCols + 32 * ks;               // first column of the step
        const int c = j0 >> 6, u0 = (j0 & 63) >> 3;
        uint32_t w[2][4], u[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t off = wbase + c * kChunkBytes + (((u0 + 2 * h + wunit) ^ wkey) << 4);
            ldsm_x4(w[h], off);
            if (PAIR) ldsm_x4(u[h], off + 8 * kChunkBytes);      // up rows: the second half of the stage
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int q = c * R + arow[nt];                      // 128-byte row of the activations
            uint32_t b[4];
            ldsm_x4(b, abase + q * 128 + (((u0 + aunit) ^ (q & 7)) << 4));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                mma_bf16(acc[h][nt], w[h][0], w[h][1], w[h][2], w[h][3], b[2 * h], b[2 * h + 1]);
                if (PAIR) mma_bf16(accu[h][nt], u[h][0], u[h][1], u[h][2], u[h][3], b[2 * h], b[2 * h + 1]);
            }
        }
    }
}

// Argmax key of (logit v, token i): larger v first, then the lower id; an
// unsigned 64-bit max over keys is the argmax in any order of merging.
KS_DEV unsigned long long argmax_key(float v, int i) {
    const uint32_t b = __float_as_uint(v);
    const uint32_t ord = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return ((unsigned long long)ord << 32) | (0xFFFFFFFFu - (uint32_t)i);
}

// Residual phases: this lane's residual values and the next norm's gains of
// item `it`, all loaded together before the item's sums are added up.  Loaded
// where they are used, each waited behind the store of the one before, and an
// item's epilogue took 3.6 us, at the end of every W_o and W_down.
template <int NT>
struct ResidIn {
    float x[NT][4];
    float gain[2];
    KS_DEV void load(const ChainArgs& a, const Phase& P, int k, int it) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = it * 16 + g + 8 * h;
            gain[h] = n < P.N ? __bfloat162float(a.gain[k][n]) : 0.f;
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int n = it * 16 + g + 8 * (i >> 1), r = nt * 8 + 2 * t4 + (i & 1);
                x[nt][i] = n < P.N && r < a.R ? __ldcg(a.x + (size_t)r * a.d + n) : 0.f;
            }
    }
};

// Item epilogue (after the warp-order sum).  Fragment (nt, i) of lane (g, t) is
// feature it * 16 + g + 8 (i >> 1), row nt * 8 + 2 t + (i & 1).
template <int NT>
KS_DEV void epilogue(const ChainArgs& a, const Phase& P, int it, const ResidIn<NT>& in, float (&acc)[NT][4],
                     float (&accu)[NT][4], const float* scale, float (&run_v)[NT][2], int (&run_i)[NT][2]) {
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t4 = lane & 3;
    float ssq[NT][2], bv[NT][2];
    int bi[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            ssq[nt][c] = 0.f;
            bv[nt][c] = -INFINITY;
            bi[nt][c] = INT_MAX;
        }
    const bool resid = P.kind == CH_O || P.kind == CH_DOWN;
    float* cap = nullptr;
    if (resid && a.capture) cap = a.capture + (size_t)(2 * P.layer + 1 + (P.kind == CH_DOWN)) * a.capture_plane;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int n = it * 16 + g + 8 * (i >> 1);
            const int r = nt * 8 + 2 * t4 + (i & 1);
            if (n >= P.N || r >= a.R) continue;
            const float v = acc[nt][i] * scale[r];
            switch (P.kind) {
                case CH_QKV:
                    a.qkv[(size_t)r * a.nqkv + n] = v;
                    break;
                case CH_GU:
                    a.act[(size_t)r * a.F + n] = __float2bfloat16_rn(silu(v) * (accu[nt][i] * scale[r]));
                    break;
                case CH_LM:
                    a.logits[(size_t)r * a.vocab + n] = v;
                    if (better(v, n, bv[nt][i & 1], bi[nt][i & 1])) {
                        bv[nt][i & 1] = v;
                        bi[nt][i & 1] = n;
                    }
                    break;
                default: {  // residual add; the new residual feeds the next RMSNorm
                    const float nx = in.x[nt][i] + v;
                    a.x[(size_t)r * a.d + n] = nx;
                    if (cap) cap[(size_t)r * a.d + n] = nx;
                    a.xg[(size_t)r * a.d + n] = __float2bfloat16_rn(nx * in.gain[i >> 1]);
                    ssq[nt][i & 1] = fmaf(nx, nx, ssq[nt][i & 1]);
                }
            }
        }
    if (resid || P.kind == CH_LM) {
        // over the 8 lanes with the same t (features g and g + 8 of the item)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int r = nt * 8 + 2 * t4 + c;
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    if (resid) {
                        ssq[nt][c] += __shfl_xor_sync(0xffffffffu, ssq[nt][c], o);
                    } else {
                        const float ov = __shfl_xor_sync(0xffffffffu, bv[nt][c], o);
                        const int oi = __shfl_xor_sync(0xffffffffu, bi[nt][c], o);
                        if (better(ov, oi, bv[nt][c], bi[nt][c])) {
                            bv[nt][c] = ov;
                            bi[nt][c] = oi;
                        }
                    }
                }
                if (resid) {
                    if (g == 0 && r < a.R) a.ss[it * kMaxRows + r] = ssq[nt][c];
                } else if (better(bv[nt][c], bi[nt][c], run_v[nt][c], run_i[nt][c])) {
                    run_v[nt][c] = bv[nt][c];   // this CTA's best of the phase so far
                    run_i[nt][c] = bi[nt][c];
                }
            }
    }
}

// 1 / rms of each of the R rows from the 16-feature partial sums of squares
// of the residual (ss[group][row]): lane l adds groups l, l + 32, ... in that
// order, then a butterfly, and lane 0's total is used; the same order for
// every R.  A group's row sums are contiguous, so all rows load together.
template <int NT>
KS_DEV void row_scales(const ChainArgs& a, int lane, float* out) {
    constexpr int kRows = NT * 8;
    const int R = a.R;   // <= kRows
    const int groups = (a.d + 15) >> 4;
    float s[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) s[r] = 0.f;
#pragma unroll 8
    for (int q = lane; q < groups; q += 32) {
        const float4* src = reinterpret_cast<const float4*>(a.ss + (size_t)q * kMaxRows);
#pragma unroll
        for (int v = 0; v < kRows / 4; ++v) {
            if (4 * v < R) {
                const float4 f = __ldcg(src + v);
                s[4 * v] += f.x;
                s[4 * v + 1] += f.y;
                s[4 * v + 2] += f.z;
                s[4 * v + 3] += f.w;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        if (r < R) {
            const float t = warp_sum(s[r]);
            if (lane == 0) out[r] = rsqrtf(t / (float)a.d + a.eps);
        }
    }
    __syncwarp();
}

// The whole CTA, as it leaves: the last CTA of the launch to leave resets the
// queues and counters of its counter set for a later launch (with all its
// threads: the launch is complete, and its dependents may go on, only then).
KS_DEV void count_out(int n_phases, int* queue, int* done, int* exits, int* blocks) {
    __shared__ int last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(exits, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = threadIdx.x; i < n_phases * kMaxBlocks; i += kThreads) blocks[i] = 0;
    for (int i = threadIdx.x; i < n_phases; i += kThreads) queue[i] = 0;
    if (threadIdx.x == 0) {
        *done = 0;
        *exits = 0;
    }
}

template <int NT, int CTAS_PER_SM>
__global__ void __launch_bounds__(kThreads, CTAS_PER_SM) chain_kernel(const __grid_constant__ ChainArgs a) {
    // A draft pass after the dynamic exit: nothing to do.  The flag only
    // changes between passes, so every CTA of the launch sees the same value.
    if (a.stop && *a.stop) return;
    extern __shared__ unsigned char smem_raw[];
    // 1024-byte aligned: the 128-byte swizzle pattern repeats every 1024 bytes
    __nv_bfloat16* ring = reinterpret_cast<__nv_bfloat16*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    __shared__ __align__(8) uint64_t full[kMaxStages];
    __shared__ __align__(8) uint64_t empty[kMaxStages];
    __shared__ __align__(8) uint64_t pub[kMaxStages];
    __shared__ int slot_k[kMaxStages], slot_it[kMaxStages], slot_kt[kMaxStages];
    __shared__ int slot_last[kMaxStages];   // the stage ends this CTA's last item of its phase
    __shared__ float ones[kMaxRows];        // the input scale of phases without a norm
    __shared__ float scale[kMaxRows];       // 1 / rms of the rows (epilogue warp only)
    __shared__ float red[2][4][2][NT * 4][32];   // [buffer][consumer warp][gate, up][fragment][lane]
    __shared__ int red_k[2], red_it[2], red_last[2];
    __shared__ __align__(8) uint64_t red_full[2];   // 4 consumer warps arrive
    __shared__ __align__(8) uint64_t red_free[2];   // the epilogue warp arrives
    __shared__ int void_job;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = a.R, S = a.stages;
    const int stage_elems = 4 * kBoxElems + 4 * 256 * R;
    int* queue = a.counters;
    int* done = a.counters + kChainMaxPhases;             // LM head items finished
    int* exits = a.counters + kChainMaxPhases + 1;
    int* blocks = a.counters + kChainMaxPhases + 2;       // [phase][kMaxBlocks]

    if (tid == 0) {
        // A job whose status word already holds an error is void (the word
        // stays set until the model is created again): the CTA skips its
        // work, so each later launch of the job ends at once instead of
        // running into bounded waits of its own.  One thread reads the word
        // (it can change during the launch) and the barrier below hands the
        // decision to the whole CTA.
        void_job = __ldcg(a.err) != 0;
        for (int i = 0; i < S; ++i) {
            mbar_init(&full[i], 2);
            mbar_init(&empty[i], 4);
            mbar_init(&pub[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&red_full[i], 4);
            mbar_init(&red_free[i], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < kMaxRows) ones[tid] = 1.f;
    __syncthreads();
    if (void_job) {   // still counted out, so the launch's counters are reset
        count_out(a.n_phases, queue, done, exits, blocks);
        return;
    }

    if (warp == kWarpW) {
        // -------------------------------------------------- weight loader
        if (lane == 0) {
            bool ok = true;
            int t = 0;
            auto issue = [&](int k, const Phase& P, int it, int kt, bool last_item) -> bool {
                const int slot = t % S;
                // self-check: every box coordinate below follows from these ranges
                if (k < 0 || k >= a.n_phases || it < 0 || it >= P.n_items || kt < 0 || kt >= P.tpi) {
                    set_err(a.err, kErrCheckW);
                    return false;
                }
                if (t >= S && !mbar_wait(&empty[slot], (uint32_t)(((t / S) - 1) & 1), kWaitLimitNs)) return false;
                slot_k[slot] = k;
                slot_it[slot] = it;
                slot_kt[slot] = kt;
                slot_last[slot] = last_item;
                mbar_expect_tx(&full[slot], kWBytes);
                __nv_bfloat16* st = ring + (size_t)slot * stage_elems;
                const CUtensorMap* wm = &a.wmap[k];
                unsigned char* sb = reinterpret_cast<unsigned char*>(st);
                if (maps_3d(P)) {
                    if (P.kind == CH_GU) {   // 8 gate chunks, then 8 up chunks
                        tma_3d(sb, wm, 0, it * 16, 8 * kt, &full[slot]);
                        tma_3d(sb + 8 * kChunkBytes, wm, 0, P.N + it * 16, 8 * kt, &full[slot]);
                    } else {
                        tma_3d(sb, wm, 0, it * 16, 16 * kt, &full[slot]);
                    }
                } else if (P.kind == CH_GU) {
                    for (int c = 0; c < 8; ++c) {
                        tma_2d(sb + c * kChunkBytes, wm, kt * 512 + 64 * c, it * 16, &full[slot]);
                        tma_2d(sb + (8 + c) * kChunkBytes, wm, kt * 512 + 64 * c, P.N + it * 16, &full[slot]);
                    }
                } else {
                    for (int c = 0; c < 16; ++c)
                        tma_2d(sb + c * kChunkBytes, wm, kt * 1024 + 64 * c, it * 16, &full[slot]);
                }
                mbar_arrive(&pub[slot]);
                ++t;
                return true;
            };
            // Work assignment per phase: the CTA's first item is fixed by its
            // index (item blockIdx.x, if the phase has that many), so phases
            // with about one item per CTA (W_o, W_down, QKV) spread over every
            // CTA; further items come from the phase's atomic queue, offset by
            // the grid size.  This launch's queues were zeroed by the launch
            // before the previous one (counter sets alternate), which has
            // completed.  Weight boxes need no input, so the first S stages
            // go out while the previous kernel runs.  No deadlock: every CTA
            // of the grid is co-resident once the kernels before it finish,
            // and a CTA finishes its items of a phase before it waits for the
            // next phase's inputs.
            const int grid = (int)gridDim.x;
            int k = 0;
            Phase P = decode(a, 0);
            int it = (int)blockIdx.x;
            while (ok) {
                if (it >= P.n_items) {
                    if (++k >= a.n_phases) break;
                    P = decode(a, k);
                    it = (int)blockIdx.x;
                    continue;
                }
                // claimed ahead: its latency hides behind the stream (the
                // ticket is first needed at the item's last stage, so its
                // round trip overlaps the item's other stages)
                const int next = P.n_items > grid ? grid + atomicAdd(&queue[k], 1) : INT_MAX;
                for (int kt = 0; kt < P.tpi && ok; ++kt)
                    ok = issue(k, P, it, kt, kt == P.tpi - 1 && next >= P.n_items);
                it = next;
            }
            if (ok) {  // sentinel stage: no more work
                const int slot = t % S;
                if (t >= S && !mbar_wait(&empty[slot], (uint32_t)(((t / S) - 1) & 1), kWaitLimitNs)) {
                    ok = false;
                } else {
                    slot_k[slot] = -1;
                    mbar_arrive(&full[slot]);
                    mbar_arrive(&pub[slot]);
                }
            }
            if (!ok) set_err(a.err, kErrWait);
            // (a dependent launch starts only after this grid's predecessor
            // completed, so the alternating counter sets never overlap)
            grid_dependency_wait();
            grid_launch_dependents();
        }
    } else if (warp == kWarpA) {
        // ---------------------------------------------- activation loader
        // Every lane waits for a stage's record itself: when lane 0 waited and
        // a shuffle told the others (which orders no memory), they read the
        // record unsynchronised, and a lane that saw the slot's previous stage
        // could leave for the exit barrier alone, with lane 0 left for ever at
        // the next warp-wide operation.
        grid_dependency_wait();   // the first phase's input comes from the previous kernel
        int cur = -1, ready = 0, prev_n = 0;
        Phase P;
        bool ok = true;
        for (int t = 0;; ++t) {
            const int slot = t % S;
            if (!__all_sync(0xffffffffu, mbar_wait(&pub[slot], (uint32_t)((t / S) & 1), kWaitLimitNs))) {
                ok = false;
                break;
            }
            const int k = slot_k[slot];
            if (k < 0) {
                if (lane == 0) mbar_arrive(&full[slot]);
                break;
            }
            const int kt = slot_kt[slot];
            if (k >= a.n_phases || kt < 0) {   // self-check of the stage record (the same in every lane)
                if (lane == 0) set_err(a.err, kErrCheckA);
                ok = false;
                break;
            }
            if (k != cur) {
                cur = k;
                P = decode(a, k);
                prev_n = k > 0 ? decode(a, k - 1).N : 0;
                ready = 0;      // blocks of phase k - 1 known to be complete
            }
            if (kt >= P.tpi) {
                if (lane == 0) set_err(a.err, kErrCheckA);
                ok = false;
                break;
            }
            if (k > 0 && kt >= ready) {
                // wait for the block of phase k - 1 that this stage reads; the
                // lanes look at the blocks from `ready` on together, so that
                // one round trip finds all that are complete
                const uint64_t t0 = global_ns();
                for (;;) {
                    const int b = ready + lane;
                    const bool done_b = b < P.tpi && ld_relaxed(&blocks[(k - 1) * kMaxBlocks + b]) >=
                                                         block_rowgroups(prev_n, stage_cols(P.kind), b);
                    const uint32_t open = ~__ballot_sync(0xffffffffu, done_b);
                    ready += open == 0 ? 32 : __ffs(open) - 1;
                    if (ready > kt) break;
                    if (__any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) {
                        ok = false;
                        break;
                    }
                }
                if (!ok) break;
                fence_acq_rel();             // the counters were read relaxed: order the rows behind them
                fence_proxy_async_global();
                __syncwarp();
            }
            if (lane == 0) {
                const int chunks = P.kind == CH_GU ? 8 : 16;
                mbar_expect_tx(&full[slot], (uint32_t)(chunks * 128 * R));
                unsigned char* dst = reinterpret_cast<unsigned char*>(ring + (size_t)slot * stage_elems) + kWBytes;
                const CUtensorMap* am = amap_of(a, P.kind);
                if (maps_3d(P)) tma_3d(dst, am, 0, 0, chunks * kt, &full[slot]);
                else for (int c = 0; c < chunks; ++c) tma_2d(dst + c * 128 * R, am, (chunks * kt + c) * 64, 0, &full[slot]);
            }
            __syncwarp();
        }
        if (!ok && lane == 0) set_err(a.err, kErrWait);
    } else if (warp < 4) {
        // ------------------------------------------------------ consumers
        // The warps go their own pace: a stage is read when its barrier says
        // so and freed by all four, and their sums meet through the partials
        // buffers.  One whose bounded wait gives up leaves by itself; the
        // others' waits then end the same way.
        float acc[kChains][NT][4], accu[kChains][NT][4];
        bool failed = false;
        int n_items = 0;   // items finished by this CTA (selects the partials buffer)
        int cur = -1;
        Phase P;
        for (int t = 0;; ++t) {
            const int slot = t % S;
            // the vote also brings the lanes together: they leave the wait's
            // loop one by one, and ldmatrix and mma need the whole warp
            if (!__all_sync(0xffffffffu, mbar_wait(&full[slot], (uint32_t)((t / S) & 1), kWaitLimitNs))) {
                failed = true;
                break;
            }
            const int k = slot_k[slot];
            const int it = slot_it[slot], kt = slot_kt[slot];
            const bool last_item = slot_last[slot] != 0;
            const int b = n_items & 1;
            if (k < 0) {
                // no more stages: tell the epilogue warp to stop
                if (n_items >= 2 && !mbar_wait(&red_free[b], (uint32_t)(((n_items >> 1) - 1) & 1), kWaitLimitNs))
                    failed = true;
                if (warp == 0 && lane == 0) red_k[b] = -1;
                __syncwarp();
                if (lane == 0) mbar_arrive(&red_full[b]);
                break;
            }
            if (k >= a.n_phases || kt < 0 || it < 0) {   // self-check (the same record in every warp)
                if (lane == 0) set_err(a.err, kErrCheckC);
                failed = true;
                break;
            }
            if (k != cur) {
                cur = k;
                P = decode(a, k);
            }
            if (kt >= P.tpi || it >= P.n_items) {
                if (lane == 0) set_err(a.err, kErrCheckC);
                failed = true;
                break;
            }
            if (kt == 0) {
#pragma unroll
                for (int c = 0; c < kChains; ++c)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[c][nt][i] = accu[c][nt][i] = 0.f;
            }
            const uint32_t st = smem_u32(ring + (size_t)slot * stage_elems);
            if (P.kind == CH_GU) mma_stage<NT, true>(st, R, warp, lane, acc, accu);
            else mma_stage<NT, false>(st, R, warp, lane, acc, accu);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot]);   // this warp is done with the stage
            if (kt != P.tpi - 1) continue;

            // item done: add the chains in chain order and hand this warp's
            // sums to the epilogue warp through partials buffer b (double
            // buffered: the consumers move straight on to the next item)
#pragma unroll
            for (int c = 1; c < kChains; ++c)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[0][nt][i] += acc[c][nt][i];
                        accu[0][nt][i] += accu[c][nt][i];
                    }
            if (n_items >= 2 &&
                !__all_sync(0xffffffffu, mbar_wait(&red_free[b], (uint32_t)(((n_items >> 1) - 1) & 1), kWaitLimitNs))) {
                failed = true;
                break;
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    red[b][warp][0][nt * 4 + i][lane] = acc[0][nt][i];
                    if (P.kind == CH_GU) red[b][warp][1][nt * 4 + i][lane] = accu[0][nt][i];
                }
            if (warp == 0 && lane == 0) {
                red_k[b] = k;
                red_it[b] = it;
                red_last[b] = last_item;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&red_full[b]);
            ++n_items;
        }
        if (failed && lane == 0) set_err(a.err, kErrWait);
    } else if (warp == kWarpE) {
        // --------------------------------------------------- epilogue warp
        grid_dependency_wait();   // epilogues write buffers the previous kernel uses
        float acc[NT][4], accu[NT][4];
        float run_v[NT][2];       // LM head: this CTA's best (logit, id) per row
        int run_i[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                run_v[nt][c] = -INFINITY;
                run_i[nt][c] = INT_MAX;
            }
        int lm_items = 0;         // LM head items finished by this CTA
        int cur = -1, next_cols = 0;   // the phase P describes, the columns of the next one's stages
        Phase P;
        int scale_k = -1;         // the phase whose row scales `scale` holds
        bool ok = true;
        for (int n = 0;; ++n) {
            const int b = n & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&red_full[b], (uint32_t)((n >> 1) & 1), kWaitLimitNs))) {
                ok = false;
                break;
            }
            const int k = red_k[b];
            if (k < 0) break;
            const int it = red_it[b];
            const bool last_item = red_last[b] != 0;
            if (k < a.n_phases && k != cur) {
                cur = k;
                P = decode(a, k);
                next_cols = k + 1 < a.n_phases ? stage_cols(decode(a, k + 1).kind) : 0;
            }
            if (k >= a.n_phases || it < 0 || it >= P.n_items) {   // self-check
                set_err(a.err, kErrCheckE);
                ok = false;
                break;
            }
            ResidIn<NT> in;
            if (!normed_input(P.kind)) in.load(a, P, k, it);
            // the four warps' K quarters, added in warp order
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[nt][i] = red[b][0][0][nt * 4 + i][lane];
                    accu[nt][i] = (P.kind == CH_GU) ? red[b][0][1][nt * 4 + i][lane] : 0.f;
                }
#pragma unroll
            for (int w = 1; w < 4; ++w)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[nt][i] += red[b][w][0][nt * 4 + i][lane];
                        if (P.kind == CH_GU) accu[nt][i] += red[b][w][1][nt * 4 + i][lane];
                    }
            __syncwarp();
            if (lane == 0) mbar_arrive(&red_free[b]);   // partials read: the buffer is free
            if (normed_input(P.kind) && k != scale_k) {
                // This CTA's first item of a normed phase: its last stage
                // waited for every block of phase k - 1 (an item's stages
                // cover them all), so every row group's partial sums of
                // squares are written.
                scale_k = k;
                row_scales<NT>(a, lane, scale);
            }
            epilogue<NT>(a, P, it, in, acc, accu, normed_input(P.kind) ? scale : ones, run_v, run_i);
            lm_items += P.kind == CH_LM;
            if (k + 1 < a.n_phases) {
                // publish this row group to the next phase's stages that read it
                fence_proxy_async_global();
                __syncwarp();
                if (lane == 0) {
                    __threadfence();
                    atomicAdd(&blocks[k * kMaxBlocks + (it * 16) / next_cols], 1);
                }
            }
            if (last_item && P.kind == CH_LM) {
                // this CTA's last LM head item: merge its per-row best into the
                // global keys, then count its items
                const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int r = nt * 8 + 2 * t4 + c;
                        if (g == 0 && r < R && run_i[nt][c] != INT_MAX)
                            atomicMax(&a.best[r], argmax_key(run_v[nt][c], run_i[nt][c]));
                    }
                __syncwarp();
                int fin = 0;
                if (lane == 0) {
                    __threadfence();
                    fin = atomicAdd(done, lm_items) + lm_items == P.n_items;
                }
                if (__shfl_sync(0xffffffffu, fin, 0)) {
                    // every CTA has merged: read the keys (and leave them zero)
                    __threadfence();
                    if (lane < R) {
                        const unsigned long long key = atomicExch(&a.best[lane], 0ull);
                        a.tokens[lane] = key == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
                    }
                }
            }
        }
        if (!ok && lane == 0) set_err(a.err, kErrWait);
    }

    // the last CTA to leave resets the queues and counters for the next launch
    __syncthreads();
    count_out(a.n_phases, queue, done, exits, blocks);
}

}  // namespace

size_t chain_counter_ints() { return (size_t)kChainMaxPhases + 2 + (size_t)kChainMaxPhases * kMaxBlocks; }

cudaError_t launch_chain(const ChainArgs& args, cudaStream_t s) {
    if (args.R < 1 || args.R > kMaxRows || args.n_phases < 1 || args.n_phases > kChainMaxPhases ||
        args.err == nullptr || args.counters == nullptr)
        return cudaErrorInvalidValue;
    ChainArgs a = args;
    const int per_sm = a.R <= 8 ? 2 : 1;
    const size_t stage_bytes = kWBytes + 4u * 256u * 2u * (size_t)a.R;
    a.stages = (int)((per_sm == 2 ? kRingBudget2 : kRingBudget1) / stage_bytes);
    if (a.stages > kMaxStages) a.stages = kMaxStages;
    const size_t smem = (size_t)a.stages * stage_bytes + 1024;  // + alignment slack
    auto run = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        // two CTAs per SM when they fit (they normally do); fewer only slows
        // the launch down, since no CTA waits for one that is not running
        int fit = per_sm;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, kThreads, smem) != cudaSuccess || fit < 1)
            fit = 1;
        cfg.gridDim = dim3(std::min(fit, per_sm) * sm_count());
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, a);
    };
    return per_sm == 2 ? run(chain_kernel<1, 2>) : run(chain_kernel<2, 1>);
}

}  // namespace ks
