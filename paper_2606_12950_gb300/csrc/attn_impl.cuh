// attn_impl.cuh -- paged decode attention kernel for sm_103a.
//
// One decode query per (sequence, query head) attends over the sequence's
// cached K/V (the decode phase, paper §II "LLM inference cost model"), which
// sits in fixed-size blocks of one shared pool reached through a per-sequence
// block table (§II / §III-C).  Per (s, h), with g = h / G:
//     out = sum_j softmax_j(scale * q . K_j) V_j
// evaluated with an online softmax in base 2 and fp32 accumulation.
//
// Work decomposition (all decided on the device from the lengths):
//   unit  = one tile of one (sequence, KV head) run: 16 tokens at d = 128,
//           32 at d = 64 (kUnit), 8 KB of K and V either way; a run of n
//           tokens has ceil(n/kUnit) units; units are ordered (s, g, tile).
//   part  = a contiguous unit range: the units are cut into equal ranges, one
//           per resident CTA, and each of those into equal ranges, one per
//           warp: every warp streams the same number of bytes (+-2 tiles)
//           whatever the length distribution.  A part is a warp's range, or
//           with MERGE a CTA's.
//   piece = the units of one run in one warp's range.  A run inside one part
//           is finished in place; a run cut by part boundaries leaves one
//           fp32 partial (max, sum, unnormalised output) per part, which the
//           combine kernel below merges in part order, a CTA's partials
//           first.
// Each warp streams its own contiguous range of units through its own
// shared-memory stage, issuing its own 2-D TMA loads (128-byte swizzle) of
// each unit's K and V tiles with one mbarrier for K and one for V: the next
// unit's K streams in while the warp does softmax and P.V on the current one,
// the next V while it does the next q.K.  (Measured on GB300: one issuing
// thread per SM cannot keep HBM busy with these 2 KB boxes; one per warp
// can.)  The pool rows of a warp's units are resolved from the block table in
// the prologue, while the memory system is idle, so no table load sits on the
// streaming path, and each run's q rows (and, for the run's last tile, this
// step's new K/V rows) are staged into the warp's shared buffers by cp.async
// one piece ahead.
//
// MERGE: the warps of a CTA that share a run merge their states in shared
// memory at the CTA's end, so that the CTA leaves the run's output, or one
// record instead of six.  The combine then has far fewer records to fetch, at
// the cost of a barrier and the merge (about 1 us) at the end of every CTA.
// - Without step overlap the combine is on the critical path, and the merge
//   pays at every size.  Same box, merged and not: 48 sequences at 8 query
//   heads a KV head 76.4 and 77.9 us, three co-located models 266.6 and
//   275.6, the 64-sequence layer 69.0 and 71.2, 1024 long contexts 690.3 and
//   695.7.
// - Where the next step's decode kernel overlaps the combine (chain 3), only
//   the CTAs' later end shows: 69.8 and 68.1 us for the 64-sequence layer.
//   There each warp leaves its record.  The bits are the same: the combine
//   merges a CTA's records in the same order and arithmetic first.
// - Small batches always merge (kMergeUnits).  What bounds them is latency: a
//   warp takes its units one after another, and every record is one more to
//   fetch, so their units go to as many warps as there are.  One sequence of
//   8193 tokens (32 q / 8 KV heads, 33.6 MB) has 38 records a run instead of
//   128; a step took 18.0 us before and 14.4 after (of it, the combine's
//   column slices: 2.3).  8 sequences of 601-3500 tokens (40 q / 8 KV heads,
//   67 MB, 4.5 units a warp): 20.3 us, 21.1 with the line at 4 units.
//
// Grid-to-grid order: the kernel is launched as a programmatic dependent.
// Alone it releases the next grid and waits for the one before; as part of
// a chain (beside the shared-prefix kernel, or the later batches of several
// co-located ones) it starts without waiting, reads what earlier grids wrote
// through L2 only, and waits at its end (AttnArgs::chain).  Right after a
// split-K combine (step overlap) it starts without waiting too, while the
// combine finishes, and waits before its first write of the output or the
// workspace, which the combine uses.  The step's
// table sync may ride in its parameters (AttnArgs::sync_words); a grid
// alone then computes its work split from those lengths before its wait.
//
// Two compute variants share this skeleton:
//   FmaCompute : CUDA-core FFMA2 dot products and weighted sums.
//   MmaCompute : warp-level tensor-core MMA (m16n8k16 bf16 -> fp32); tokens
//                on M, the query-head group on N (padded to 8), d on K for
//                q.K and on M for P.V; P is moved from accumulator layout to
//                operand layout with movmatrix.
#pragma once

#include <algorithm>
#include <cstdint>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "kvpool.h"
#include "ptx.cuh"

namespace kvp {

// Warps per CTA, each streaming and computing its own units: up to kWarps
// (AttnArgs::nwarps).  Two CTAs of six warps on an SM keep 12 units in
// flight there, which config 2 (64 sequences on all 152 SMs) streams
// fastest; beside the shared-prefix kernel, on fewer SMs, eight do.
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kPlainWarps = 6;
constexpr int kStages = 1;  // units in flight per warp (each a K and a V tile)
constexpr int kTile = 16;                         // tokens per TMA box: the least block size
// Tokens per unit.  A warp's work on a unit is one dependent chain (wait for
// K, q.K, softmax, wait for V, P.V, the next requests) of much the same
// length whatever d is.  At d = 64 a 16-token unit is only 4 KB, and that
// chain, not HBM, set the pace: 128 sequences of lognormal length (209k
// tokens, 32 q / 8 KV heads, 429 MB) took 83.2 us a step with 16-token units
// (78.9 with two units in flight a warp, 79.7 with eight warps a CTA) and
// 75.1 with 32-token ones, which bring d = 64 to the bytes per chain of
// d = 128 (5.7 against 5.2 TB/s).
template <int D>
constexpr int kUnit = D == 64 ? 32 : 16;
template <int D>
constexpr int kSub = kUnit<D> / kTile;            // boxes' rows per unit
// a part's least tokens (4 units at d = 128, 2 at d = 64): with 128 at d = 64
// a step of four short sequences took 18.5 us instead of 15.5
constexpr int kMinPartTokens = 64;
// Below this many units a warp (by the table's width) a warp may have a single
// unit and the CTAs merge in every mode.
constexpr int kMergeUnits = 8;
// Whose records a decode grid leaves, and how the combine finds a run's: each
// warp's and each CTA's (MERGE) by run, or CTAs' by part (see attn_run).
enum { kRecWarps = 0, kRecCtas = 1, kRecCtasByPart = 2 };
// Where a state's running maximum starts.  Finite, so that a token whose score
// is -inf gets weight 0 also before any other (2^(-inf - m), not 2^NaN), and so
// that no record of a part has m = -inf, which stands for "no record" in the
// merges: a part whose scores are all NaN leaves this m with l = NaN, and the
// output is NaN, however the run was cut.
constexpr float kMaxStart = -3.402823466e+38f;  // the lowest float
constexpr uint32_t kHalfBytes = kTile * 128;      // one 64-column box: 16 rows x 128 B
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // bounded mbarrier waits: 2 s

// Loads of data written by earlier grids: through L2 only (ld.global.cg) when
// the kernel did not wait for the grid before it (a chained grid: beside the
// shared-prefix kernel, a later batch of paged_decode_attn_multi, or a step
// overlapping the previous step's combine), so that no line an earlier
// kernel left in this SM's L1 is read; plain otherwise.
template <class T>
__device__ __forceinline__ T ld_prior(const T *p, bool l2_only)
{
    return l2_only ? __ldcg(p) : *p;
}

// Words of a table sync carried by the decode kernel's parameters (lengths,
// then (flat index, value) pairs of changed table entries): 512 bytes, which
// every launch carries.  A 1.8 KB block cost the launch more than the
// separate sync kernel saved (measured on config 2).
constexpr int kSyncWords = 128;

struct AttnArgs {
    const uint16_t *q;
    uint16_t *out;
    const uint16_t *k_new;   // fused append: this step's K/V rows [S][Hkv][d], or null
    const uint16_t *v_new;
    uint16_t *pool;          // pool base (rows of d bf16), for the fused append's writes
    const int32_t *table;
    const int32_t *ctx_lens;
    int32_t *err;
    float *ws_part;
    int2 *ws_run;            // per run: the parts of its records, [x, y); y = x if it has none.
                             // kRecCtasByPart: per part, the run that starts in it and goes on
                             // (x), and the one that ends in it and started earlier (y); or -1
    int64_t rows_per_page;   // page_bytes / (d * 2)
    int64_t pool_pages;
    int32_t pages_per_block;
    int32_t max_blocks;
    int32_t S;
    int32_t Hkv;
    int32_t bs;
    int32_t bs_shift;        // log2(bs), or -1
    int32_t rows_cap;        // boxes whose pool rows are resolved up front
    int32_t P;               // CTAs
    int32_t nwarps;          // warps per CTA (<= kWarps)
    int32_t min_units;       // least units of a warp (but in a CTA with fewer units than warps);
                             // to attn_run: in a small batch, 0 = 1
    float qk_scale;          // scale * log2(e)
    // shared-prefix (cascade) mode: tokens of each sequence's prefix handled
    // by the prefix kernel ([S], multiples of 16; null = none), its records
    // and key-split count (read by the combine)
    const int32_t *skip;
    const float *ws_pre;
    int32_t KS;
    // place in a chain of grids: 0 alone (release the next grid, then wait
    // for the one before); 1 first of a chain (wait, then release: the next
    // grid relies on this wait); 2 chained (release, no wait at the start,
    // a wait at the exit: see the kernel); 3 right after a split-K combine
    // of this library, which released this grid only after its own wait, so
    // every grid before that combine has completed (release, no wait at the
    // start, a wait before the first write of the output or the workspace,
    // which the combine still uses, and at the exit); 4 beside the
    // shared-prefix kernel while the previous step's shared-prefix combine
    // finishes (release, no wait at the start; the plan kernel's two flags,
    // below, stand in for the waits: the first before anything the plan
    // kernel writes is read, the second before the first write of the output
    // or the workspace; a wait for the prefix grid at the exit)
    int32_t chain;
    // chain 4: the plan kernel sets flags[0] = epoch once the plan, the
    // skips and the table sync are written, and flags[1] = epoch once every
    // grid before it has completed
    const uint64_t *flags;
    uint64_t epoch;
    // fused table sync (paged_decode_attn_seqtab): this step's lengths of
    // rows [0, sync_nlens) and its changed table entries travel here.  The
    // kernel takes the lengths and those entries from here, and the CTAs
    // write them to sync_lens / sync_table for later kernels.  Null: none.
    int32_t *sync_table;
    int32_t *sync_lens;
    int32_t sync_nlens;
    int32_t sync_npatch;
    int32_t sync_words[kSyncWords];
};

__device__ __forceinline__ void report(int32_t *err, int code) { atomicCAS(err, 0, code); }

// bounded wait on an mbarrier phase; a wait that exceeds the limit records
// KV_ERR_DEVICE_TIMEOUT and makes every later wait of this warp return at once
__device__ __forceinline__ void wait_phase(uint32_t bar, uint32_t parity, int32_t *err, bool &dead)
{
    if (dead) return;
    if (mbar_try_wait(bar, parity)) return;
    uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return;
        if ((it & 1023u) == 0 && global_timer_ns() - t0 > kWaitLimitNs) {
            report(err, KV_ERR_DEVICE_TIMEOUT);
            dead = true;
            return;
        }
    }
}

// bounded wait until another grid has stored `epoch` in *flag (release
// store; this load acquires); a wait past the limit records
// KV_ERR_DEVICE_TIMEOUT and returns
__device__ __forceinline__ void wait_flag(const uint64_t *flag, uint64_t epoch, int32_t *err)
{
    if (ld_acquire_gpu(flag) == epoch) return;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        __nanosleep(64);
        if (ld_acquire_gpu(flag) == epoch) return;
        if ((it & 255u) == 0 && global_timer_ns() - t0 > kWaitLimitNs) {
            report(err, KV_ERR_DEVICE_TIMEOUT);
            return;
        }
    }
}

// shared-memory byte offset of 16-byte chunk c (8 bf16 of columns 8c..8c+7)
// of tile row r, in the 128-byte-swizzled layout TMA writes
__device__ __forceinline__ uint32_t swz(int r, int c)
{
    return (uint32_t)((c >> 3) * kHalfBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// ------------------------------------------------------------ CUDA cores ---
template <int D, int G>
struct FmaCompute {
    static constexpr int kMinBlocks = 1;                     // registers allow one CTA per SM
    static constexpr int LPT = (G * D / 8 <= 64) ? 8 : 16;  // lanes per token
    static constexpr int EPL = D / LPT;                      // elements per lane
    static constexpr int NCH = EPL / 8;                      // 16-byte chunks per lane
    static constexpr int NGRP = 32 / LPT;                    // tokens in flight per warp
    static constexpr int TPG = kUnit<D> / NGRP;              // tokens per group per unit
    static_assert(EPL % 8 == 0, "lane slice must be whole 16-byte chunks");

    float2 q[G][EPL / 2];
    float2 o[G][EPL / 2];
    float m[G];
    float l[G];
    float p[TPG][G];
    int grp, sub, nv;

    // qrow: the run's G query rows, staged in shared memory
    __device__ __forceinline__ void begin(const uint16_t *qrow, float qk_scale, int lane)
    {
        grp = lane / LPT;
        sub = lane % LPT;
#pragma unroll
        for (int h = 0; h < G; ++h) {
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const int c = sub + j * LPT;
                uint4 w = *reinterpret_cast<const uint4 *>(qrow + h * D + c * 8);
                uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    q[h][j * 4 + e] = make_float2(bf_lo(ws[e]) * qk_scale, bf_hi(ws[e]) * qk_scale);
            }
#pragma unroll
            for (int e = 0; e < EPL / 2; ++e) o[h][e] = make_float2(0.f, 0.f);
            m[h] = kMaxStart;
            l[h] = 0.f;
        }
    }

    // q.K for the tile's tokens, online-softmax update, weights p
    __device__ __forceinline__ void scores(const uint8_t *Ks, int nvalid)
    {
        nv = nvalid;
        float sc[TPG][G];
#pragma unroll
        for (int i = 0; i < TPG; ++i) {
            const int t = grp + i * NGRP;
            float2 acc[G];
#pragma unroll
            for (int h = 0; h < G; ++h) acc[h] = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                uint4 w = *reinterpret_cast<const uint4 *>(Ks + swz(t, sub + j * LPT));
                uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float2 kv = make_float2(bf_lo(ws[e]), bf_hi(ws[e]));
#pragma unroll
                    for (int h = 0; h < G; ++h) acc[h] = __ffma2_rn(q[h][j * 4 + e], kv, acc[h]);
                }
            }
#pragma unroll
            for (int h = 0; h < G; ++h) sc[i][h] = acc[h].x + acc[h].y;
        }
        // dot products are split over LPT lanes: butterfly sum
#pragma unroll
        for (int off = 1; off < LPT; off <<= 1)
#pragma unroll
            for (int i = 0; i < TPG; ++i)
#pragma unroll
                for (int h = 0; h < G; ++h) sc[i][h] += __shfl_xor_sync(0xffffffffu, sc[i][h], off);
        float tmax[G];
#pragma unroll
        for (int h = 0; h < G; ++h) tmax[h] = -INFINITY;
#pragma unroll
        for (int i = 0; i < TPG; ++i) {
            const bool ok = grp + i * NGRP < nvalid;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                sc[i][h] = ok ? sc[i][h] : -INFINITY;
                tmax[h] = fmaxf(tmax[h], sc[i][h]);
            }
        }
#pragma unroll
        for (int off = LPT; off < 32; off <<= 1)
#pragma unroll
            for (int h = 0; h < G; ++h) tmax[h] = fmaxf(tmax[h], __shfl_xor_sync(0xffffffffu, tmax[h], off));
        // lazy rescale: keep the running max unless the tile exceeds it by
        // more than 2^8 (o and l share the stale max, so the ratio is exact)
#pragma unroll
        for (int h = 0; h < G; ++h) {
            if (tmax[h] > m[h] + 8.f) {
                const float a = fast_exp2(m[h] - tmax[h]);
                l[h] *= a;
#pragma unroll
                for (int e = 0; e < EPL / 2; ++e) o[h][e] = make_float2(o[h][e].x * a, o[h][e].y * a);
                m[h] = tmax[h];
            }
        }
#pragma unroll
        for (int i = 0; i < TPG; ++i)
#pragma unroll
            for (int h = 0; h < G; ++h) {
                p[i][h] = fast_exp2(sc[i][h] - m[h]);
                l[h] += p[i][h];
            }
    }

    __device__ __forceinline__ void softmax() {}

    // o += p * V for the tile's valid tokens
    __device__ __forceinline__ void pv(uint8_t *Vs)
    {
#pragma unroll
        for (int i = 0; i < TPG; ++i) {
            const int t = grp + i * NGRP;
            if (t < nv) {
#pragma unroll
                for (int j = 0; j < NCH; ++j) {
                    uint4 w = *reinterpret_cast<const uint4 *>(Vs + swz(t, sub + j * LPT));
                    uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float2 vv = make_float2(bf_lo(ws[e]), bf_hi(ws[e]));
#pragma unroll
                        for (int h = 0; h < G; ++h)
                            o[h][j * 4 + e] = __ffma2_rn(make_float2(p[i][h], p[i][h]), vv, o[h][j * 4 + e]);
                    }
                }
            }
        }
    }

    // end of a piece: the bf16 output o / l (whole run in this warp), or the
    // fp32 partial (o unnormalised, m, l) of this warp's part of the run
    __device__ __forceinline__ void store(uint16_t *orow, float *slot, bool split, int lane)
    {
#pragma unroll
        for (int off = LPT; off < 32; off <<= 1)
#pragma unroll
            for (int h = 0; h < G; ++h) {
                l[h] += __shfl_xor_sync(0xffffffffu, l[h], off);
#pragma unroll
                for (int e = 0; e < EPL / 2; ++e) {
                    o[h][e].x += __shfl_xor_sync(0xffffffffu, o[h][e].x, off);
                    o[h][e].y += __shfl_xor_sync(0xffffffffu, o[h][e].y, off);
                }
            }
        if (grp == 0) {
#pragma unroll
            for (int h = 0; h < G; ++h)
#pragma unroll
                for (int j = 0; j < NCH; ++j) {
                    const int c = sub + j * LPT;
                    if (!split) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            __nv_bfloat162 b2 =
                                __floats2bfloat162_rn(o[h][j * 4 + e].x / l[h], o[h][j * 4 + e].y / l[h]);
                            w[e] = *reinterpret_cast<uint32_t *>(&b2);
                        }
                        *reinterpret_cast<uint4 *>(orow + h * D + c * 8) = make_uint4(w[0], w[1], w[2], w[3]);
                    } else {
                        float4 *dst = reinterpret_cast<float4 *>(slot + h * D + c * 8);
                        dst[0] = make_float4(o[h][j * 4 + 0].x, o[h][j * 4 + 0].y, o[h][j * 4 + 1].x, o[h][j * 4 + 1].y);
                        dst[1] = make_float4(o[h][j * 4 + 2].x, o[h][j * 4 + 2].y, o[h][j * 4 + 3].x, o[h][j * 4 + 3].y);
                    }
                }
        }
        if (split && lane == 0) {
#pragma unroll
            for (int h = 0; h < G; ++h) {
                slot[G * D + h] = m[h];
                slot[G * D + G + h] = l[h];
            }
        }
    }
};

// ----------------------------------------------------------- tensor cores --
template <int D, int G>
struct MmaCompute {
    static_assert(G <= 8, "query-head group must fit the n=8 MMA tile");
    static constexpr int kMinBlocks = 2;
    static constexpr int KS = D / 16;
    static constexpr int NM = kSub<D>;  // 16-token MMA tiles per unit
    uint32_t qf[KS][2];  // B operand of q.K: Q^T fragments (bf16x2)
    float acc[KS][4];    // O^T accumulators, 16 d-rows per block
    float m[2], l[2];    // heads 2*tig, 2*tig+1
    float x[NM][4];      // scores of the unit
    uint32_t pb[NM][2];  // B operand of P.V (P^T fragments)
    float qk_scale;
    int gid, tig, lane_, nv;

    // qrow: the run's G query rows, staged in shared memory
    __device__ __forceinline__ void begin(const uint16_t *qrow, float scale, int lane)
    {
        lane_ = lane;
        gid = lane >> 2;
        tig = lane & 3;
        qk_scale = scale;
#pragma unroll
        for (int kk = 0; kk < KS; ++kk) {
            if (gid < G) {
                qf[kk][0] = *reinterpret_cast<const uint32_t *>(qrow + gid * D + kk * 16 + tig * 2);
                qf[kk][1] = *reinterpret_cast<const uint32_t *>(qrow + gid * D + kk * 16 + tig * 2 + 8);
            } else {
                qf[kk][0] = 0u;
                qf[kk][1] = 0u;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[kk][e] = 0.f;
        }
        m[0] = m[1] = kMaxStart;
        l[0] = l[1] = 0.f;
    }

    // q.K.  (Two sums of every other 16 columns, a chain of MMAs half as long,
    // left the 64-sequence layer at 68.2 us against 67.8 with one.)
    __device__ __forceinline__ void scores(const uint8_t *Ks, int nvalid)
    {
        nv = nvalid;
        const uint32_t kbase = smem_u32(Ks);
        const int mat = lane_ >> 3, r8 = lane_ & 7;
#pragma unroll
        for (int mt = 0; mt < NM; ++mt) {
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < KS; ++kk) {
                uint32_t a0, a1, a2, a3;
                ldmatrix_x4(kbase + swz(mt * 16 + r8 + (mat & 1) * 8, kk * 2 + (mat >> 1)), a0, a1, a2, a3);
                mma_bf16_16816(s, a0, a1, a2, a3, qf[kk][0], qf[kk][1]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) x[mt][e] = s[e] * qk_scale;
        }
    }

    // online softmax of the scores: the weights P as P.V's operand
    __device__ __forceinline__ void softmax()
    {
        // x[0], x[1]: token gid, heads 2tig, 2tig+1; x[2], x[3]: token gid+8.
        // Rows past the valid tokens of a loaded box may hold anything; a box
        // that was not loaded (16 mt >= nv) holds an earlier unit's rows: both
        // are masked
        if (nv < kUnit<D>) {
#pragma unroll
            for (int mt = 0; mt < NM; ++mt) {
                if (mt * 16 + gid >= nv) x[mt][0] = x[mt][1] = -INFINITY;
                if (mt * 16 + gid + 8 >= nv) x[mt][2] = x[mt][3] = -INFINITY;
            }
        }
        float t0 = fmaxf(x[0][0], x[0][2]), t1 = fmaxf(x[0][1], x[0][3]);
#pragma unroll
        for (int mt = 1; mt < NM; ++mt) {
            t0 = fmaxf(t0, fmaxf(x[mt][0], x[mt][2]));
            t1 = fmaxf(t1, fmaxf(x[mt][1], x[mt][3]));
        }
        // lazy rescale (see FmaCompute::scores); the maxima over the tokens are
        // only needed once some lane's exceeds the running one by 2^8
        if (__any_sync(0xffffffffu, t0 > m[0] + 8.f || t1 > m[1] + 8.f)) {
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) {
                t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, off));
                t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, off));
            }
            if (t0 > m[0] + 8.f) {
                const float a = fast_exp2(m[0] - t0);
                l[0] *= a;
#pragma unroll
                for (int mb = 0; mb < KS; ++mb) {
                    acc[mb][0] *= a;
                    acc[mb][2] *= a;
                }
                m[0] = t0;
            }
            if (t1 > m[1] + 8.f) {
                const float a = fast_exp2(m[1] - t1);
                l[1] *= a;
#pragma unroll
                for (int mb = 0; mb < KS; ++mb) {
                    acc[mb][1] *= a;
                    acc[mb][3] *= a;
                }
                m[1] = t1;
            }
        }
#pragma unroll
        for (int mt = 0; mt < NM; ++mt) {
            const float p0 = fast_exp2(x[mt][0] - m[0]), p1 = fast_exp2(x[mt][1] - m[1]);
            const float p2 = fast_exp2(x[mt][2] - m[0]), p3 = fast_exp2(x[mt][3] - m[1]);
            l[0] += p0 + p2;
            l[1] += p1 + p3;
            __nv_bfloat162 lo = __floats2bfloat162_rn(p0, p1);
            __nv_bfloat162 hi = __floats2bfloat162_rn(p2, p3);
            pb[mt][0] = movmatrix_trans(*reinterpret_cast<uint32_t *>(&lo));
            pb[mt][1] = movmatrix_trans(*reinterpret_cast<uint32_t *>(&hi));
        }
    }

    __device__ __forceinline__ void pv(uint8_t *Vs)
    {
        // rows past the context may hold anything (even NaN bit patterns);
        // P is zero there, but 0 * NaN is NaN inside the MMA, so clear them
        if (nv < kUnit<D>) {
            const int nchunk = (kUnit<D> - nv) * (D / 8);
            for (int idx = lane_; idx < nchunk; idx += 32) {
                const int r = nv + idx / (D / 8);
                const int c = idx % (D / 8);
                *reinterpret_cast<uint4 *>(Vs + swz(r, c)) = make_uint4(0u, 0u, 0u, 0u);
            }
            __syncwarp();
        }
        const uint32_t vbase = smem_u32(Vs);
        const int mat = lane_ >> 3, r8 = lane_ & 7;
#pragma unroll
        for (int mb = 0; mb < KS; ++mb) {
#pragma unroll
            for (int mt = 0; mt < NM; ++mt) {
                uint32_t a0, a1, a2, a3;
                ldmatrix_x4_trans(vbase + swz(mt * 16 + r8 + (mat >> 1) * 8, mb * 2 + (mat & 1)), a0, a1, a2, a3);
                mma_bf16_16816(acc[mb], a0, a1, a2, a3, pb[mt][0], pb[mt][1]);
            }
        }
    }

    // end of a piece (see FmaCompute::store)
    __device__ __forceinline__ void store(uint16_t *orow, float *slot, bool split, int lane)
    {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            l[0] += __shfl_xor_sync(0xffffffffu, l[0], off);
            l[1] += __shfl_xor_sync(0xffffffffu, l[1], off);
        }
        const int h0 = 2 * tig, h1 = 2 * tig + 1;
        if (!split) {
#pragma unroll
            for (int mb = 0; mb < KS; ++mb) {
                const int d0 = mb * 16 + gid;
                if (h0 < G) {
                    orow[h0 * D + d0] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[mb][0] / l[0]));
                    orow[h0 * D + d0 + 8] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[mb][2] / l[0]));
                }
                if (h1 < G) {
                    orow[h1 * D + d0] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[mb][1] / l[1]));
                    orow[h1 * D + d0 + 8] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[mb][3] / l[1]));
                }
            }
        } else {
#pragma unroll
            for (int mb = 0; mb < KS; ++mb) {
                const int d0 = mb * 16 + gid;
                if (h0 < G) {
                    slot[h0 * D + d0] = acc[mb][0];
                    slot[h0 * D + d0 + 8] = acc[mb][2];
                }
                if (h1 < G) {
                    slot[h1 * D + d0] = acc[mb][1];
                    slot[h1 * D + d0 + 8] = acc[mb][3];
                }
            }
            if (gid == 0) {
                if (h0 < G) {
                    slot[G * D + h0] = m[0];
                    slot[G * D + G + h0] = l[0];
                }
                if (h1 < G) {
                    slot[G * D + h1] = m[1];
                    slot[G * D + G + h1] = l[1];
                }
            }
        }
        (void)lane;
    }
};

// ----------------------------------------------------------- work units ---
// Index arithmetic.  It is on the critical path of every step (lengths, parts,
// table rows: 4.4 us from a grid's start to its first loads, of which two
// round trips to L2 are 1.2) and again at each run boundary.  So parts take
// 32-bit arithmetic with one division, quotients below 2^20 an estimate from
// the approximate reciprocal, a warp looks up its own rows without a CTA
// barrier, and the run after a piece is stepped to instead of searched for.
// Against 64-bit divisions, a CTA-wide lookup and a search per piece (same
// box): the 64-sequence layer (435 MB) 70.1 -> 67.8 us, 256 chains beside
// their prefix 100.7 -> 95.5, 128 sequences at d = 64 74.0 -> 69.8, three
// co-located models 281.7 -> 277.5, 1024 long contexts 705.7 -> 699.0.
//
// x / d for a quotient below 2^20 (x and d positive and below 2^31), inv =
// 1 / d to within 2 ulp: three roundings of 2^-23 at most make the estimate
// less than one off, so its floor is off by one at most.
__device__ __forceinline__ int32_t div_est(uint32_t x, uint32_t d, float inv)
{
    int32_t q = (int32_t)((float)x * inv);
    const int32_t r = (int32_t)(x - (uint32_t)q * d);
    if (r < 0) --q;
    if (r >= (int32_t)d) ++q;
    return q;
}
__device__ __forceinline__ float inv_of(int32_t d) { return __fdividef(1.f, (float)d); }

// A run: the units of one (sequence, KV head).
struct Run {
    int32_t s, g;   // sequence, KV head
    int32_t nt;     // units
    int32_t begin;  // id of the first one
};

// Context length of sequence s, read once per CTA in the prologue and clamped
// to the table's reach with the error reported.
__device__ __forceinline__ int32_t load_len(const AttnArgs &a, int s, int32_t *raw_out)
{
    const int32_t raw = a.sync_table ? a.sync_words[s] : ld_prior(a.ctx_lens + s, a.chain >= 2);
    const int32_t cap = a.max_blocks * a.bs;
    *raw_out = raw;
    if (raw < 0 || raw > cap) {
        report(a.err, KV_ERR_DEVICE_BOUNDS);
        return raw < 0 ? 0 : cap;
    }
    return raw;
}

// leading tokens of sequence s (context n) left to the prefix kernel: 0
// outside shared-prefix mode; a value that is not a multiple of 16 in
// [0, n] is reported and clamped
__device__ __forceinline__ int32_t load_skip(const AttnArgs &a, int s, int32_t n)
{
    if (!a.skip) return 0;
    int32_t k = __ldcg(a.skip + s);
    if (k < 0 || k > n || (k % kTile)) {
        report(a.err, KV_ERR_DEVICE_BOUNDS);
        k = k < 0 ? 0 : (k > n ? n : k);
        k -= k % kTile;
    }
    return k;
}

// The CTA's copy of the per-sequence values, after T[0 .. S]: NL[s] = the
// clamped length, with bit 31 set when the stored length was out of range;
// SK[s] = the clamped skip.
__device__ __forceinline__ int32_t seq_len(const int32_t *T, int S, int s) { return T[S + 1 + s] & 0x7fffffff; }
__device__ __forceinline__ bool seq_len_clamped(const int32_t *T, int S, int s) { return T[S + 1 + s] < 0; }
__device__ __forceinline__ int32_t seq_skip(const int32_t *T, int S, int s) { return T[2 * S + 1 + s]; }

// largest s with T[s] <= u; T[s] = first unit of sequence s, T[S] = total,
// so empty sequences (T[s] == T[s+1]) are skipped
__device__ __forceinline__ int find_seq(const int32_t *T, int S, int32_t u)
{
    int lo = 0, hi = S;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (T[mid] <= u) lo = mid; else hi = mid;
    }
    return lo;
}

// units of a run of sequence s
template <int D>
__device__ __forceinline__ int32_t run_units(const int32_t *T, int S, int s)
{
    return (int32_t)((uint32_t)(seq_len(T, S, s) - seq_skip(T, S, s) + kUnit<D> - 1) / (uint32_t)kUnit<D>);
}

// the run that holds unit u
template <int D>
__device__ __forceinline__ Run run_of(const AttnArgs &a, const int32_t *T, int32_t u)
{
    Run r;
    r.s = find_seq(T, a.S, u);
    r.nt = run_units<D>(T, a.S, r.s);
    const int32_t t0 = T[r.s];
    r.g = div_est((uint32_t)(u - t0), (uint32_t)r.nt, inv_of(r.nt));
    r.begin = t0 + r.g * r.nt;
    return r;
}

// the run after r (there is one: the caller has units past r)
template <int D>
__device__ __forceinline__ Run next_run(const AttnArgs &a, const int32_t *T, Run r)
{
    r.begin += r.nt;
    if (++r.g == a.Hkv) {
        r.g = 0;
        do
            ++r.s;
        while (T[r.s + 1] == T[r.s]);  // sequences without units
        r.nt = run_units<D>(T, a.S, r.s);
    }
    return r;
}

// Block table entry idx (flat): this step's value when the table sync is
// fused into the launch and changed that entry, else the table's.
__device__ __forceinline__ int32_t table_entry(const AttnArgs &a, int64_t idx)
{
    if (a.sync_table) {
        const int32_t *pw = a.sync_words + a.sync_nlens;
        for (int j = 0; j < a.sync_npatch; ++j)
            if (pw[2 * j] == idx) return pw[2 * j + 1];
    }
    return ld_prior(a.table + idx, a.chain >= 2);
}

// Pool row of box j of unit u's K tile (TMA y coordinate; V is Hkv*bs rows
// further), kRowBad if the block table names a block outside the pool, or
// kRowNone if the context ends before the box (the table may have no entry).
constexpr int32_t kRowBad = -1, kRowNone = -2;
template <int D>
__device__ __forceinline__ int32_t unit_row(const AttnArgs &a, const int32_t *T, int32_t u, int j)
{
    const Run r = run_of<D>(a, T, u);
    const int32_t tok0 = seq_skip(T, a.S, r.s) + (u - r.begin) * kUnit<D> + j * kTile;
    if (j > 0 && tok0 >= seq_len(T, a.S, r.s)) return kRowNone;
    const int32_t blk = a.bs_shift >= 0 ? tok0 >> a.bs_shift : tok0 / a.bs;
    const int32_t phys = table_entry(a, (int64_t)r.s * a.max_blocks + blk);
    if (phys < 0 || (int64_t)phys + a.pages_per_block > a.pool_pages) return kRowBad;
    return (int32_t)((int64_t)phys * a.rows_per_page + (tok0 - blk * a.bs) + (int64_t)r.g * a.bs);
}

// per-part partial: o[G][D], m[G], l[G], padded to a multiple of 4 floats so
// every record starts 16-byte aligned
template <int D, int G>
__host__ __device__ constexpr uint32_t merge_floats() { return (G * D + 2 * G + 3) / 4 * 4; }

// one more record (m, l, o) of a run into its merged state (M, L, O), for one
// float4 column: base-2 online softmax.  A record without tokens (m = -inf)
// leaves the state as it is.
__device__ __forceinline__ void merge_record(float &M, float &L, float4 &O, float m, float l, const float4 &o)
{
    if (m == -INFINITY) return;
    const float Mn = fmaxf(M, m);
    const float sa = fast_exp2(M - Mn), sb = fast_exp2(m - Mn);
    // spelled out, so that every kernel that merges rounds alike
    L = __fmaf_rn(L, sa, __fmul_rn(l, sb));
    O.x = __fmaf_rn(O.x, sa, __fmul_rn(o.x, sb));
    O.y = __fmaf_rn(O.y, sa, __fmul_rn(o.y, sb));
    O.z = __fmaf_rn(O.z, sa, __fmul_rn(o.z, sb));
    O.w = __fmaf_rn(O.w, sa, __fmul_rn(o.w, sb));
    M = Mn;
}

// The records of one CTA's warps (m = -inf: none) as one state, for one float4
// column: the maximum first, so that the sums wait on no chain of rescales
// (one long sequence 14.2 -> 13.9 us a step, 8 sequences 19.3 -> 19.1, 48
// with 8 query heads a KV head 77.3 -> 76.8, against one record at a time).
// The CTAs (MERGE) and the combine both use it: the same bits.
template <int N>
__device__ __forceinline__ void merge_group(float &M, float &L, float4 &O, const float (&m)[N], const float (&l)[N],
                                            const float4 (&o)[N])
{
    M = m[0];
#pragma unroll
    for (int k = 1; k < N; ++k) M = fmaxf(M, m[k]);
    L = 0.f;
    O = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < N; ++k) {
        if (m[k] == -INFINITY) continue;
        const float e = fast_exp2(m[k] - M);
        L = __fmaf_rn(l[k], e, L);
        O.x = __fmaf_rn(o[k].x, e, O.x);
        O.y = __fmaf_rn(o[k].y, e, O.y);
        O.z = __fmaf_rn(o[k].z, e, O.z);
        O.w = __fmaf_rn(o[k].w, e, O.w);
    }
}

// a merged column's four outputs, bf16(O / L)
__device__ __forceinline__ void store_column(uint16_t *dst, const float4 &O, float L)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(O.x / L, O.y / L);
    __nv_bfloat162 hi = __floats2bfloat162_rn(O.z / L, O.w / L);
    *reinterpret_cast<uint2 *>(dst) = make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
}

// The pool rows of a unit's boxes.
template <int D>
struct UnitRows {
    int32_t y[kSub<D>];
};
template <int D>
__device__ __forceinline__ UnitRows<D> rows_of(const AttnArgs &a, const int32_t *T, const int32_t *rows, int32_t cu0,
                                               int32_t u)
{
    UnitRows<D> r;
    const int32_t k = (u - cu0) * kSub<D>;
#pragma unroll
    for (int j = 0; j < kSub<D>; ++j) r.y[j] = k + j < a.rows_cap ? rows[k + j] : unit_row<D>(a, T, u, j);
    return r;
}

// Load K (which = 0) or V (which = 1) of a unit into this warp's stage;
// completes on `bar`.  The whole warp, with one lane elected: a single
// diverged lane passes the operands to uniform registers one by one, in every
// unit's chain (one long sequence 13.85 -> 13.54 us a step, 1024 long contexts
// 698.4 -> 695.1, the 64-sequence layer 67.9 -> 67.7).
template <int D>
__device__ __forceinline__ void issue_half(const CUtensorMap *tmap, const AttnArgs &a, const UnitRows<D> &r, int which,
                                           uint32_t dst, uint32_t bar, uint64_t policy, uint32_t elected)
{
    constexpr int HALVES = D / 64, SUB = kSub<D>;
    uint32_t boxes = 0;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
        bad |= r.y[j] == kRowBad;
        boxes += r.y[j] >= 0 ? 1u : 0u;
    }
    if (bad) {
        if (elected) {
            report(a.err, KV_ERR_DEVICE_BOUNDS);
            mbar_arrive(bar);  // complete the phase without data
        }
        __syncwarp();
        return;
    }
    mbar_arrive_expect_tx_elected(bar, boxes * HALVES * kHalfBytes, elected);
#pragma unroll
    for (int j = 0; j < SUB; ++j)
        if (SUB == 1 || r.y[j] >= 0)
#pragma unroll
            for (int h = 0; h < HALVES; ++h)  // box (j, h): with SUB > 1, HALVES is 1
                tma_load_2d_elected(dst + (j + h) * kHalfBytes, tmap, h * 64, r.y[j] + which * a.Hkv * a.bs, bar,
                                    policy, elected);
}

template <int D, int G, class Comp, int MODE>
__global__ void __launch_bounds__(kThreads, Comp::kMinBlocks)
paged_attn_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ AttnArgs a)
{
    constexpr bool MERGE = MODE != kRecWarps, BY_PART = MODE == kRecCtasByPart;
    constexpr int HALVES = D / 64;
    constexpr int UNIT = kUnit<D>, SUB = kSub<D>;
    static_assert(HALVES == 1 || SUB == 1, "a unit's boxes follow each other in shared memory");
    constexpr uint32_t TILE_BYTES = HALVES * SUB * kHalfBytes;
    constexpr uint32_t STAGE_BYTES = 2 * TILE_BYTES;
    constexpr uint32_t MF = merge_floats<D, G>();
    extern __shared__ uint8_t smem_raw[];
    // stages need 1024-byte alignment for the 128-byte swizzle pattern
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr uint32_t QB = G * D * 2, AB = 2 * D * 2;  // q rows of a run; its new K and V rows
    const int NW = a.nwarps, NT = NW * 32;  // warps (parts) of this CTA
    uint8_t *stages = smem;                                                              // [NW][kStages][STAGE]
    uint8_t *qbufs = stages + (size_t)NW * kStages * STAGE_BYTES;                        // [NW][QB]
    uint8_t *abufs = qbufs + (size_t)NW * QB;                                            // [NW][AB]
    uint8_t *mbufs = abufs + (size_t)NW * AB;                                            // [NW] records, with MERGE
    int4 *chains = reinterpret_cast<int4 *>(mbufs + (MERGE ? (size_t)NW * MF * 4 : 0));  // [NW]
    uint64_t *bars = reinterpret_cast<uint64_t *>(chains + (MERGE ? NW : 0));    // K[w][st], V[w][st]
    int32_t *misc = reinterpret_cast<int32_t *>(bars + 2 * NW * kStages);               // [16] scratch
    int32_t *T = misc + 16;                                                              // [S + 1]
    int32_t *NL = T + a.S + 1;                                                           // [S]
    int32_t *SK = NL + a.S;                                                              // [S]
    int32_t *rows = SK + a.S;                                                            // [rows_cap]

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // the same in the warp's lanes, for the compiler too
    const int S = a.S, Hkv = a.Hkv, Hq = a.Hkv * G;

    if (tid == 0) {
        for (int i = 0; i < 2 * NW * kStages; ++i) mbar_init(smem_u32(&bars[i]), 1);
        fence_mbar_init();
    }
    if (tid == 32) prefetch_tensormap(&tmap);
    // Launched as a programmatic dependent: everything above touches only
    // this CTA.  Alone (chain 0), release the next grid and wait here for
    // the grid before (lengths, table, pool writes).  A chained grid (chain
    // 2: the decode kernel beside the shared-prefix kernel, or the second
    // and later batches of paged_decode_attn_multi) follows a grid that
    // released it only after its own wait had seen every earlier grid
    // complete; it does not wait for that grid here, so the two run side by
    // side (the later one's CTAs take the SMs the earlier one frees), and
    // waits for it at the exit (`chained`; all but CTAs without units, and
    // CTA 0 always), so that a combine after it sees every chained grid's
    // records.  Data from earlier grids is then
    // read through L2 (ld_prior).  The first grid of a chain (chain 1)
    // waits before it releases the next.  With the lengths carried in the
    // parameters (fused table sync) and no shared prefix, the first prologue
    // below reads nothing that another grid writes and writes only shared
    // memory, so a grid alone runs it before its wait, beside the grid
    // before it (`early`).  After a combine (chain 3) nothing before that
    // combine is still running: the kernel reads and writes the table, the
    // lengths and the pool at once, and each thread waits for the combine
    // (`ready`) before it first writes the output or the workspace.  Beside
    // the prefix kernel of a step that overlaps the previous step's
    // shared-prefix combine (chain 4), the plan kernel's flags take the place
    // of those waits: the first before the lengths, skips and table are read,
    // the second before the first write of the output or the workspace.
    const bool early = a.sync_table != nullptr && a.skip == nullptr && (a.chain == 0 || a.chain == 3);
    if (a.chain != 1) grid_launch_dependents();
    if (a.chain <= 1 && !early) grid_dependency_wait();
    if (a.chain == 1) grid_launch_dependents();
    const bool chained = a.chain >= 2;
    bool ready = a.chain != 3 && a.chain != 4;  // the output and the workspace may be written
    auto make_ready = [&]() {
        if (!ready) {
            if (a.chain == 4)
                wait_flag(a.flags + 1, a.epoch, a.err);
            else
                grid_dependency_wait();
            ready = true;
        }
    };
    if (a.chain == 4) {
        if (tid == 0) wait_flag(a.flags, a.epoch, a.err);
        __syncthreads();
    }
    auto write_sync = [&]() {
        // fused table sync: the grids before have completed (the wait
        // before this), and no CTA of this grid reads what is written here
        const int stride = a.P * NT, i0 = (int)blockIdx.x * NT + tid;
        for (int i = i0; i < a.sync_nlens; i += stride) a.sync_lens[i] = a.sync_words[i];
        const int32_t *pw = a.sync_words + a.sync_nlens;
        for (int j = i0; j < a.sync_npatch; j += stride) a.sync_table[pw[2 * j]] = pw[2 * j + 1];
    };
    if (a.sync_table && !early) write_sync();

    // ---- prologue 1: T[s] = first unit of sequence s ----
    {
        const int per = (S + NT - 1) / NT;
        const int lo = min(S, tid * per), hi = min(S, lo + per);
        int32_t local = 0;
        for (int s = lo; s < hi; ++s) {
            int32_t raw;
            const int32_t n = load_len(a, s, &raw);
            const int32_t k = load_skip(a, s, n);
            NL[s] = n | (raw != n ? (int32_t)0x80000000 : 0);
            SK[s] = k;
            const int32_t ne = n - k;
            local += ((ne + UNIT - 1) / UNIT) * Hkv;
        }
        int32_t incl = local;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        if (lane == 31) misc[warp] = incl;
        __syncthreads();
        int32_t sums = lane < NW ? misc[lane] : 0;  // of the warps up to this lane's
#pragma unroll
        for (int off = 1; off < kWarps; off <<= 1) {
            const int32_t v = __shfl_up_sync(0xffffffffu, sums, off);
            if (lane >= off) sums += v;
        }
        const int32_t base = __shfl_sync(0xffffffffu, sums, warp > 0 ? warp - 1 : 0);
        const int32_t tot = __shfl_sync(0xffffffffu, sums, kWarps - 1);
        int32_t run = (warp > 0 ? base : 0) + incl - local;
        for (int s = lo; s < hi; ++s) {  // this thread's own NL / SK entries
            T[s] = run;
            run += run_units<D>(T, S, s) * Hkv;
        }
        if (tid == 0) T[S] = tot;
        if (early) {
            if (a.chain == 0) grid_dependency_wait();
            write_sync();
        }
        for (int s = lo; s < hi; ++s) {  // sequences with no tile: writes after any wait
            const int32_t n = NL[s] & 0x7fffffff, ne = n - SK[s];
            if (ne != 0 || (s % a.P) != (int)blockIdx.x) continue;
            make_ready();
            // the fused append needs the new token outside a shared prefix
            if (a.skip && a.k_new && n > 0) report(a.err, KV_ERR_DEVICE_BOUNDS);
            // an empty context has no softmax: its output is defined as
            // zero; a sequence whose whole context is a shared prefix gets
            // its output from the prefix records alone
            if (n == 0)
                for (int i = 0; i < Hq * D; ++i) a.out[(int64_t)s * Hq * D + i] = 0;
            if (!BY_PART)
                for (int g = 0; g < Hkv; ++g) a.ws_run[(int64_t)s * Hkv + g] = make_int2(0, 0);
        }
        __syncthreads();
    }

    // The W units are cut into NC equal ranges, one per CTA, and a CTA's range
    // into equal ranges, one per warp: a warp gets at least a.min_units units
    // when the batch is small (fewer partials to write and merge; enough warps
    // still stream to fill HBM).  The parts are the warps' ranges, numbered
    // blockIdx * NW + warp, or with MERGE the CTAs' ranges.  Every part is
    // non-empty, and a run's contributors are exactly the parts from its
    // first unit's to its last unit's.
    const int32_t W = T[S];
    const int32_t fine = a.min_units > 1 ? W / (NW * a.min_units) : (W + NW - 1) / NW;
    const int32_t NC = W > 0 ? min(max(fine, 1), a.P) : 0;
    const int32_t bid = (int32_t)blockIdx.x;
    auto no_part = [&]() {  // the CTA (without MERGE: this warp) has no units
        if (BY_PART && tid == 0) {
            make_ready();
            a.ws_run[bid] = make_int2(-1, -1);
        }
        // CTA 0 waits whatever its share, so this grid's completion means the
        // one before's.  The others leave: waiting, they would hold SM slots
        // that a third co-located batch needs (2, 2 and 2 sequences with 8, 8 and
        // 32 KV heads: 28.4 us a step with them waiting, 24.8 without).
        if (chained && bid == 0) grid_dependency_wait();
    };
    if (bid >= NC) return no_part();
    // first unit of CTA i: i * W / NC, with W = wq * NC + wr
    const int32_t wq = (int32_t)((uint32_t)W / (uint32_t)NC), wr = W - wq * NC;
    const float nc_inv = inv_of(NC);
    auto cta_begin = [&](int32_t i) {
        return NC < 32768 ? i * wq + div_est((uint32_t)i * (uint32_t)wr, (uint32_t)NC, nc_inv)
                          : (int32_t)((int64_t)i * W / NC);
    };
    const int32_t cu0 = cta_begin(bid), cu1 = cta_begin(bid + 1), nu = cu1 - cu0;  // this CTA's units
    const int32_t nw = min(NW, nu);  // warps with units (all but where W < NW)
    if (!MERGE && warp >= nw) return no_part();  // no CTA-wide barrier below this point without MERGE
    // this warp's units
    const int32_t nq = (int32_t)((uint32_t)nu / (uint32_t)nw), nr = nu - nq * nw;
    const float nw_inv = inv_of(nw);
    auto warp_begin = [&](int w) {  // w * nu / nw
        return w < nw ? cu0 + w * nq + div_est((uint32_t)(w * nr), (uint32_t)nw, nw_inv) : cu1;
    };
    const int32_t u0 = warp_begin(warp), u1 = warp_begin(warp + 1);
    const int32_t part = MERGE ? bid : bid * NW + warp;
    const int32_t g0 = MERGE ? cu0 : u0, g1 = MERGE ? cu1 : u1;  // this part's units

    // ---- prologue 2: resolve the block table for this warp's units while the
    // memory system is idle (later lookups would queue behind the TMA stream)
    {
        const int32_t k0 = (u0 - cu0) * SUB, k1 = min((u1 - cu0) * SUB, a.rows_cap);
        for (int32_t k = k0 + lane; k < k1; k += 32) rows[k] = unit_row<D>(a, T, cu0 + k / SUB, k % SUB);
        __syncwarp();
    }
    float *mbuf = reinterpret_cast<float *>(mbufs) + (size_t)warp * MF;
    if (MERGE && lane == 0) chains[warp].x = -1;

    const uint64_t policy = l2_policy_evict_first();
    // stage st of this warp: its K and V tiles and their barriers
    uint8_t *wstage = stages + (size_t)warp * kStages * STAGE_BYTES;
    auto k_of = [&](int st) { return wstage + (size_t)st * STAGE_BYTES; };
    auto bk_of = [&](int st) { return smem_u32(&bars[warp * kStages + st]); };
    auto bv_of = [&](int st) { return smem_u32(&bars[(NW + warp) * kStages + st]); };

    const uint32_t el = elect_one();
    for (int st = 0; st < kStages && u0 + st < u1; ++st) {
        const UnitRows<D> ur = rows_of<D>(a, T, rows, cu0, u0 + st);
        issue_half<D>(&tmap, a, ur, 0, smem_u32(k_of(st)), bk_of(st), policy, el);
        issue_half<D>(&tmap, a, ur, 1, smem_u32(k_of(st) + TILE_BYTES), bv_of(st), policy, el);
    }
    // A run's q rows and, for the run's last tile, its new K/V rows are staged
    // in this warp's shared buffers by cp.async one piece ahead, so that no
    // piece start or append waits on a dependent global load.
    uint8_t *qb = qbufs + (size_t)warp * QB;
    uint8_t *ab = abufs + (size_t)warp * AB;
    const uint32_t qb_addr = smem_u32(qb), ab_addr = smem_u32(ab);
    auto stage_q = [&](const Run &r) {
        const uint16_t *src = a.q + ((int64_t)r.s * Hq + (int64_t)r.g * G) * D;
        for (uint32_t c = lane; c < QB / 16; c += 32) cp_async16(qb_addr + c * 16, src + c * 8);
    };
    Run run{};
    if (!MERGE || u0 < u1) {
        run = run_of<D>(a, T, u0);
        stage_q(run);
        cp_async_commit();
    }

    bool dead = false;
    uint32_t consumed = 0;
    int2 cut = make_int2(-1, -1);  // BY_PART: the part's entry, as far as this warp holds its ends
    int32_t u = u0;
    while (u < u1) {
        const int32_t n = seq_len(T, S, run.s), skip = seq_skip(T, S, run.s);
        const int32_t run_end = run.begin + run.nt, pe = run_end < u1 ? run_end : u1;  // the piece: [u, pe)
        cp_async_wait_all();  // this piece's q rows
        __syncwarp();
        Comp comp;
        comp.begin(reinterpret_cast<const uint16_t *>(qb), a.qk_scale, lane);
        __syncwarp();  // every lane holds its q fragments: the buffer may be refilled
        // fused append: the run's last tile holds position n-1, whose K/V row
        // is this step's new token; this warp alone reads that tile
        const bool app_run = a.k_new != nullptr && pe == run_end && !seq_len_clamped(T, S, run.s);
        if (app_run && lane < AB / 16) {
            const int which = lane / (D / 8), c = lane % (D / 8);
            cp_async16(ab_addr + lane * 16, (which ? a.v_new : a.k_new) + ((int64_t)run.s * Hkv + run.g) * D + c * 8);
        }
        Run next = run;
        if (pe < u1) {  // the next piece's q rows
            next = next_run<D>(a, T, run);
            stage_q(next);
        }
        cp_async_commit();
        for (int32_t uu = u; uu < pe; ++uu) {
            const int st = (int)(consumed % kStages);
            const uint32_t par = (consumed / kStages) & 1u;
            uint8_t *Ks = k_of(st);
            uint8_t *Vs = Ks + TILE_BYTES;
            const uint32_t bk = bk_of(st), bv = bv_of(st);
            const int nvalid = min(UNIT, n - skip - (uu - run.begin) * UNIT);
            const bool more = uu + kStages < u1;  // the unit this stage takes next
            const bool app = app_run && uu == run_end - 1;
            const int arow = (n - 1 - skip) % UNIT;
            UnitRows<D> ur;
            if (more) ur = rows_of<D>(a, T, rows, cu0, uu + kStages);
            wait_phase(bk, par, a.err, dead);
            if (app) {
                cp_async_wait_all();  // the new K/V rows
                __syncwarp();
                if (lane < D / 8)
                    *reinterpret_cast<uint4 *>(Ks + swz(arow, lane)) = *reinterpret_cast<const uint4 *>(ab + lane * 16);
                __syncwarp();
            }
            comp.scores(Ks, nvalid);
            // K is asked for again as soon as its scores are done, before the
            // softmax, from rows read before the wait: 1024 long contexts 704.3
            // -> 702.5 us, one long sequence 14.7 -> 14.3.  The K stage is
            // refilled by TMA next: order the warp's generic
            // shared-memory reads before the async-proxy write
            fence_proxy_async_smem();
            __syncwarp();
            if (more) issue_half<D>(&tmap, a, ur, 0, smem_u32(Ks), bk, policy, el);
            comp.softmax();
            wait_phase(bv, par, a.err, dead);
            if (app) {
                if (lane < D / 8)
                    *reinterpret_cast<uint4 *>(Vs + swz(arow, lane)) =
                        *reinterpret_cast<const uint4 *>(ab + D * 2 + lane * 16);
                __syncwarp();
            }
            comp.pv(Vs);
            if (app) {
                // store the new row into the pool: this warp's own TMA reads of
                // the tile have completed, and no other unit covers that row
                const int j = arow / kTile;  // the box that holds the row
                const int32_t k = (uu - cu0) * SUB + j;
                const int32_t y = k < a.rows_cap ? rows[k] : unit_row<D>(a, T, uu, j);
                if (y >= 0 && lane < AB / 16) {
                    const int which = lane / (D / 8), c = lane % (D / 8);
                    const int64_t row = (int64_t)y + arow % kTile + (int64_t)which * Hkv * a.bs;
                    *reinterpret_cast<uint4 *>(a.pool + row * D + c * 8) =
                        *reinterpret_cast<const uint4 *>(ab + lane * 16);
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (more) issue_half<D>(&tmap, a, ur, 1, smem_u32(Vs), bv, policy, el);
            ++consumed;
        }

        // ---- end of a piece: the output, or this part's partial ----
        const int32_t r = run.s * Hkv + run.g;
        // a run whose prefix lives in prefix records always leaves a partial
        const bool split = run.begin < g0 || run_end > g1 || skip > 0;
        // the run's first part and its last one tell the combine where its
        // records begin and end
        const bool first = run.begin >= g0, last = run_end <= g1;
        const int end = split ? part + 1 : part;
        if (BY_PART && pe == g1 && first && !last) cut.x = r;
        if (BY_PART && u == g0 && last && !first) cut.y = r;
        uint16_t *orow = a.out + ((int64_t)run.s * Hq + (int64_t)run.g * G) * D;
        float *slot = a.ws_part + ((int64_t)r + part) * MF;
        // (MERGE) the part's share of the run; it may go on over several warps
        const int32_t lo = run.begin > g0 ? run.begin : g0, hi = run_end < g1 ? run_end : g1;
        if (!MERGE || (u == lo && pe == hi)) {
            make_ready();
            comp.store(orow, slot, split, lane);
            if (!BY_PART && lane == 0) {
                if (first) a.ws_run[r].x = part;
                if (last) a.ws_run[r].y = end;
            }
        } else if (u != lo) {  // goes on from an earlier warp, whose chain merges it
            comp.store(nullptr, mbuf, true, lane);
        } else {  // goes on in the next warp: the last piece here, so the stage is free
            comp.store(nullptr, reinterpret_cast<float *>(wstage), true, lane);
            int e = warp;
            while (warp_begin(e + 1) < hi) ++e;
            if (lane == 0)
                chains[warp] = make_int4(r, e - warp, (first ? 1 : 0) | (last ? 2 : 0), split ? 1 : 0);
        }
        u = pe;
        run = next;
    }
    if (BY_PART && lane == 0 && u0 < u1) {
        make_ready();
        if (u1 == g1) a.ws_run[part].x = cut.x;
        if (u0 == g0) a.ws_run[part].y = cut.y;
    }
    if constexpr (MERGE) {
        __syncthreads();
        // CTA-level merge: chain w is the run whose share of this CTA starts in
        // warp w and goes on through warp w + chains[w].y; its states (base-2
        // online softmax) are merged in warp order, one thread per float4
        // column, into the output (a run inside this CTA) or one record
        constexpr int NC = G * D / 4;
        for (int i = tid; i < NW * NC; i += NT) {
            const int w = i / NC, c = i % NC, h = c * 4 / D;
            const int4 ch = chains[w];
            if (ch.x < 0) continue;
            float mv[kWarps], lv[kWarps];
            float4 ov[kWarps];
#pragma unroll
            for (int k = 0; k < kWarps; ++k) {
                mv[k] = -INFINITY;
                if (k <= ch.y) {
                    const float *rec = k == 0
                                           ? reinterpret_cast<const float *>(stages + (size_t)w * kStages * STAGE_BYTES)
                                           : reinterpret_cast<const float *>(mbufs) + (size_t)(w + k) * MF;
                    mv[k] = rec[G * D + h];
                    lv[k] = rec[G * D + G + h];
                    ov[k] = *reinterpret_cast<const float4 *>(rec + c * 4);
                }
            }
            float M, L;
            float4 O;
            merge_group(M, L, O, mv, lv, ov);
            make_ready();
            if (ch.w == 0) {
                store_column(a.out + (int64_t)ch.x * (G * D) + c * 4, O, L);
            } else {
                float *slot = a.ws_part + ((int64_t)ch.x + part) * MF;
                *reinterpret_cast<float4 *>(slot + c * 4) = O;
                if (c * 4 % D == 0) {
                    slot[G * D + h] = M;
                    slot[G * D + G + h] = L;
                }
            }
            if (c == 0 && (ch.z & 1) && !BY_PART) a.ws_run[ch.x].x = part;
            if (c == 0 && (ch.z & 2) && !BY_PART) a.ws_run[ch.x].y = part + ch.w;
        }
    }
    if (chained) grid_dependency_wait();
}

// ------------------------------------------------------------ combine ---
// Split-K combine: for each (sequence, KV head) run cut by part boundaries
// (or with a shared prefix), merge its records (m_k, l_k, o_k) in order:
//     M = max_k m_k,  out = sum_k 2^(m_k - M) o_k / sum_k 2^(m_k - M) l_k
// (base-2 online-softmax state).  CS CTAs per run, each covering a CS-th of its
// G*D output columns: NG thread groups of G*D/(4*CPT*CS) threads (CPT float4
// columns each) take records k = grp, grp + NG, ..., then merge their states
// by halves in a fixed order, so the result depends only on the run's shape.
// (Merged one after another by the first group, 29 groups made a step of four
// short sequences 3 µs longer: 15.4 µs against 12.4.)  Runs finished inside
// the attention kernel return at once; with very many runs (kRecCtasByPart) a
// CTA per part takes the run that starts there and goes on.
struct CombineArgs {
    uint16_t *out;
    const int2 *ws_run;    // as in AttnArgs
    const float *ws_part;
    int32_t S;
    int32_t Hkv;
    const int32_t *skip;   // cascade mode: sequences with skip > 0 also merge
    const float *ws_pre;   // KS prefix records [k][S][Hkv], ahead of their parts
    int32_t KS;
};

constexpr int kCombineMaxThreads = 1024;
constexpr int kCombineBatch = 8;  // records each thread loads per round trip, with few runs

// CTAs per run (CS) and thread groups per combine CTA.
//
// Where each run has a CTA (CS = 1; six loads in flight per thread, which 64
// registers hold): enough groups for about 8 records per thread, up to 1024 threads,
// and at least 128 threads (one group when a run's output has 128 float4
// columns or more).  Small CTAs leave room on the SMs for the next step's
// decode CTAs, which start as the combine's CTAs finish: on the
// Llama-3-8B-shaped layer (64 sequences, 32 q / 8 KV heads) 128-thread CTAs
// took 54.5-54.9 µs per step against 55.1-55.4 with 256 (six same-box
// pairs), at a cost of about 1 µs in 296 for three co-located models, whose
// heavy-tailed runs take more round trips with one group.
//
// Few runs leave most SMs idle while one SM fetches a run's records (one
// sequence of 8193 tokens: 8 runs of 128 records, 2 MB through 8 SMs, 8.9 µs
// of a 22 µs step).  Up to kSlicedCtas CTAs an SM, a run's columns are spread
// over 8 or 4 CTAs, each with groups for about 8 records a thread, at most
// 16.  That step: 20.7 µs with CS = 1 and 15.8 with CS = 8 (both with the
// groups merged by halves, below).  The line, on 64 runs of 6 records (8
// sequences, 40 q / 8 KV heads, CTA-level parts): CS = 8 19.9 µs, CS = 1 20.2.
constexpr int kSlicedCtas = 4;
template <int D, int G, int CS>
inline int combine_groups(double records_per_run)
{
    constexpr int NC = G * D / 4 / CS;
    constexpr int floor_threads = CS == 1 ? 128 : 64;
    const int base = NC >= floor_threads ? 1 : floor_threads / NC;
    const int most = CS == 1 ? kCombineMaxThreads / NC : std::max(base, std::min(16, kCombineMaxThreads / 2 / NC));
    int want = (int)(records_per_run / 8.0 + 0.999);
    return want < base ? base : (want > most ? most : want);
}

// Columns per thread CPT: 1, or 2 for the one-group form of shared-prefix
// mode.  There every member run is one CTA, and the agent chains have 2048
// of them: at one column a thread (128 threads a run) and 64 registers only
// eight CTAs fit an SM and the last 850 runs wait for a second wave; at two
// columns a thread (64 threads a run, registers held to 64, no shared
// memory) sixteen fit and one wave covers 2432 runs.  Each column merges the
// same records in the same order either way, so the bits do not change.
template <int D, int G, int CPT, int CS = 1>
struct CombineShape {
    static constexpr int NC = G * D / 4 / CS;  // float4 columns of a CTA: a CS-th of a run's output
    static constexpr int NCT = NC / CPT;   // threads of a group
    static constexpr int MAX_THREADS = CPT > 1 ? NCT : CS == 1 ? kCombineMaxThreads : kCombineMaxThreads / 2;
    static constexpr int MIN_CTAS = CPT == 1 ? 1 : 28 / ((NCT + 31) / 32);  // 28 warps an SM: 72 registers
    static constexpr int BATCH = CPT > 1 ? 4 : CS == 1 ? 6 : kCombineBatch;
};

// shared memory of a CTA of `threads` threads: the groups' states for the
// merge (none with one group)
template <int D, int G, int CPT, int CS>
inline size_t combine_smem_bytes(int threads)
{
    return threads > CombineShape<D, G, CPT, CS>::NCT ? (size_t)threads * CPT * (2 * sizeof(float) + sizeof(float4)) : 0;
}

// The run of this CTA (-1: none) and the parts of its records, [at.x, at.y).
template <int MODE>
__device__ __forceinline__ int combine_run_of(const CombineArgs &c, int2 &at)
{
    const int b = blockIdx.x;
    at = c.ws_run[b];
    if constexpr (MODE != kRecCtasByPart) return b;
    const int r = at.x;
    at = make_int2(b, b);
    // The run ends in the next part whose entry names it.  Each warp looks for
    // itself, a part a lane; a CTA's threads need not be whole warps (80 of
    // them with five query heads of 64), so the last warp may have fewer lanes.
    const int ln = (int)threadIdx.x & 31, parts = gridDim.x;
    const int lanes = min(32, (int)blockDim.x - ((int)threadIdx.x & ~31));
    const unsigned mask = 0xffffffffu >> (32 - lanes);
    if (r >= 0)
        for (int q = b + 1; q < parts && at.y == b; q += lanes) {
            const unsigned hit = __ballot_sync(mask, q + ln < parts && c.ws_run[q + ln].y == r);
            if (hit) at.y = q + __ffs((int)hit);
        }
    return r;
}

template <int D, int G, int CPT, int CS, int MODE>
__global__ void __launch_bounds__(CombineShape<D, G, CPT, CS>::MAX_THREADS, CombineShape<D, G, CPT, CS>::MIN_CTAS)
combine_kernel(const __grid_constant__ CombineArgs c)
{
    using Sh = CombineShape<D, G, CPT, CS>;
    constexpr uint32_t MF = merge_floats<D, G>();
    constexpr int NCT = Sh::NCT;
    constexpr int B = Sh::BATCH;
    static_assert(Sh::NC % CPT == 0 && NCT <= kCombineMaxThreads, "whole columns per thread");
    const int NG = (int)blockDim.x / NCT;  // groups of NCT threads
    extern __shared__ float4 s_dyn[];      // [CPT][blockDim] O, then M, then L (when NG > 1)
    grid_dependency_wait();  // the attention grid's partials and run table
    // Release the next grid only now, when every grid before this one has
    // completed: a decode grid that follows without a wait of its own (step
    // overlap) relies on it, and until its own wait writes nothing that this
    // grid reads or writes.
    grid_launch_dependents();
    int2 at;
    const int r = combine_run_of<MODE>(c, at);
    if (MODE == kRecCtasByPart && r < 0) return;  // no run starts in this part and goes on
    const int2 info = at;
    const int s = r / c.Hkv, g = r % c.Hkv;
    const int npre = (c.skip != nullptr && c.skip[s] > 0) ? c.KS : 0;
    const int cnt = info.y - info.x + npre;
    if (cnt == 0) return;  // finished inside the attention kernel (or empty)
    const float *base = c.ws_part + ((int64_t)r + info.x) * MF;
    uint16_t *orow = c.out + ((int64_t)s * c.Hkv * G + (int64_t)g * G) * D;
    const int tid = threadIdx.x;
    const int grp = tid / NCT;
    int col[CPT], h[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        col[j] = (int)blockIdx.y * Sh::NC + tid % NCT + j * NCT;
        h[j] = (col[j] * 4) / D;
    }
    // online merge of this group's records per column: M running max, L and
    // O relative to M; records k = grp, grp + NG, ... are loaded B at a time
    float M[CPT], L[CPT];
    float4 O[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        M[j] = -INFINITY;
        L[j] = 0.f;
        O[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // record k: prefix record k, or, past those, the suffix's (r = s * Hkv + g)
    auto record = [&](int k) {
        return k < npre ? c.ws_pre + ((int64_t)k * (int)gridDim.x + r) * MF : base + (int64_t)(k - npre) * MF;
    };
    if constexpr (MODE != kRecWarps) {
        for (int k0 = grp; k0 < cnt; k0 += NG * B) {
            float mv[B][CPT], lv[B][CPT];
            float4 ov[B][CPT];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = k0 + b * NG;
#pragma unroll
                for (int j = 0; j < CPT; ++j) mv[b][j] = -INFINITY;
                if (k < cnt) {
                    const float *sl = record(k);
#pragma unroll
                    for (int j = 0; j < CPT; ++j) {
                        mv[b][j] = sl[G * D + h[j]];
                        lv[b][j] = sl[G * D + G + h[j]];
                        ov[b][j] = *reinterpret_cast<const float4 *>(sl + col[j] * 4);
                    }
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int j = 0; j < CPT; ++j) merge_record(M[j], L[j], O[j], mv[b][j], lv[b][j], ov[b][j]);
        }
    } else {
        // a record per warp: those of a CTA are merged first, as the CTA itself
        // does when it merges them (MERGE), so that both ways give the same bits
        static_assert(CPT == 1, "no shared prefix: its decode CTAs have kWarps warps");
        constexpr int CW = kPlainWarps;
        const int first = info.x;
        for (int b0 = (first / CW + grp) * CW; b0 < info.y; b0 += NG * CW) {
            float mv[CW], lv[CW];
            float4 ov[CW];
#pragma unroll
            for (int b = 0; b < CW; ++b) {
                const int p = b0 + b;
                mv[b] = -INFINITY;
                if (p >= first && p < info.y) {
                    const float *sl = base + (int64_t)(p - first) * MF;
                    mv[b] = sl[G * D + h[0]];
                    lv[b] = sl[G * D + G + h[0]];
                    ov[b] = *reinterpret_cast<const float4 *>(sl + col[0] * 4);
                }
            }
            float Mc, Lc;
            float4 Oc;
            merge_group(Mc, Lc, Oc, mv, lv, ov);
            merge_record(M[0], L[0], O[0], Mc, Lc, Oc);
        }
    }
    if (NG > 1) {
        const int nt = (int)blockDim.x;
        float4 *s_O = s_dyn;
        float *s_M = reinterpret_cast<float *>(s_dyn + CPT * nt);
        float *s_L = s_M + CPT * nt;
        // the first `to` groups take in the others, half of them at a time
        // while there are more than four (a barrier a round costs more than
        // merging three states)
        for (int n = NG; n > 1;) {
            const int to = n <= 4 ? 1 : (n + 1) / 2;
            if (grp >= to && grp < n)
#pragma unroll
                for (int j = 0; j < CPT; ++j) {
                    s_M[j * nt + tid] = M[j];
                    s_L[j * nt + tid] = L[j];
                    s_O[j * nt + tid] = O[j];
                }
            __syncthreads();
            if (grp < to)
                for (int q = to; grp + q < n; q += to)
#pragma unroll
                    for (int j = 0; j < CPT; ++j) {
                        const int i = j * nt + tid + q * NCT;
                        merge_record(M[j], L[j], O[j], s_M[i], s_L[i], s_O[i]);
                    }
            n = to;
        }
        if (grp != 0) return;
    }
#pragma unroll
    for (int j = 0; j < CPT; ++j) store_column(orow + col[j] * 4, O[j], L[j]);
}

// host helpers ---------------------------------------------------------------
constexpr int kRowsCap = 2048;

// units that the batch's table has room for
inline int64_t table_units(const AttnArgs &a, int D)
{
    const int unit = D == 64 ? kUnit<64> : kUnit<128>;
    return (int64_t)a.S * a.Hkv * (((int64_t)a.max_blocks * a.bs + unit - 1) / unit);
}
// fewer than kMergeUnits units a warp (by the table's width)
inline bool small_batch(const AttnArgs &a, int D, int P, int nwarps)
{
    return table_units(a, D) < (int64_t)kMergeUnits * P * nwarps;
}

// shared memory of a decode CTA; with boxes = 1, what it would be with a unit
// of a box (the S that a call may have, see attn_run)
template <int D, int G>
inline size_t attn_smem_bytes(int S, int rows_cap, int nwarps, bool merge, int boxes = kSub<D>)
{
    const size_t stage = 2ull * (D / 64) * boxes * kHalfBytes;
    // per warp: q rows, new K/V rows; a record, its chain
    const size_t bufs = (size_t)G * D * 2 + 2 * D * 2 + (merge ? merge_floats<D, G>() * 4 + 16 : 0);
    return 1024 + (size_t)nwarps * (kStages * stage + bufs) + (2 * nwarps * kStages) * 8 + 64 + (size_t)(3 * S + 1) * 4 +
           (size_t)rows_cap * 4;
}

// partial records: one per (run, part) pair that a run can touch (parts:
// at most kWarps per CTA)
inline size_t attn_partial_slots(int S, int Hkv, int P) { return (size_t)S * Hkv + (size_t)P * kWarps; }

}  // namespace kvp
