// cascade_impl.cuh -- shared-prefix ("cascade") attention for sequences whose
// block tables start with the same physical blocks.
//
// Sequences that share a prefix by reference (agent stages building on one
// system prompt, §III-B / §III-C) hold identical K/V for its tokens, so the
// prefix's contribution to every sharer's decode query is one dense
// contraction per KV head: all sharers' query heads of that KV head form the
// rows, the prefix tokens the columns.  The prefix K/V is then read once per
// (row tile, key split) from L2 instead of once per sharer, and the work runs
// on the fifth-generation tensor cores as a small flash-attention forward:
//   S = Q K^T     tcgen05.mma, M = 128 query rows, N = 128 keys, fp32 in TMEM
//   softmax       one thread per row, S read from TMEM, base 2, lazy rescale
//   O += P V      tcgen05.mma, P (bf16) from TMEM, V from shared memory, O in TMEM
// with 128-key K/V tiles streamed by TMA through a 2-stage ring.  Beside the
// suffix stream, which keeps HBM's queues full, a tile's loads take several
// microseconds, longer than the tensor work on the tile before: so K and V of
// a stage are released and reloaded apart (K as soon as the tile's scores are
// done), and the producer asks L2 for the tiles kPreAhead further on.  With
// 4096-token prefixes of 3 groups (24 CTAs) beside 190 suffixes the step took
// 135 us with one barrier a stage and no requests ahead (4.5 us a tile, 2.7
// alone on the GPU) and 115 with both and the record stores of the epilogue;
// 2 or 8 tiles ahead instead of 4: 116 and 116.  The
// softmax writes P (bf16) back over S in TMEM, and the P.V MMA reads its A
// operand from there, so P never touches shared memory.  A CTA holds two Q
// tiles that share every K/V tile: while one tile's four warps run the
// softmax, the tensor core works on the other tile.  One warp issues the
// MMAs, two the TMA loads (K's and V's), one thread owns each row.
//
// What paced it (SM clocks of one CTA, 128 members of two 8192-token prefixes,
// cycles per key tile of both Q tiles, 4450 in all):
// - the MMA issue, 70-100 cycles each from a single diverged lane: operands
//   pass to uniform registers one by one there.  A whole warp now runs the
//   loop and an elected lane issues: 43-56.
// - waits of 500-1800 for the next K tile: one warp issued K's and V's boxes
//   and 32 L2 requests a tile, one after another.  K and V now have a warp
//   each, and ask L2 for 4 KB at a time after their loads.
// - P is handed over in halves, so that P.V starts on the first while the
//   second is computed.
// Now 3390 (2048 at the tensor core's rate).  200 suffixes of about 500 tokens
// with one 8192-token prefix 96.5 -> 82.3 us a step, 128 of about 100 with two
// of 4096 tokens 47.0 -> 40.5, 12 of about 500 with 4096 tokens 20.2 -> 19.1.
// Looking at four barriers at once instead of in turn gave nothing more.
//
// Each CTA leaves, per (sharer, KV head), one fp32 record (unnormalised o,
// running max m, sum l) in the same format as the decode kernel's split
// partials; the combine kernel merges prefix and suffix records, which is
// exact because the softmax over the whole context factorises over any
// partition of the keys.
#pragma once

#include "attn_impl.cuh"

namespace kvp {

constexpr int kPreRows = 128;             // query rows (sharer, head) per Q tile: the MMA's M
constexpr int kPreQTiles = 2;             // Q tiles per CTA, sharing every K/V tile
constexpr int kPreKeys = 128;             // prefix tokens per pipeline tile: S's N, P.V's K
constexpr int kPreChunk = 64;             // granularity of prefix lengths and key splits
constexpr int kPreStages = 2;
constexpr int kPreSoftWarps = 4;          // per Q tile: one thread per query row
constexpr int kPreThreads = (kPreQTiles * kPreSoftWarps + 3) * 32;  // + K and V load warps + MMA warp
constexpr int kPreAhead = 4;              // key tiles asked of L2 ahead of their loads
constexpr int kPreRowsCap = 256;          // 16-token sub-tiles resolved up front
constexpr int kMaxKeySplits = 8;
constexpr int kCascadeWords = 4080;       // most plan words (the plan kernel's parameters, then the workspace)
// TMEM per Q tile: S [0, 128) fp32, P over S's first 64 columns (bf16 pairs), O [128, 128 + d)
constexpr uint32_t kPreTmemCols = 256;

struct CascadeArgs {
    const uint16_t *q;
    const uint16_t *pool;  // pool base (rows of d bf16)
    const int32_t *table;
    int32_t *err;
    float *ws_pre;        // [kMaxKeySplits][S][Hkv] records of merge_floats<D, G>() floats
    int32_t *ws_skip;     // [S]: shared-prefix tokens per sequence (0 = none)
    int64_t rows_per_page;
    int64_t pool_pages;
    int32_t pages_per_block;
    int32_t max_blocks;
    int32_t S;
    int32_t Hkv;
    int32_t bs;
    int32_t KS;           // key splits of every group's prefix
    int32_t n_groups;
    int32_t n_members;
    float qk_scale;       // scale * log2(e)
    int32_t overlap;      // 1: release the decode grid before the wait (it waits on the plan kernel's flags)
    // the plan in the workspace, written by the plan kernel before this grid
    // reads it: [n_groups + 1] first row tile of each group | [n_groups + 1]
    // first member index | [n_groups] prefix tokens | [n_members] member
    // sequences | [S] skip
    const int32_t *plan;
};

// members per CTA: whole query-head groups of consecutive members in each of
// its Q tiles
template <int G>
__host__ __device__ constexpr int pre_members_per_tile() { return kPreQTiles * (kPreRows / G); }

// Pool row (TMA y) of the K sub-tile holding prefix tokens 16q .. 16q+15 for
// KV head g, read from the lead member's table; -1 if outside the pool.
__device__ __forceinline__ int32_t pre_sub_row(const CascadeArgs &c, int lead, int g, int32_t q)
{
    const int32_t tok = q * kTile;
    const int32_t phys = c.table[(int64_t)lead * c.max_blocks + tok / c.bs];
    if (phys < 0 || (int64_t)phys + c.pages_per_block > c.pool_pages) return -1;
    return (int32_t)((int64_t)phys * c.rows_per_page + (int64_t)g * c.bs + tok % c.bs);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// shared-memory layout of the prefix kernel (offsets from a 1024-byte aligned
// base): Q [tiles][halves][128 rows][128 B] | stages x (K, V) [halves][128
// keys][128 B] | mbarriers | TMEM address | sub-tile rows
template <int D>
struct PreSmem {
    static constexpr int HALVES = D / 64;
    static constexpr uint32_t KV_HALF = kPreKeys * 128;       // 128 keys x 64 columns
    static constexpr uint32_t KV_TILE = HALVES * KV_HALF;     // K (or V) of one key tile
    static constexpr uint32_t STAGE = 2 * KV_TILE;
    static constexpr uint32_t Q_HALF = kPreRows * 128;
    static constexpr uint32_t Q_TILE = HALVES * Q_HALF;
    static constexpr uint32_t Q_OFF = 0;
    static constexpr uint32_t ST_OFF = kPreQTiles * Q_TILE;
    static constexpr uint32_t BAR_OFF = ST_OFF + kPreStages * STAGE;
    // full and empty per stage, of K and of V; per Q tile: s_full, p_full of
    // each half, o_done; fin; q_ready
    static constexpr int NBARS = 4 * kPreStages + 4 * kPreQTiles + 2;
    static constexpr uint32_t SLOT_OFF = BAR_OFF + NBARS * 8;
    static constexpr uint32_t ROWS_OFF = SLOT_OFF + 16;
    static constexpr uint32_t BYTES = ROWS_OFF + kPreRowsCap * 4;
};

template <int D, int G>
__global__ void __launch_bounds__(kPreThreads, 1)
cascade_prefix_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CascadeArgs c)
{
    using L = PreSmem<D>;
    constexpr int HALVES = L::HALVES;
    constexpr uint32_t MF = merge_floats<D, G>();
    constexpr int MQ = kPreRows / G;               // members per Q tile
    constexpr int MT = pre_members_per_tile<G>();  // members per CTA (kPreQTiles Q tiles)
    constexpr int NSUB = kPreKeys / kTile;         // 16-token sub-tiles per key tile
    constexpr int CSUB = kPreChunk / kTile;        // sub-tiles per 64-key chunk
    constexpr uint32_t O_COL = kPreKeys;           // within a Q tile's TMEM columns
    constexpr int SOFT_THREADS = kPreQTiles * kPreSoftWarps * 32;
    static_assert(O_COL + D <= kPreTmemCols, "S (with P over it) and O fit a Q tile's TMEM columns");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(smem);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::BAR_OFF);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + L::SLOT_OFF);
    int32_t *rows = reinterpret_cast<int32_t *>(smem + L::ROWS_OFF);
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    constexpr int FULL_K = 0, EMPTY_K = kPreStages, FULL_V = 2 * kPreStages, EMPTY_V = 3 * kPreStages;
    constexpr int QB = 4 * kPreStages, FIN = QB + 4 * kPreQTiles, Q_READY = FIN + 1;
    auto s_full = [&](int a) { return bar(QB + 4 * a); };
    auto p_full = [&](int a, int half) { return bar(QB + 4 * a + 1 + half); };  // P of keys 64 half .. 64 half + 63
    auto o_done = [&](int a) { return bar(QB + 4 * a + 3); };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int bid = blockIdx.x;
    const int ks = bid % c.KS;
    bid /= c.KS;
    const int g = bid % c.Hkv;
    const int tile = bid / c.Hkv;

    if (tid == 0) {
        for (int i = 0; i < 4 * kPreStages; ++i) mbar_init(bar(i), 1);
        for (int a = 0; a < kPreQTiles; ++a) {
            mbar_init(s_full(a), 1);
            mbar_init(p_full(a, 0), kPreSoftWarps * 32);
            mbar_init(p_full(a, 1), kPreSoftWarps * 32);
            mbar_init(o_done(a), 1);
        }
        mbar_init(bar(FIN), 1);
        mbar_init(bar(Q_READY), SOFT_THREADS);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), kPreQTiles * kPreTmemCols);
        tmem_relinquish();
    }
    if (tid == 32) prefetch_tensormap(&tmap);
    // barriers initialised and TMEM allocated: everything below may use them
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    bool dead = false;
    constexpr int LOAD_WARP = kPreQTiles * kPreSoftWarps, MMA_WARP = LOAD_WARP + 2;  // K's, V's; MMA
    // Wait for the grid before (the plan kernel; through it the table sync
    // and the previous step's combine), then release the decode kernel that
    // follows: it runs beside this grid on the SMs this grid leaves free and
    // relies on this wait having completed in every CTA here.  When the step
    // overlaps the previous step's combine, the decode kernel waits on the
    // plan kernel's flags instead and is released first.  The plan is read
    // and the records written only after the wait: the plan kernel wrote the
    // plan, and the previous combine read the records.
    if (c.overlap) grid_launch_dependents();
    grid_dependency_wait();
    if (!c.overlap) grid_launch_dependents();

    const int32_t *tile_off = c.plan;
    const int32_t *mem_off = tile_off + c.n_groups + 1;
    const int32_t *tokens = mem_off + c.n_groups + 1;
    const int32_t *members = tokens + c.n_groups;
    // This CTA's group, member range and prefix, looked up by each warp: 32
    // groups a round trip (through L2: another kernel wrote the plan; a
    // round trip is 0.7 us, more beside the suffix stream, and the first loads
    // wait for these).
    int mo = 0, mend = 0, ntok = 0, tile0 = 0;
    for (int i0 = 0; i0 < c.n_groups; i0 += 32) {
        const int i = min(i0 + lane, c.n_groups - 1);
        const int t_a = __ldcg(tile_off + i), t_b = __ldcg(tile_off + i + 1);
        const int m_a = __ldcg(mem_off + i), m_b = __ldcg(mem_off + i + 1), tk = __ldcg(tokens + i);
        const unsigned hit = __ballot_sync(0xffffffffu, t_b > tile);
        if (hit) {
            const int l = __ffs((int)hit) - 1;
            tile0 = __shfl_sync(0xffffffffu, t_a, l);  // the group's first row tile
            mo = __shfl_sync(0xffffffffu, m_a, l);
            mend = __shfl_sync(0xffffffffu, m_b, l);
            ntok = __shfl_sync(0xffffffffu, tk, l);
            break;
        }
    }
    const int lead = __ldcg(members + mo);
    const int m0 = mo + (tile - tile0) * MT;                    // this CTA's members [m0, m1)
    const int m1 = min(m0 + MT, mend);
    const int ch_all = ntok / kPreChunk;                        // 64-key chunks of the prefix
    const int ch0 = ks * ch_all / c.KS, ch1 = (ks + 1) * ch_all / c.KS;  // non-empty: KS <= ch_all
    const int nch = ch1 - ch0;
    const int nt = (nch + 1) / 2;                                // key tiles; the last may hold one chunk
    const int nsub = nch * CSUB;
    // valid keys of key tile t: 128, or 64 for a final half tile
    auto tile_keys = [&](int t) { return min(kPreKeys, (nch - 2 * t) * kPreChunk); };

    // Q rows (member, head) of KV head g into the swizzled K-major layout the
    // MMA reads: softmax thread t fills row t % 128 of Q tile t / 128; rows
    // past the CTA's members are zero.  The MMA thread waits for q_ready.
    const int Hq = c.Hkv * G;
    const int qa_tile = tid / kPreRows, r = tid % kPreRows;  // Q tile and row of a softmax thread
    const int mrow = m0 + qa_tile * MQ + r / G;               // its member index
    const bool row_ok = tid < SOFT_THREADS && r < MQ * G && mrow < m1;
    if (tid < SOFT_THREADS) {
        const uint16_t *qrow = row_ok ? c.q + ((int64_t)__ldcg(members + mrow) * Hq + (int64_t)g * G + r % G) * D
                                      : nullptr;
        uint8_t *qdst = smem + L::Q_OFF + qa_tile * L::Q_TILE;
        uint4 qv[D / 8];
#pragma unroll
        for (int ch = 0; ch < D / 8; ++ch)
            qv[ch] = row_ok ? *reinterpret_cast<const uint4 *>(qrow + ch * 8) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int ch = 0; ch < D / 8; ++ch)
            *reinterpret_cast<uint4 *>(qdst + (ch / 8) * L::Q_HALF + swz(r, ch % 8)) = qv[ch];
        fence_proxy_async_smem();  // Q (generic stores) is read by the tensor cores
        mbar_arrive(bar(Q_READY));
    }

    if (warp == LOAD_WARP || warp == LOAD_WARP + 1) {
        // ---- TMA producer warps, one of K and one of V: each resolves the pool
        // rows of the CTA's key range from the block table (both write the same
        // rows), then streams its half of key tile t into stage t % stages,
        // one box per lane (one issuing thread per SM cannot keep the loads
        // flowing; a warp's boxes are issued one after another, so that one
        // warp for both held the next K back) ----
        const bool is_v = warp != LOAD_WARP;
        for (int i = lane; i < min(nsub, kPreRowsCap); i += 32) rows[i] = pre_sub_row(c, lead, g, ch0 * CSUB + i);
        __syncwarp();
        const uint64_t pol = l2_policy_evict_normal();  // the prefix is re-read by every row tile
        constexpr int NBOX = NSUB * HALVES;               // boxes per full key tile
        static_assert(NBOX <= 32, "one box per lane");
        const int full0 = is_v ? FULL_V : FULL_K, empty0 = is_v ? EMPTY_V : EMPTY_K;
        // box (j, h): rows 16j .. 16j + 15, columns 64h .. 64h + 63 of a key tile
        const int j = lane / HALVES, h = lane % HALVES;
        auto row_of = [&](int q) {  // of sub-tile q: -1 outside the pool
            const int32_t y = q < kPreRowsCap ? rows[q] : pre_sub_row(c, lead, g, ch0 * CSUB + q);
            return y < 0 ? y : y + (is_v ? c.Hkv * c.bs : 0);
        };
        for (int t = 0; t < nt; ++t) {
            const int st = t % kPreStages;
            const int vsub = tile_keys(t) / kTile;        // sub-tiles loaded this tile
            const bool mine = lane < NBOX && j < vsub;
            const int32_t y = mine ? row_of(t * NSUB + j) : 0;
            const bool ok = __all_sync(0xffffffffu, y >= 0);
            const uint32_t full = bar(full0 + st);
            if (t >= kPreStages) wait_phase(bar(empty0 + st), (uint32_t)(t / kPreStages - 1) & 1u, c.err, dead);
            if (lane == 0) {
                if (ok) {
                    mbar_arrive_expect_tx(full, (uint32_t)vsub * HALVES * (kTile * 128));
                } else {
                    report(c.err, KV_ERR_DEVICE_BOUNDS);
                    mbar_arrive(full);  // complete the phase without data
                }
            }
            __syncwarp();
            if (ok && mine)
                tma_load_2d(sbase + L::ST_OFF + st * L::STAGE + (is_v ? L::KV_TILE : 0) + h * L::KV_HALF +
                                j * (kTile * 128),
                            &tmap, h * 64, y, full, pol);
            // the tile kPreAhead further on, into L2: a sub-tile's rows are
            // consecutive in the pool
            const int qa = (t + kPreAhead) * NSUB + lane;
            if (lane < NSUB && qa < nsub) {
                const int32_t ya = row_of(qa);
                if (ya >= 0) bulk_prefetch_l2(c.pool + (int64_t)ya * D, kTile * D * 2);
            }
            __syncwarp();
        }
        // drain: the last stages' loads have landed (already waited on by the
        // MMA warp unless a wait ran out)
        if (lane == 0)
            for (int t = max(0, nt - kPreStages); t < nt; ++t)
                wait_phase(bar(full0 + t % kPreStages), (uint32_t)(t / kPreStages) & 1u, c.err, dead);
    } else if (warp == MMA_WARP) {
        // ---- MMA issuer.  Per Q tile a and key tile t: S_a = Q_a K_t^T into
        // TMEM, then, once the tile's warps have written P (bf16) over S,
        // O_a += P V_t with P read from TMEM.  The tensor pipe runs one
        // thread's MMAs in issue order, so S_a(t+1), issued after
        // P.V_a(t), overwrites P only after that MMA has read it.  Order:
        // S_0(0) S_1(0) | PV_0(t) S_0(t+1) PV_1(t) S_1(t+1) | ... ----
        const uint32_t el = elect_one();
        constexpr uint32_t ID_S = idesc_bf16_f32(kPreRows, kPreKeys, 0, 0);
        constexpr uint32_t ID_S_HALF = idesc_bf16_f32(kPreRows, kPreChunk, 0, 0);
        constexpr uint32_t ID_O = idesc_bf16_f32(kPreRows, D, 0, 1);
        auto issue_s = [&](int a, int t) {
            const uint32_t ka = sbase + L::ST_OFF + (t % kPreStages) * L::STAGE;
            const uint32_t qa = sbase + L::Q_OFF + a * L::Q_TILE;
            const uint32_t id = tile_keys(t) == kPreKeys ? ID_S : ID_S_HALF;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
                umma_bf16(tbase + a * kPreTmemCols, smem_desc_sw128(qa + (kk / 4) * L::Q_HALF + (kk % 4) * 32, 16, 1024),
                          smem_desc_sw128(ka + (kk / 4) * L::KV_HALF + (kk % 4) * 32, 16, 1024), id, kk > 0, el);
            umma_commit(s_full(a), el);
        };
        auto issue_pv = [&](int a, int t, int half) {
            const uint32_t va = sbase + L::ST_OFF + (t % kPreStages) * L::STAGE + L::KV_TILE;
            constexpr int STEPS = kPreChunk / 16;
#pragma unroll
            for (int i = 0; i < STEPS; ++i) {
                const int kk = half * STEPS + i;
                umma_bf16_tmem_a(tbase + a * kPreTmemCols + O_COL, tbase + a * kPreTmemCols + kk * 8,
                                 smem_desc_sw128(va + kk * (16 * 128), L::KV_HALF, 1024), ID_O, t > 0 || kk > 0, el);
            }
        };
        wait_phase(bar(Q_READY), 0u, c.err, dead);
        wait_phase(bar(FULL_K + 0), 0u, c.err, dead);
        tc_fence_after();
        for (int a = 0; a < kPreQTiles; ++a) issue_s(a, 0);
        umma_commit(bar(EMPTY_K + 0), el);
        for (int t = 0; t < nt; ++t) {
            const bool next = t + 1 < nt;
            for (int a = 0; a < kPreQTiles; ++a) {
                if (a == 0)
                    wait_phase(bar(FULL_V + t % kPreStages), (uint32_t)(t / kPreStages) & 1u, c.err, dead);
                wait_phase(p_full(a, 0), (uint32_t)t & 1u, c.err, dead);
                tc_fence_after();
                issue_pv(a, t, 0);
                wait_phase(p_full(a, 1), (uint32_t)t & 1u, c.err, dead);
                if (tile_keys(t) > kPreChunk) {
                    tc_fence_after();
                    issue_pv(a, t, 1);
                }
                umma_commit(o_done(a), el);
                if (a == kPreQTiles - 1) umma_commit(bar(EMPTY_V + t % kPreStages), el);
                if (next) {
                    if (a == 0) wait_phase(bar(FULL_K + (t + 1) % kPreStages), (uint32_t)((t + 1) / kPreStages) & 1u,
                                           c.err, dead);
                    tc_fence_after();
                    issue_s(a, t + 1);
                    if (a == kPreQTiles - 1) umma_commit(bar(EMPTY_K + (t + 1) % kPreStages), el);
                }
            }
        }
        // every MMA of this thread has completed before TMEM is released
        umma_commit(bar(FIN), el);
        wait_phase(bar(FIN), 0u, c.err, dead);
    } else if (tid < SOFT_THREADS) {
        // ---- softmax: thread tid owns row r of Q tile qa_tile (TMEM lane r) ----
        const int a = qa_tile;
        const uint32_t trow = tbase + a * kPreTmemCols + ((uint32_t)((warp % 4) * 32) << 16);
        const float scale = c.qk_scale;
        float m_run = kMaxStart, l_run = 0.f;
        for (int t = 0; t < nt; ++t) {
            const int nk = tile_keys(t);  // 128 or 64
            // S_a(t) complete: so is every earlier MMA of the tile, in
            // particular P.V_a(t-1), so O is stable and P's columns are free
            wait_phase(s_full(a), (uint32_t)t & 1u, c.err, dead);
            tc_fence_after();
            // The row's maximum (scores read twice: 128 in registers spilled,
            // 96.7 -> 123.5 us on the step above).  m_ref, the reference of o,
            // l and P, is raised (lazy rescale) only when the tile exceeds it
            // by more than 2^8; then O and l are scaled by 2^(m_old - m_new)
            // first, so every stored p stays <= 2^8.
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            uint32_t v[2][32];
#pragma unroll
            for (int cp = kPreKeys / kPreChunk - 1; cp >= 0; --cp)
                if (cp * kPreChunk < nk) {
                    tmem_ld32(trow + cp * kPreChunk, v[0]);
                    tmem_ld32(trow + cp * kPreChunk + 32, v[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 64; ++i) mx[i & 3] = fmaxf(mx[i & 3], __uint_as_float(v[i >> 5][i & 31]));
                }
            const float cmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale;
            if (cmax > m_run + 8.f) {
                const float al = fast_exp2(m_run - cmax);  // 0 when nothing came before
                l_run *= al;
                if (t >= 1) {  // O holds earlier tiles
                    uint32_t o[32];
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb) {
                        tmem_ld32(trow + O_COL + cb * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * al);
                        tmem_st32(trow + O_COL + cb * 32, o);
                    }
                }
                m_run = cmax;
            }
            // p = 2^(s * scale - m_ref) as bf16 pairs over the first columns
            // of S (the A operand of P.V), one 64-key half at a time: the MMA
            // thread starts on the first while the second is computed
#pragma unroll
            for (int cp = 0; cp < kPreKeys / kPreChunk; ++cp) {
                if (cp * kPreChunk < nk) {
                    if (cp > 0) {  // the first half's scores are still in v
                        tmem_ld32(trow + cp * kPreChunk, v[0]);
                        tmem_ld32(trow + cp * kPreChunk + 32, v[1]);
                        tmem_wait_ld();
                    }
                    uint32_t w[32];
                    float r4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int i = 0; i < 64; i += 2) {
                        const uint32_t(&x)[32] = v[i >> 5];
                        const float p0 = fast_exp2(fmaf(__uint_as_float(x[i & 31]), scale, -m_run));
                        const float p1 = fast_exp2(fmaf(__uint_as_float(x[(i + 1) & 31]), scale, -m_run));
                        r4[(i >> 1) & 3] += p0 + p1;
                        w[i / 2] = pack_bf16(p0, p1);
                    }
                    l_run += (r4[0] + r4[1]) + (r4[2] + r4[3]);
                    tmem_st32(trow + cp * 32, w);
                    tmem_wait_st();
                    tc_fence_before();
                }
                mbar_arrive(p_full(a, cp));
            }
        }
        // ---- this CTA's record per (sharer, KV head) ----
        wait_phase(o_done(a), (uint32_t)(nt - 1) & 1u, c.err, dead);
        tc_fence_after();
        float *rec = row_ok && !dead
                         ? c.ws_pre + (((int64_t)ks * c.S + __ldcg(members + mrow)) * c.Hkv + g) * MF
                         : nullptr;
        const int hl = r % G;
        // O leaves through shared memory, 32 columns at a time, so that eight
        // lanes write 128 consecutive bytes of a record (a lane writing its
        // own row spread each store over 32 lines: the last step of a CTA,
        // from the last P on, took 6 us).  The buffer is the stage that the
        // last key tile did not use: every MMA that reads it was issued
        // before the P.V just completed.
        float *xb = reinterpret_cast<float *>(smem + L::ST_OFF + (nt % kPreStages) * L::STAGE) + warp * 32 * 32;
        static_assert(SOFT_THREADS / 32 * 32 * 32 * 4 <= L::STAGE, "a 32 x 32 block per softmax warp");
        const unsigned long long orow = rec ? reinterpret_cast<unsigned long long>(rec + hl * D) : 0ull;
        uint32_t v[32];
#pragma unroll
        for (int cb = 0; cb < D / 32; ++cb) {
            tmem_ld32(trow + O_COL + cb * 32, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<uint4 *>(xb + lane * 32 + ((i ^ (lane & 7)) * 4)) =
                    make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rr = i * 4 + lane / 8, ch = lane % 8;  // row, 16-byte chunk
                const unsigned long long dst = __shfl_sync(0xffffffffu, orow, rr);
                const uint4 w = *reinterpret_cast<const uint4 *>(xb + rr * 32 + ((ch ^ (rr & 7)) * 4));
                if (dst) *reinterpret_cast<uint4 *>(reinterpret_cast<float *>(dst) + cb * 32 + ch * 4) = w;
            }
            __syncwarp();
        }
        if (rec) {
            rec[G * D + hl] = m_run;
            rec[G * D + G + hl] = l_run;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tbase, kPreQTiles * kPreTmemCols);
}

template <int D>
inline size_t cascade_smem_bytes()
{
    return 1024 + (size_t)PreSmem<D>::BYTES;
}

}  // namespace kvp
