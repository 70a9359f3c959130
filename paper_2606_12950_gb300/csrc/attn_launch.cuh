// attn_launch.cuh -- host-side launch of one paged-attention instantiation:
// stage count, shared memory, grid (one CTA per resident slot unless the
// caller asks for a given number of work partitions).
#pragma once

#include <algorithm>
#include <atomic>

#include "cascade_impl.cuh"
#include "stream_order.h"

namespace kvp {

// shared memory of one CTA: up to 227 KB; the block-table window (rows of the
// CTA's units resolved in the prologue) is kRowsCap entries
constexpr size_t kSmemMax = 227 * 1024;

// Resident CTAs per SM of kernel fn at this block size and dynamic shared
// memory, queried once per (block size, shared-memory size) and cached in
// the caller's slot, one slot per kernel instantiation: the runtime query
// costs microseconds of host time on every launch.
struct OccCache {
    static constexpr int kSlots = 4;  // a call may query two shapes (its workspace's, its launch's)
    // (smem * 2048 + threads) << 8 | CTAs per SM, one word so that a reader
    // sees a key only with its own value
    std::atomic<long long> slot[kSlots] = {{-1}, {-1}, {-1}, {-1}};
    std::atomic<unsigned> next{0};
};

template <class Fn>
int cached_occupancy(Fn fn, int threads, size_t smem, int *occ, OccCache &c)
{
    const long long key = (long long)smem * 2048 + threads;
    for (int i = 0; i < OccCache::kSlots; ++i) {
        const long long w = c.slot[i].load(std::memory_order_relaxed);
        if (w >= 0 && (w >> 8) == key) {
            *occ = (int)(w & 255);
            return KV_OK;
        }
    }
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, threads, smem) != cudaSuccess) return KV_ERR_CUDA;
    const unsigned i = c.next.fetch_add(1, std::memory_order_relaxed) % OccCache::kSlots;
    c.slot[i].store(key << 8 | (long long)(o & 255), std::memory_order_relaxed);
    *occ = o;
    return KV_OK;
}

// The combine over c's runs: `groups` thread groups a CTA, CS CTAs a run.
template <int D, int G, int CPT, int CS, int MODE>
int combine_launch(const CombineArgs &c, int groups, cudaLaunchConfig_t cfg, int parts = 0)
{
    const int threads = groups * CombineShape<D, G, CPT, CS>::NCT;
    cfg.gridDim = dim3((unsigned)(MODE == kRecCtasByPart ? parts : c.S * c.Hkv), (unsigned)CS);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = combine_smem_bytes<D, G, CPT, CS>(threads);
    if (cudaLaunchKernelEx(&cfg, combine_kernel<D, G, CPT, CS, MODE>, c) != cudaSuccess) return KV_ERR_CUDA;
    kvp_note_stream(cfg.stream, true);
    return KV_OK;
}

// Few runs: each run's columns spread over CS CTAs (kSlicedCtas).
template <int D, int G, int MODE>
int combine_run(const CombineArgs &c, double per_run, int sm_count, const cudaLaunchConfig_t &cfg)
{
    const int runs = c.S * c.Hkv;
    if (8 * runs <= kSlicedCtas * sm_count)
        return combine_launch<D, G, 1, 8, MODE>(c, combine_groups<D, G, 8>(per_run), cfg);
    if (4 * runs <= kSlicedCtas * sm_count)
        return combine_launch<D, G, 1, 4, MODE>(c, combine_groups<D, G, 4>(per_run), cfg);
    return combine_launch<D, G, 1, 1, MODE>(c, combine_groups<D, G, 1>(per_run), cfg);
}

// what: kLaunchQuery (only *P_out), kLaunchBoth (attention, then combine),
// kLaunchAttention, kLaunchCombine
enum { kLaunchQuery = 0, kLaunchBoth = 1, kLaunchAttention = 2, kLaunchCombine = 3 };

template <int D, int G, class Comp>
int attn_run(const CUtensorMap *tmap, AttnArgs a, int P_req, int sm_count, cudaStream_t st, int what, int *P_out)
{
    auto fn = paged_attn_kernel<D, G, Comp, kRecWarps>;
    auto fn_merge = paged_attn_kernel<D, G, Comp, kRecCtas>;
    auto fn_by_part = paged_attn_kernel<D, G, Comp, kRecCtasByPart>;
    static std::atomic<bool> attr_set{false};
    if (!attr_set.load()) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(fn_merge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(fn_by_part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess)
            return KV_ERR_CUDA;
        attr_set.store(true);
    }
    // six warps a CTA, eight beside the shared-prefix kernel (kPlainWarps)
    const int most_warps = a.skip != nullptr ? kWarps : kPlainWarps;
    // S too large for the per-CTA sequence index beside a box of K and of V a
    // warp (14109 sequences at d = 128, 16349 at d = 64, one query head a KV
    // head).  A unit of two boxes (d = 64) does not lower that limit: past
    // 14301 sequences fewer warps take their stages from what the index leaves,
    // three at the least.  There a CTA is alone on its SM either way.
    if (attn_smem_bytes<D, G>(a.S, kRowsCap, most_warps, false, 1) > kSmemMax) return KV_ERR_INVALID_ARG;
    a.nwarps = most_warps;
    while (attn_smem_bytes<D, G>(a.S, kRowsCap, a.nwarps, false) > kSmemMax) --a.nwarps;
    size_t smem = attn_smem_bytes<D, G>(a.S, kRowsCap, a.nwarps, false);
    int occ = 0;
    static OccCache occ_cache;
    if (cached_occupancy(fn, a.nwarps * 32, smem, &occ, occ_cache) != KV_OK) return KV_ERR_CUDA;
    const int resident = std::max(1, occ) * std::max(1, sm_count);
    const int P = P_req > 0 ? P_req : resident;
    *P_out = P;
    if (what == kLaunchQuery) return KV_OK;
    a.rows_cap = kRowsCap;
    a.bs_shift = -1;
    for (int k = 4; k < 31; ++k)
        if (a.bs == 1 << k) a.bs_shift = k;
    a.P = P;
    // Where the table has room for fewer than kMergeUnits units a warp, warps
    // may have a single unit and the CTAs merge their warps' records (MERGE).
    // This rule sees the table's width, not the lengths, so that a call gives
    // the same bits whether the lengths come with it or not.  Larger batches
    // merge too, unless the next step's decode kernel overlaps the combine
    // (chain 3): then only the CTAs' later end shows.  The bits are the same
    // either way (the combine merges a CTA's records first).  Beside a shared
    // prefix only the first rule holds.  In no case if the buffers cost a CTA per SM.
    // A caller may ask for more CTAs than are resident: the rule takes those
    // that are: single units would only make waves of CTAs that start and end (8
    // sequences of 300 to 2000 tokens, 32 q / 8 KV heads, 12.6 us with no splits
    // given: with 456 17.8 and 13.0 this way, with 1000 22.4 and 13.6).
    const int slots = std::min(P, resident);
    const bool small = small_batch(a, D, slots, a.nwarps);
    int32_t small_min_units = std::max(1, a.min_units);
    if (P > resident) {
        const int64_t warps = (int64_t)slots * a.nwarps;
        small_min_units = std::max(small_min_units, (int32_t)((table_units(a, D) + warps - 1) / warps));
    }
    small_min_units = std::min(small_min_units, kMinPartTokens / kUnit<D>);
    bool merge = false;
    a.min_units = kMinPartTokens / kUnit<D>;
    // (with fewer warps the combine, which merges kPlainWarps records at a time,
    // would not give a CTA's bits)
    if (a.nwarps == most_warps && (small || (a.chain != 3 && a.skip == nullptr))) {
        const size_t smem_merge = attn_smem_bytes<D, G>(a.S, kRowsCap, a.nwarps, true);
        int occ_merge = 0;
        static OccCache merge_cache;
        if (smem_merge <= kSmemMax) {
            if (cached_occupancy(fn_merge, a.nwarps * 32, smem_merge, &occ_merge, merge_cache) != KV_OK)
                return KV_ERR_CUDA;
            merge = occ_merge >= occ;
        }
        if (merge) {
            fn = fn_merge;
            smem = smem_merge;
            if (small) a.min_units = small_min_units;
        }
    }
    // At most one run per part starts there and goes on.  With several waves
    // of runs (eight runs a part: two waves of 128-thread combine CTAs) the
    // combine gets a CTA per part instead of one per run, most of which only
    // had to find their run whole: three co-located models (6560, 1640 and 816
    // runs) 266.4 -> 261.0 us, 1024 long contexts (8192) 691.4 -> 686.6, 1000
    // sequences of 400 tokens (8000) 263.5 -> 257.2.  With 960 and 1024 runs the
    // look for the run's end costs more than it saves: 92.8 -> 93.5 and 69.0 ->
    // 69.9.
    // (Never with runs few enough for column slices: the order of the merge
    // would differ from the overlapped form's.)
    const int64_t n_runs = (int64_t)a.S * a.Hkv;
    const bool by_part = merge && a.skip == nullptr && n_runs >= 8 * (int64_t)P && 4 * n_runs > (int64_t)kSlicedCtas * sm_count;
    if (by_part) fn = fn_by_part;
    // both kernels are programmatic dependents of what precedes them in the
    // stream: they may be scheduled early and wait on the device
    // (griddepcontrol.wait) for the previous grid to complete
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P);
    cfg.blockDim = dim3((unsigned)(a.nwarps * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (what != kLaunchCombine) {
        if (cudaLaunchKernelEx(&cfg, fn, *tmap, a) != cudaSuccess) return KV_ERR_CUDA;
        kvp_note_stream(st, false);
    }
    if (what == kLaunchAttention) return KV_OK;
    CombineArgs c{a.out, a.ws_run, a.ws_part, a.S, a.Hkv, a.skip, a.ws_pre, a.KS};
    cudaLaunchConfig_t ccfg = cfg;
    // records per run (of warps; of CTAs if the batch is small): at most one
    // per part, spread over the runs, plus the prefix records in
    // shared-prefix mode
    const int runs = a.S * a.Hkv;
    const double per_run = (double)P * (merge && small ? 1 : a.nwarps) / std::max(1, runs) + 1.0 + (a.skip ? a.KS : 0);
    if constexpr (G * D / 4 >= 128) {
        // one group in shared-prefix mode: two columns a thread, so that
        // every member run fits in one wave
        if (a.skip != nullptr && combine_groups<D, G, 1>(per_run) == 1)
            return combine_launch<D, G, 2, 1, kRecCtas>(c, 1, ccfg);
    }
    if (by_part) return combine_launch<D, G, 1, 1, kRecCtasByPart>(c, combine_groups<D, G, 1>(per_run), ccfg, P);
    return merge || a.skip != nullptr ? combine_run<D, G, kRecCtas>(c, per_run, sm_count, ccfg)
                                      : combine_run<D, G, kRecWarps>(c, per_run, sm_count, ccfg);
}

// Shared-prefix kernel: with launch = false only reports the CTAs that fit
// on the GPU at once (occupancy x SMs) in *P_out.
template <int D, int G>
int cascade_run(const CUtensorMap *tmap, const CascadeArgs *c, int grid, int sm_count, cudaStream_t st, bool launch,
                int *P_out)
{
    auto fn = cascade_prefix_kernel<D, G>;
    const size_t smem = cascade_smem_bytes<D>();
    static std::atomic<bool> attr_set{false};
    if (!attr_set.load()) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return KV_ERR_CUDA;
        attr_set.store(true);
    }
    if (!launch) {
        int occ = 0;
        static OccCache occ_cache;
        if (cached_occupancy(fn, kPreThreads, smem, &occ, occ_cache) != KV_OK) return KV_ERR_CUDA;
        *P_out = std::max(1, occ) * std::max(1, sm_count);
        return KV_OK;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kPreThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, fn, *tmap, *c) != cudaSuccess) return KV_ERR_CUDA;
    kvp_note_stream(st, false);
    return KV_OK;
}

}  // namespace kvp

// one entry per head dim; variant 1 = CUDA cores, 2 = tensor-core MMA
int kvp_attn_d64(int variant, int G, const CUtensorMap *tmap, const kvp::AttnArgs *a, int P_req, int sm_count,
                 cudaStream_t st, int what, int *P_out);
int kvp_attn_d128(int variant, int G, const CUtensorMap *tmap, const kvp::AttnArgs *a, int P_req, int sm_count,
                  cudaStream_t st, int what, int *P_out);
int kvp_cascade_d64(int G, const CUtensorMap *tmap, const kvp::CascadeArgs *c, int grid, int sm_count,
                    cudaStream_t st, bool launch, int *P_out);
int kvp_cascade_d128(int G, const CUtensorMap *tmap, const kvp::CascadeArgs *c, int grid, int sm_count,
                     cudaStream_t st, bool launch, int *P_out);
