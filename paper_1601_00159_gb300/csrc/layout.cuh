// The end of a batch on the device, shared by the kernels that may finish one: the sizes after
// the batch, the decision to rebuild the index layer, and the layout of its levels.
#pragma once

#include "common.cuh"

namespace pi {

// Whether the batch re-lays-out the storage layer: new nodes must be placed, or delete-flagged
// nodes exceed 1/8 of it. Only reads what stays as it is while the batch ends.
__device__ __forceinline__ bool merge_needed(const BatchMeta* bm) {
    const uint32_t tombs = (uint32_t)((int32_t)bm->tombs0 + bm->tomb_delta);
    return bm->new_count > 0 || (tombs > 0 && (uint64_t)tombs * 8u > bm->size0);
}

__device__ __forceinline__ uint64_t suffix_sum64(uint64_t v, uint32_t lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + (uint32_t)o < 32u) v += y;
    }
    return v;
}

// Applies the batch's deltas, switches storage buffers after a merge, decides the rebuild, and
// lays the index levels out top-first with their sentinels. Called by one whole warp, once per
// batch, after every other access to these counters; lane i has level i + 1 (heights reach 32).
// Each lane reads its level's words in one round trip and the sums over levels are warp
// scans: on one thread, word after word, this step took 8 us of a batch (5.2 us of kernel time
// between events, an empty launch's, as a warp).
__device__ __forceinline__ void level_layout(const RebuildArgs& a, bool merged) {
    constexpr uint32_t kAll = 0xffffffffu;
    DevMeta* m = a.m;
    BatchMeta* bm = a.bm;
    const uint32_t lane = threadIdx.x & 31u, l = lane + 1u;
    if (__shfl_sync(kAll, __ldcg(&m->error), 0)) return;
    const uint32_t cnt = (uint32_t)((int32_t)__ldcg(&m->cnt[l]) + __ldcg(&bm->delta[l]));
    const uint32_t old_n = __ldcg(&m->n[l]), old_base = __ldcg(&m->base[l]);
    const uint32_t chg = __ldcg(&bm->chg_hist[l]) + (l == 32u ? __ldcg(&bm->chg_hist[33]) : 0u);
    uint32_t tombs = (uint32_t)((int32_t)__ldcg(&m->tombs) + __ldcg(&bm->tomb_delta));
    uint32_t size = __ldcg(&m->size), cur = __ldcg(&m->cur), lcur = __ldcg(&m->lcur);
    const uint32_t oH = __ldcg(&m->H), oLb = __ldcg(&m->Lb);
    const uint32_t exact = __ldcg(&m->levels_exact), dirty = __ldcg(&bm->index_dirty);
    const uint32_t updates = __ldcg(&m->updates) + __ldcg(&bm->changes);
    const uint32_t newc = __ldcg(&bm->new_count), big = __ldcg(&bm->fix_big);
    const uint32_t batches = __ldcg(&m->batches), rebuilds = __ldcg(&m->rebuilds);
    const uint32_t incs = __ldcg(&m->inc_rebuilds);
    if (merged) {
        size = size - tombs + newc;
        tombs = 0;
        cur ^= 1u;
    }
    if (size > a.st_cap) {  // cannot happen when the host reserved capacity
        if (lane == 0) atomicOr(a.err, kErrBounds);
        return;
    }
    bool rebuild = a.force_rebuild || merged;
    if (!rebuild && dirty)
        rebuild = a.rebuild_policy == 0 ||
                  (uint64_t)updates * 100u >= (uint64_t)a.threshold_pct * (uint64_t)(size ? size : 1u);
    m->cnt[l] = cnt;
    if (lane == 0) {
        m->size = size;
        m->tombs = tombs;
        m->cur = cur;
        a.st.keys[cur][size] = kMaxKey;
        a.st.vals[cur][size] = 0;
        a.st.meta[cur][size] = 0;
        m->updates = rebuild ? 0u : updates;
        m->sort_fix_big = big;
        if (a.force_rebuild != 2u) m->batches = batches + 1u;
        bm->merged = merged ? 1u : 0u;
        bm->rebuild = rebuild ? 1u : 0u;
        if (rebuild) m->rebuilds = rebuilds + 1u;
        else if (dirty) m->levels_exact = 0;  // deferred: the levels now lag the storage layer
    }
    if (!rebuild) return;
    // the layout being replaced, for an incremental rebuild
    bm->old_n[l] = old_n;
    bm->old_base[l] = old_base;
    const uint32_t have = __ballot_sync(kAll, l >= 2u && cnt > 0u);
    const uint32_t H = have ? 32u - (uint32_t)__clz(have) : 1u;
    // entries of the levels from l up to H, sentinels included
    const uint64_t S = suffix_sum64(l >= 2u && l <= H ? (uint64_t)cnt + 1u : 0ull, lane);
    const uint32_t Lb0 = a.min_lb > 2u ? a.min_lb : 2u;
    const uint64_t need = Lb0 <= H ? __shfl_sync(kAll, S, (int)((Lb0 - 1u) & 31u)) : 0ull;
    // Lowest level that fits: bottom levels are dropped (the descent then scans longer
    // storage gaps) rather than overrun the capacity; the host grows it later.
    const uint32_t fits = __ballot_sync(kAll, l >= Lb0 && l <= H && S <= (uint64_t)a.index_cap);
    const uint32_t Lb = Lb0 > H ? Lb0 : (fits ? (uint32_t)__ffs(fits) : H + 1u);
    const bool built = l >= Lb && l <= H;
    const uint32_t n = built ? cnt : 0u, base = built ? (uint32_t)(S - cnt - 1u) : 0u;
    m->n[l] = n;
    m->base[l] = base;
    const uint32_t total = (uint32_t)__reduce_max_sync(kAll, built ? base + n + 1u : 0u);
    const uint32_t pins = __ballot_sync(kAll, built && base + n + 1u <= a.smem_top);
    const uint32_t Ls = pins ? (uint32_t)__ffs(pins) : H + 1u;
    const uint32_t pinned = __reduce_max_sync(kAll, (pins >> lane) & 1u ? base + n + 1u : 0u);
    // Incremental when the storage layer kept its layout and the old levels are exact:
    // the new levels are the old ones plus the batch's membership changes, written to
    // the other buffer. The per-level change lists must fit their arrays.
    bool inc = !merged && a.force_rebuild == 0 && exact && Lb == oLb && oLb <= oH && Lb <= H;
    {
        const uint32_t Hm = H > oH ? H : oH;
        const uint64_t ge = suffix_sum64(chg, lane);
        const uint64_t lists = suffix_sum64(l >= Lb && l <= Hm ? ge + 1u : 0ull, lane);
        inc = inc && __shfl_sync(kAll, lists, 0) <= a.lst_cap;
    }
    lcur ^= inc ? 1u : 0u;
    const uint32_t cnt_below = __shfl_up_sync(kAll, cnt, 1);
    if (built) {
        (lcur ? a.lkeys1 : a.lkeys)[base + n] = kMaxKey;
        (lcur ? a.ldown1 : a.ldown)[base + n] = l > Lb ? cnt_below : size;
    }
    if (lane == 0) {
        bm->old_H = oH;
        bm->inc = inc ? 1u : 0u;
        m->H = H;
        m->Lb = Lb;
        m->index_total = total;
        m->index_need = (uint32_t)need;
        m->grow_request = Lb > Lb0 ? 1u : 0u;
        m->Ls = Ls;
        m->smem_entries = pinned;
        m->lcur = lcur;
        if (inc) m->inc_rebuilds = incs + 1u;
        m->levels_exact = 1;
    }
}

// The last step of a batch, by one warp: the device meta goes to the batch's mailbox slot, which
// the host reads once the batch's event has completed, and the next batch's counters are
// cleared (their previous user, the rebuild of the batch before this one, has finished: this
// batch's descent waited for it). In the kernel these cost no copy or memset on the stream.
__device__ __forceinline__ void post_batch(const RebuildArgs& a) {
    const uint32_t lane = threadIdx.x & 31u;
    constexpr uint32_t kMetaWords = sizeof(DevMeta) / 4, kBatchWords = sizeof(BatchMeta) / 4;
    static_assert(sizeof(DevMeta) % 4 == 0 && sizeof(BatchMeta) % 4 == 0, "word copies");
    __syncwarp();
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.m);
    uint32_t* dst = reinterpret_cast<uint32_t*>(a.mbox);
    uint32_t* nxt = reinterpret_cast<uint32_t*>(a.bm_next);
    for (uint32_t w = lane; w < kMetaWords; w += 32u) dst[w] = __ldcg(&src[w]);
    for (uint32_t w = lane; w < kBatchWords; w += 32u) nxt[w] = 0u;
}

}  // namespace pi
