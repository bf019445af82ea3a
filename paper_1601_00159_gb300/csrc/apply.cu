// K4 + K5: single ownership and query execution (Algorithms 3 and 4, Section 3.2.4).
//
// In the paper each execution thread owns the storage nodes between its first
// interception and the next thread's, handing queries over to its neighbour so that
// no node has two writers; within a thread the queries run in order. Here the whole
// sorted batch is one array and ownership is computed, not negotiated:
//  * a key run is a maximal stretch of equal keys in the sorted batch (its queries are
//    in arrival order, by the stable sort);
//  * every query reports the state of its key just before it: that is the effect of
//    the last insert/delete before it in its run, or, if there is none, the state the
//    descent found in the storage layer. An inclusive max-scan over
//        e_i = 2i+3 if query i writes, 2i+2 if it heads a run, 0 otherwise
//    gives, at i-1, either the index of that last write (odd) or the run head (even);
//  * the LAST query of each run is the run's only owner: it writes the run's final
//    state to the storage node (value, delete flag), or emits a new node when the key
//    is not in the storage layer and ends up present (Algorithm 4, insertNode).
//
// The max-scan is split across kernels so no tile of k_apply ever waits on another:
// the descent's first kernel already walks the sorted batch and leaves each 2048-query
// tile's exclusive max prefix of e (tile_pref); k_apply is then fully data-parallel. The descent stored one result per distinct key -- per local
// run head (a query whose key differs from the previous one, and the first query of
// every 256-query sub-tile) in sorted order -- so a query's storage-layer state is
// found at its run head's dense index.
// New nodes, and the changes of built levels' membership, go to their places in key order in
// the same pass: a tile's first place comes from a decoupled look-back over the tiles' counts,
// which only tiles that have some wait for. The CTA that finishes last ends the batch: it
// decides whether the storage layer is re-laid-out, and if not, lays out the index levels.
// (Staging the new nodes per tile, a scan and a packing kernel, and a one-thread level layout
// were three more launches: 6000 mixed queries on 2^20 keys 61.0 -> 55.6 us a batch with one
// pass; 2^22 skewed queries on 2^27 keys 556.6 -> 548.4.)

#include "layout.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;
constexpr int kApThreads = 512;                  // k_apply: two CTAs per SM at 64 registers
constexpr int kItems = kApplyTile / kApThreads;  // 4 sorted queries per thread
constexpr uint32_t kSeqMask = (1u << 30) - 1u;

__device__ __forceinline__ void store_result(pi_result_t* res, uint32_t seq, uint64_t v, uint32_t st) {
    uint4 w;
    w.x = (uint32_t)v;
    w.y = (uint32_t)(v >> 32);
    w.z = st;
    w.w = 0u;
    *reinterpret_cast<uint4*>(res + seq) = w;
}

// Largest ownership marker e_i before the tile at tb, by the whole CTA, for a tile whose
// first query continues the run before it (markers grow with i, so the nearest tile that
// has one decides; tile 0 heads the first run). Small batches only: their descent keeps no
// tile prefixes, and a run crosses few tiles.
__device__ uint32_t marker_before(const ApplyArgs& a, uint32_t tb, uint32_t* s_tmp) {
    while (tb > 0) {
        tb -= kApplyTile;
        uint32_t agg = 0;
#pragma unroll
        for (int k = 0; k < kItems; ++k) {  // whole tiles of valid queries: the run reaches past them
            const uint32_t i = tb + (uint32_t)k * kApThreads + threadIdx.x;
            const uint32_t op = a.sp[i] >> 30;
            const bool head = i == 0 || a.sk[i] != a.sk[i - 1];
            agg = max(agg, (op == 1u || op == 2u) ? 2u * i + 3u : (head ? 2u * i + 2u : 0u));
        }
        uint32_t most;
        block_excl_max<kApThreads>(agg, s_tmp, &most);
        if (most) return most;
    }
    return 0;
}

// kSmall: a batch from k_rank_locate, whose storage-layer state is kept per query instead of
// per distinct key.
template <bool kSmall>
__global__ void __launch_bounds__(kApThreads, 2) k_apply(ApplyArgs a, RebuildArgs rb, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_tmp[33];
    __shared__ uint32_t s_tile, s_last, s_base[2];
    __shared__ int s_fail;
    __shared__ int32_t s_delta[kLevelSlots];
    __shared__ int32_t s_tomb;
    __shared__ uint32_t s_changes, s_dirty;
    __shared__ uint32_t s_chist[kLevelSlots];  // built-level membership changes by height

    const int tid = threadIdx.x;
    if (tid == 0) {
        s_tile = atomicAdd(&a.bm->tile_ctr[kCtrApply], 1u);  // tiles in the order CTAs start
        s_fail = 0;
    }
    if (block_sees_error(&a.m->error)) return;
    const uint32_t n = a.n;
    const uint32_t qv = n - a.bm->invalid;
    const uint32_t cur = a.m->cur;
    const uint32_t Lb = a.m->Lb;  // lowest built index level: changes below it leave the index alone
    uint64_t* SV = a.st.vals[cur];
    uint8_t* SM = a.st.meta[cur];
    const uint32_t tile = s_tile, ntiles = gridDim.x;
    if (tid < kLevelSlots) {
        s_delta[tid] = 0;
        s_chist[tid] = 0;
    }
    if (tid == 0) {
        s_tomb = 0;
        s_changes = 0;
        s_dirty = 0;
    }
    const uint32_t base = tile * kApplyTile + tid * kItems;

    uint64_t key[kItems];
    uint32_t pay[kItems];
    uint32_t e[kItems];
    uint32_t dres[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t i = base + k;
        key[k] = i < qv ? a.sk[i] : kMaxKey;
        pay[k] = i < n ? a.sp[i] : 0u;
    }
    const uint64_t kprev = (base > 0 && base - 1 < qv) ? a.sk[base - 1] : kMaxKey;
    const uint64_t knext = (base + kItems < qv) ? a.sk[base + kItems] : kMaxKey;
    // the descent's prefixes for this tile (its markers' maximum before it, the dense
    // index of its first local run head), loaded with the batch (a block barrier below
    // would keep them from being hoisted)
    uint32_t tpref = kSmall ? 0u : a.tile_pref[tile];
    const uint32_t dbase = kSmall ? 0u : a.sub_pref[tile * (kApplyTile / kSubTile)];
    if (kSmall) {
        const uint32_t tb = tile * kApplyTile;
        if (tb > 0 && tb < qv && a.sk[tb] == a.sk[tb - 1]) tpref = marker_before(a, tb, s_tmp);
    }
    uint32_t agg = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t i = base + k;
        const bool valid = i < qv;
        const uint64_t prev = k ? key[k - 1] : kprev;
        const bool head = valid && (i == 0 || key[k] != prev);
        const uint32_t op = pay[k] >> 30;
        const bool write = valid && (op == 1u || op == 2u);
        e[k] = write ? 2u * i + 3u : (head ? 2u * i + 2u : 0u);
        agg = max(agg, e[k]);
    }
    const uint32_t texcl = block_excl_max<kApThreads>(agg, s_tmp, nullptr);
    uint32_t M = max(tpref, texcl);
    // dense index of each query's local run head: the tile's first one plus the local
    // heads before it in the tile (a local head is a run head or a 256-query sub-tile's
    // first query, as the descent counted them)
    uint32_t lh = 0, nh = 0, hidx = 0;
    if (!kSmall) {
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t i = base + k;
            const uint64_t prev = k ? key[k - 1] : kprev;
            const bool local = i < qv && (i == 0 || key[k] != prev || (i % kSubTile) == 0);
            lh |= (local ? 1u : 0u) << k;
            nh += local ? 1u : 0u;
        }
        hidx = dbase + block_excl_sum<kApThreads>(nh, s_tmp, nullptr);  // dense index of the next head
    }
    uint32_t new_here = 0, new_mask = 0, chg_here = 0, chg_mask = 0;
    // Per query: its run head's result index, and the gathers of its prior state, all
    // issued before any store so that their latencies overlap: the run head's state, or,
    // when an earlier query of its run wrote (the marker names it), that query's payload.
    uint32_t fromw = 0, insw = 0, flx = 0;  // bit k: from an earlier write; that write inserts; flags
    uint64_t val[kItems];
    uint32_t pj[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t mex = M;
        const uint32_t minc = max(M, e[k]);
        M = minc;
        e[k] = minc;  // keep the inclusive value for the owners and the new-node pass
        dres[k] = kSmall ? base + k : hidx + ((lh >> k) & 1u) - 1u;  // this query's run head's result
        hidx += (lh >> k) & 1u;
        const uint64_t prev = k ? key[k - 1] : kprev;
        const bool q = base + k < qv;
        const bool fw = q && (base + k != 0 && key[k] == prev) && (mex & 1u);
        fromw |= (fw ? 1u : 0u) << k;
        flx |= (q ? (uint32_t)a.flags[dres[k]] : 0u) << (2 * k);
        val[k] = q ? a.val0[dres[k]] : 0ull;
        pj[k] = fw ? a.sp[(mex - 3u) >> 1] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        if (!((fromw >> k) & 1u)) {
            if (!((flx >> (2 * k + 1)) & 1u)) val[k] = 0ull;  // the run head's key is not live
            continue;
        }
        const bool ins = (pj[k] >> 30) == 1u;
        insw |= (ins ? 1u : 0u) << k;
        val[k] = ins ? a.uvals[pj[k] & kSeqMask] : 0ull;
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t i = base + k;
        if (i >= n) continue;
        const uint32_t seq = pay[k] & kSeqMask;
        if (i >= qv) {
            store_result(a.results, seq, 0ull, PI_R_INVALID);
            continue;
        }
        const uint32_t dj = dres[k];
        const bool exists = (flx >> (2 * k)) & 1u, live0 = (flx >> (2 * k + 1)) & 1u;
        const bool pl = ((fromw >> k) & 1u) ? ((insw >> k) & 1u) != 0 : live0;
        store_result(a.results, seq, val[k], pl ? PI_R_PRESENT : PI_R_ABSENT);

        const uint64_t next = (k + 1 < kItems) ? key[k + 1] : knext;
        const bool last = next != key[k];
        const uint32_t minc = e[k];
        if (!last || !(minc & 1u)) continue;  // not the owner, or the run never writes
        const uint32_t jw = (minc - 3u) >> 1;
        const uint32_t pw = (jw == i) ? pay[k] : a.sp[jw];
        const bool fin_live = (pw >> 30) == 1u;
        if (exists) {
            const uint32_t r = a.loc[dj] - 1u;
            if (a.wcount) atomicAdd(&a.wcount[r], 1u);
            const uint8_t mt = SM[r];
            const uint32_t h = mt & kHeightMask;
            if (fin_live) {
                SV[r] = a.uvals[pw & kSeqMask];
                SM[r] = (uint8_t)h;
            } else {
                SM[r] = (uint8_t)(h | kTomb);
            }
            if (fin_live != live0) {
                atomicAdd(&s_tomb, fin_live ? -1 : 1);
                atomicAdd(&s_changes, 1u);
                atomicAdd(&s_delta[1], fin_live ? 1 : -1);
                for (uint32_t l = 2; l <= h; ++l) {
                    atomicAdd(&s_delta[l], fin_live ? 1 : -1);
                    // the rebuild's per-tile count of the node's 4096-node tile
                    atomicAdd(&a.lcnt[(size_t)(l - 2) * a.lstride + (r >> 12)], fin_live ? 1u : 0xFFFFFFFFu);
                }
                if (h >= Lb) {
                    s_dirty = 1;
                    chg_here++;
                    chg_mask |= 1u << k;
                }
            }
        } else if (fin_live) {
            new_here++;
            new_mask |= 1u << k;
        }
    }
    // Places of the tile's new nodes and level changes. Warp 0 looks back over the new
    // nodes' counts, warp 1 over the changes'. A tile without any publishes its zero and goes
    // on, but for every 64th, so that a look-back finds a prefix within two rounds.
    uint32_t tile_new = 0, tile_chg = 0, slot = 0, cslot = 0;
    if (__syncthreads_or(new_here != 0)) slot = block_excl_sum<kApThreads>(new_here, s_tmp, &tile_new);
    if (__syncthreads_or(chg_here != 0)) cslot = block_excl_sum<kApThreads>(chg_here, s_tmp, &tile_chg);
    if (tid < 64) {
        const uint32_t c = tid < 32 ? tile_new : tile_chg;
        uint64_t* desc = a.desc + (tid < 32 ? 0u : ntiles);
        if (c || (tile & 63u) == 0) {
            bool ok = true;
            const uint32_t ex = lookback_warp_wide<false, 8>(desc, tile, epoch, c, a.err, &ok);
            if ((tid & 31) == 0) {
                s_base[tid >> 5] = ex;
                if (!ok) s_fail = 1;
            }
        } else if ((tid & 31) == 0) {
            lookback_publish(desc, tile, epoch, 0u);
        }
    }
    if (tile_new || tile_chg) {
        __syncthreads();
        if (s_fail) return;
    }
    if (new_mask) {
        uint32_t o = s_base[0] + slot;
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (!(new_mask & (1u << k))) continue;
            const uint32_t i = base + k;
            const uint32_t jw = (e[k] - 3u) >> 1;
            const uint32_t pw = (jw == i) ? pay[k] : a.sp[jw];
            const uint32_t h = tower_height(key[k], a.hp);
            a.nn.keys[o] = key[k];
            a.nn.vals[o] = a.uvals[pw & kSeqMask];
            a.nn.loc[o] = a.loc[dres[k]];
            a.nn.height[o] = (uint8_t)h;
            ++o;
            atomicAdd(&s_changes, 1u);
            atomicAdd(&s_delta[1], 1);
            for (uint32_t l = 2; l <= h; ++l) atomicAdd(&s_delta[l], 1);
            if (h >= 2) s_dirty = 1;
        }
    }
    // Built-level membership changes, for an incremental rebuild.
    if (chg_mask) {
        uint32_t o = s_base[1] + cslot;
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (!(chg_mask & (1u << k))) continue;
            const uint32_t r = a.loc[dres[k]] - 1u;
            const uint8_t mt = SM[r];  // as this kernel left it
            const uint32_t h = mt & kHeightMask;
            a.chg.keys[o] = key[k];
            a.chg.pos[o] = r;
            a.chg.hl[o] = (uint8_t)(h | ((mt & kTomb) ? 0u : 0x80u));
            ++o;
            atomicAdd(&s_chist[h < (uint32_t)kLevelSlots ? h : kLevelSlots - 1], 1u);
        }
    }
    __syncthreads();
    if (tid < kLevelSlots && s_chist[tid]) atomicAdd(&a.bm->chg_hist[tid], s_chist[tid]);
    if (tid < kLevelSlots && s_delta[tid]) atomicAdd(&a.bm->delta[tid], s_delta[tid]);
    if (tid == 64) {
        if (s_tomb) atomicAdd(&a.bm->tomb_delta, s_tomb);
        if (s_changes) atomicAdd(&a.bm->changes, s_changes);
        if (s_dirty) atomicOr(&a.bm->index_dirty, 1u);
        if (tile_new) atomicAdd(&a.bm->new_count, tile_new);
        if (tile_chg) atomicAdd(&a.bm->nchg, tile_chg);
    }
    // Arrival: the barrier orders every thread's stores before thread 0's fence, which (being
    // cumulative) releases them before its count; the last CTA then sees all of them.
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.bm->tile_ctr[kCtrApplyDone], 1u) == ntiles - 1u ? 1u : 0u;
        if (s_last) __threadfence();
    }
    __syncthreads();
    if (!s_last || tid >= 32) return;
    const bool merge = merge_needed(a.m, a.bm);
    if (merge) {
        if (tid == 0) a.bm->merged = 1u;  // the merge's kernels end the batch
    } else {
        level_layout(rb, false);
    }
}

// Debug check of single ownership (Section 3.2.4): after k_apply, every storage node
// has been written by at most one query. Counts are summed into DevMeta::owner_writes
// and cleared for the next batch.
__global__ void __launch_bounds__(kThreads) k_owner_check(ApplyArgs a) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_sum;
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    const uint32_t size = a.m->size;
    uint32_t sum = 0;
    for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < size; i += gridDim.x * kThreads) {
        const uint32_t c = a.wcount[i];
        if (c) {
            sum += c;
            if (c > 1u) atomicOr(a.err, kErrOwner);
            a.wcount[i] = 0u;
        }
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&s_sum, sum);
    __syncthreads();
    if (threadIdx.x == 0 && s_sum) atomicAdd(&a.m->owner_writes, s_sum);
}

}  // namespace

cudaError_t launch_apply(const ApplyArgs& a, const RebuildArgs& rb, bool small, uint32_t& epoch, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const uint32_t tiles = (a.n + kApplyTile - 1) / kApplyTile;
    if (small) launch_dep(k_apply<true>, tiles, kApThreads, 0, s, a, rb, ++epoch);
    else launch_dep(k_apply<false>, tiles, kApThreads, 0, s, a, rb, ++epoch);  // tile prefixes come from the descent
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_owner_check(const ApplyArgs& a, cudaStream_t s, int num_sms) {
    if (!a.wcount) return cudaSuccess;
    launch_dep(k_owner_check, (uint32_t)num_sms * 8u, kThreads, 0, s, a);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace pi
