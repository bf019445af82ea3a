// Single ownership and query execution (Algorithms 3 and 4, Section 3.2.4).
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
// The descent left the storage-layer state at each local run head (a query whose key differs
// from the previous one, and the first query of every 128-query block) and each block's
// largest e. A warp takes a block and scans it on its own: the nearest local head before a
// query, by its number, has its state, and a block that continues a run looks back over 256
// blocks' marks, then the groups', for the run's last write: two steps or three however long the
// run is. (Over the blocks' marks alone, a batch that is one key's run took time with the square of its
// length: 2^23 searches 1043 us, now 336.) So no warp waits for another until the counts of the
// tile: with block-wide scans, barriers were the largest stall.
// New nodes, and the changes of built levels' membership, go to their places in key order in
// the same pass: a tile's first place comes from a decoupled look-back over the tiles' counts,
// which only tiles that have some wait for. Half of the kernel's time is its scattered 16-byte
// result stores (2^22 searches: 84 us, and 43 with the results stored in order), the rest its
// chain of dependent reads, so the owners' reads are issued with the results' at each step of
// the chain: 2^22 skewed queries with 10% updates 117 -> 97 us.
// (Staging the new nodes per tile, a scan and a packing kernel were two more launches.)

#include "common.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;
constexpr int kApThreads = 256;         // k_apply: four CTAs per SM at 64 registers
constexpr int kItems = 4;               // sorted queries per thread
constexpr uint32_t kTile = kApThreads * kItems;
static_assert(kApplyTile % kTile == 0 && kTile >= kDescendTile, "the descent's tiles hold whole blocks");
constexpr uint32_t kSeqMask = (1u << 30) - 1u;
static_assert(kApplyBlock == 32u * kItems, "a warp's queries");

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
// has one decides; tile 0 heads the first run). Small batches only: they have no marks, and a
// run crosses few tiles.
__device__ uint32_t marker_before_tile(const ApplyArgs& a, uint32_t tb, uint32_t* s_tmp) {
    while (tb > 0) {
        tb -= kTile;
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

// The nearest nonzero of the last kMarkBlocks of marks[0, n), by a whole warp (four loads at a time:
// with all eight in flight the kernel spilled 44 bytes a thread instead of 12).
__device__ __forceinline__ uint32_t last_mark(const uint32_t* marks, uint32_t n) {
    uint32_t most = 0;  // markers grow with their place, so the largest is the nearest
#pragma unroll 4
    for (uint32_t u = 0; u < kMarkBlocks / 32u; ++u) {
        const uint32_t x = 32u * u + (threadIdx.x & 31u);
        most = max(most, x < n ? marks[n - 1u - x] : 0u);
    }
    return __reduce_max_sync(0xffffffffu, most);
}

// Largest marker before block blk, which continues the run before it: of the blocks before it, or,
// when the first step finds none, of the groups. Those start with the group of the last block not
// looked at: the blocks of it that come after that one were looked at, and hold none. The block
// that is sought is filled up to its end by the run, as is the next one, so its group has its marker.
__device__ __forceinline__ uint32_t marker_before_block(const ApplyArgs& a, uint32_t blk) {
    uint32_t mk = last_mark(a.blk_mark, blk);
    if (mk || blk <= kMarkBlocks) return mk;
#pragma unroll 1
    for (uint32_t n = (blk - 1u) / kMarkBlocks; mk == 0u && n; n = n > kMarkBlocks ? n - kMarkBlocks : 0u)
        mk = last_mark(a.grp_mark, n);
    return mk;
}

// kSmall: a batch from k_rank_locate, whose storage-layer state is kept at every query, and which
// comes without marks.
template <bool kSmall>
__global__ void __launch_bounds__(kApThreads, 4) k_apply(ApplyArgs a, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_tmp[33];
    __shared__ uint32_t s_tile, s_base[2], s_warp[kApThreads / 32];
    __shared__ int s_fail;
    __shared__ int32_t s_delta[kLevelSlots];
    __shared__ int32_t s_tomb;
    __shared__ uint32_t s_changes, s_dirty;
    __shared__ uint32_t s_chist[kLevelSlots];  // built-level membership changes by height

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kLevelSlots) {
        s_delta[tid] = 0;
        s_chist[tid] = 0;
    }
    if (tid == 0) {
        s_tile = atomicAdd(&a.bm->tile_ctr[kCtrApply], 1u);  // tiles in the order CTAs start
        s_fail = 0;
        s_tomb = 0;
        s_changes = 0;
        s_dirty = 0;
    }
    if (block_sees_error(&a.m->error)) return;
    const uint32_t n = a.n;
    const uint32_t qv = n - a.bm->invalid;
    const uint32_t cur = a.m->cur;
    const uint32_t Lb = a.m->Lb;  // lowest built index level: changes below it leave the index alone
    uint64_t* SV = a.st.vals[cur];
    uint8_t* SM = a.st.meta[cur];
    const uint32_t tile = s_tile, ntiles = gridDim.x;
    const uint32_t blk = tile * (kTile / kApplyBlock) + (uint32_t)warp;
    const uint32_t base = blk * kApplyBlock + (uint32_t)lane * kItems;

    uint64_t key[kItems];
    uint32_t pay[kItems];
    {  // 16-byte loads; the arrays are padded past the batch
        ulonglong2 k01 = {kMaxKey, kMaxKey}, k23 = {kMaxKey, kMaxKey};
        uint4 p = {0, 0, 0, 0};
        if (base < n) {
            k01 = reinterpret_cast<const ulonglong2*>(a.sk + base)[0];
            k23 = reinterpret_cast<const ulonglong2*>(a.sk + base)[1];
            p = *reinterpret_cast<const uint4*>(a.sp + base);
        }
        key[0] = base < qv ? k01.x : kMaxKey;
        key[1] = base + 1u < qv ? k01.y : kMaxKey;
        key[2] = base + 2u < qv ? k23.x : kMaxKey;
        key[3] = base + 3u < qv ? k23.y : kMaxKey;
        pay[0] = p.x;
        pay[1] = p.y;
        pay[2] = p.z;
        pay[3] = p.w;
    }
    uint64_t kprev = __shfl_up_sync(0xffffffffu, key[kItems - 1], 1);
    if (lane == 0) kprev = (base > 0 && base - 1 < qv) ? a.sk[base - 1] : kMaxKey;
    uint64_t knext = __shfl_down_sync(0xffffffffu, key[0], 1);
    if (lane == 31) knext = (base + kItems < qv) ? a.sk[base + kItems] : kMaxKey;
    // the marker before the block, wanted where it continues a run
    uint32_t mark = 0;
    const uint32_t head0 = !kSmall && blk * kApplyBlock < n ? a.blk_head[blk] : 0u;
    if (kSmall) {
        const uint32_t tb = tile * kTile;
        if (tb > 0 && tb < qv && a.sk[tb] == a.sk[tb - 1]) mark = marker_before_tile(a, tb, s_tmp);
    } else if (__shfl_sync(0xffffffffu, base < qv && base > 0 && kprev == key[0], 0)) {
        mark = marker_before_block(a, blk);
    }
    // M: the largest marker before each query; dres: the nearest local head at or before it
    uint32_t e[kItems], dres[kItems];
    uint32_t agg = 0, heads = 0;
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
        heads += head || (valid && i % kApplyBlock == 0) ? 1u : 0u;
        dres[k] = heads;
    }
    uint32_t M;
    if (kSmall) {
        M = max(mark, block_excl_max<kApThreads>(agg, s_tmp, nullptr));
    } else {
        uint32_t x = agg, h = heads;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o), z = __shfl_up_sync(0xffffffffu, h, o);
            if (lane >= o) {
                x = max(x, y);
                h += z;
            }
        }
        x = __shfl_up_sync(0xffffffffu, x, 1);
        M = lane ? max(mark, x) : mark;
        const uint32_t dtile = a.windows ? kApplyTile : kDescendTile;
        h += head0 + base / dtile * dtile - heads - 1u;  // (wraps for a block past the valid queries: not used)
#pragma unroll
        for (int k = 0; k < kItems; ++k) dres[k] += h;
    }
    uint32_t new_here = 0, new_mask = 0, chg_here = 0, chg_mask = 0;
    // Per query, all gathers of a step issued before any store so that their latencies overlap:
    // the run head's state, or, when an earlier query of its run wrote (the marker names it),
    // that query's payload; for the run's owner (its last query, if the run writes) the
    // storage place and the payload of the run's last write.
    uint32_t fromw = 0, insw = 0, flx = 0, own = 0;  // bit k: from an earlier write; that write inserts; flags; owner
    uint64_t val[kItems];
    uint32_t pj[kItems], pw[kItems], at[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t i = base + k;
        if (kSmall) dres[k] = i;
        const uint32_t mex = M;
        const uint32_t minc = max(M, e[k]);
        M = minc;
        const uint64_t prev = k ? key[k - 1] : kprev, next = (k + 1 < kItems) ? key[k + 1] : knext;
        const bool q = i < qv;
        const bool fw = q && (i != 0 && key[k] == prev) && (mex & 1u);
        const bool ow = q && next != key[k] && (minc & 1u);
        const uint32_t jw = (minc - 3u) >> 1;
        fromw |= (fw ? 1u : 0u) << k;
        own |= (ow ? 1u : 0u) << k;
        flx |= (q ? (uint32_t)a.flags[dres[k]] : 0u) << (2 * k);
        val[k] = q ? a.val0[dres[k]] : 0ull;
        pj[k] = fw ? a.sp[(mex - 3u) >> 1] : 0u;
        at[k] = ow ? a.loc[dres[k]] : 0u;
        pw[k] = !ow ? 0u : (jw == i ? pay[k] : a.sp[jw]);
    }
    uint64_t nv[kItems];  // the owner's new value
    uint32_t mt[kItems];  // its node's state byte
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const bool ow = (own >> k) & 1u, exists = (flx >> (2 * k)) & 1u;
        nv[k] = ow && (pw[k] >> 30) == 1u ? a.uvals[pw[k] & kSeqMask] : 0ull;
        mt[k] = ow && exists ? SM[at[k] - 1u] : 0u;
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
        const bool exists = (flx >> (2 * k)) & 1u, live0 = (flx >> (2 * k + 1)) & 1u;
        const bool pl = ((fromw >> k) & 1u) ? ((insw >> k) & 1u) != 0 : live0;
        store_result(a.results, seq, val[k], pl ? PI_R_PRESENT : PI_R_ABSENT);
        if (!((own >> k) & 1u)) continue;
        const bool fin_live = (pw[k] >> 30) == 1u;
        if (exists) {
            const uint32_t r = at[k] - 1u;
            if (a.wcount) atomicAdd(&a.wcount[r], 1u);
            const uint32_t h = mt[k] & kHeightMask;
            if (fin_live) SV[r] = nv[k];
            if (fin_live != live0) {
                SM[r] = (uint8_t)(h | (fin_live ? 0u : kTomb));
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
                    mt[k] = h | (fin_live ? 0x80u : 0u);  // as the change list has it
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
    uint32_t both = new_here | (chg_here << 16), incl = both;  // a tile's counts stay below 2^16
    if (__any_sync(0xffffffffu, both != 0)) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    const uint32_t wc = lane < kApThreads / 32 ? s_warp[lane] : 0u;
    const uint32_t tot = __reduce_add_sync(0xffffffffu, wc);
    const uint32_t wb = __reduce_add_sync(0xffffffffu, lane < warp ? wc : 0u) + incl - both;
    const uint32_t tile_new = tot & 0xFFFFu, tile_chg = tot >> 16;
    if (tid < 64) {
        const uint32_t c = tid < 32 ? tile_new : tile_chg;
        uint64_t* desc = a.desc + (tid < 32 ? 0u : ntiles);
        if (c || (tile & 63u) == 0) {
            bool ok = true;
            const uint32_t ex = lookback_warp_wide<8>(desc, tile, epoch, c, a.err, &ok);
            if (lane == 0) {
                s_base[tid >> 5] = ex;
                if (!ok) s_fail = 1;
            }
        } else if (lane == 0) {
            lookback_publish(desc, tile, epoch, 0u);
        }
    }
    if (!tot && !s_changes) return;  // block-uniform: no node came, went or changed its state
    __syncthreads();
    if (s_fail) return;
    if (new_mask) {
        uint32_t o = s_base[0] + (wb & 0xFFFFu);
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (!(new_mask & (1u << k))) continue;
            const uint32_t h = tower_height(key[k], a.hp);
            a.nn.keys[o] = key[k];
            a.nn.vals[o] = nv[k];
            a.nn.loc[o] = at[k];
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
        uint32_t o = s_base[1] + (wb >> 16);
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (!(chg_mask & (1u << k))) continue;
            const uint32_t h = mt[k] & kHeightMask;
            a.chg.keys[o] = key[k];
            a.chg.pos[o] = at[k] - 1u;
            a.chg.hl[o] = (uint8_t)mt[k];
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

cudaError_t launch_apply(const ApplyArgs& a, bool small, uint32_t& epoch, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    const uint32_t tiles = (a.n + kTile - 1) / kTile;
    if (small) launch_dep(k_apply<true>, tiles, kApThreads, 0, s, a, ++epoch);
    else launch_dep(k_apply<false>, tiles, kApThreads, 0, s, a, ++epoch);
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
