// Storage-layer merge and index-layer rebuild (Sections 4.1 and 4.4.4), plus the
// bulk build of a new index (Section 3.1) and the test-support export.
//
// Storage layer: contiguous sorted arrays keys / vals / meta (meta = height | F_del),
// double buffered. A delete only sets F_del (Algorithm 4), so a deleted node keeps its
// place and a later insert of the same key revives it in place. The storage layer is
// re-laid-out (merge) only when new nodes must be placed, or when delete-flagged nodes
// exceed 1/8 of it; the merge drops every delete-flagged node.
//
// Rebuild: the paper's daemon scans the storage layer and puts the key of every
// valid node of height > 1 into the index-layer arrays. Here one pass over the storage
// layer does it for all levels at once: per tile of 4096 nodes, the state bytes arrive in
// shared memory by TMA bulk copy, and level by level the tile compacts its nodes of
// height >= l (a prefix sum), gathers their keys and writes them with their down pointers, from
// the tile's offset in the level on. The offsets are a scan of the tiles' counts, which the kernels that change
// the nodes keep current.
//
// Level sizes are not counted by the rebuild: the apply kernel keeps them current as
// deltas, so the layout (level bases, sentinels) is known before the pass and the pass writes
// every entry exactly once.

#include <cstddef>

#include "layout.cuh"
#include "relevel.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;
constexpr int kNodes = 4096;             // storage nodes per tile
constexpr int kPer = kNodes / kThreads;  // 16 per thread
constexpr uint32_t kCtrMerge = 9, kCtrMergeDone = 10, kCtrCreate = 11, kCtrRebuild = 16, kCtrPrep = 17;

// ---------------------------------------------------------------------------------
// Merge: old live nodes + new nodes -> the other storage buffer, in key order. A new node with
// loc = x goes right before old node x.
//
// The merged sequence (size old positions and the new nodes between them) is cut into chunks of
// kChunk elements, so every chunk is the same work however the new nodes fall: cut by old
// positions, a batch that appends its keys at the end left them all to one CTA. New node j sits
// at position loc[j] + j of the sequence, so the cut at d has the new nodes with
// loc[j] + j < d before it, which a warp finds 32 probes a round. Each CTA takes consecutive chunks:
//   1. its cuts, all at once by its warps, and the live nodes among its old ones (no read when
//      nothing is delete-flagged); a look-back over the CTAs, numbered in the order they
//      start, gives its first output place;
//   2. per chunk, whose old nodes arrive in shared memory by TMA bulk copies one chunk ahead,
//      a blocked pass over the state bytes and the new nodes' insertion points gives every
//      position its output offset, and a striped pass writes the live nodes, coalesced.
// The pass also counts, per output tile, the nodes of each built level (the rebuild's offsets
// come from these), so nothing reads the new meta bytes again for them. A tile's counts are
// cleared by the CTA whose chunks reach the tile's start, before that CTA publishes: outputs
// never lie beyond their place in the sequence, so whoever adds to a tile has looked back past
// that publication. The CTA that finishes last lays out the levels; a batch that needs no merge
// has that done by the first CTA.
// Bound by HBM: 17 B read and 17 B written per node. With plain loads, issued and waited for
// within the chunk, the copy ran at 42% of the memory rate, its warps waiting for loads and at
// barriers; the copies ahead take the loads out of the chunk, and three barriers are left in it,
// whose waits the other three CTAs of the SM fill. 2^18 new keys spread over 17.3 M nodes 187 ->
// 140 us (100 at the copy rate); 78,000 keys appended to 4.2 M 89 -> 58.
constexpr uint32_t kMergeTile = 1280;              // positions of a chunk's tile
constexpr uint32_t kChunk = kMergeTile - 32;       // 15 positions of alignment and the slot after the last fit
constexpr uint32_t kCuts = 256;                    // cuts found at once
constexpr int kMergePer = (int)kMergeTile / kThreads;
constexpr int kStages = 2;

struct MergeStage {
    uint64_t keys[kMergeTile];
    uint64_t vals[kMergeTile];
    uint8_t meta[kMergeTile];
};
struct MergeSmem {
    MergeStage st[kStages];
    // per position: its new nodes' last one in the chunk, plus one; then live old nodes before it |
    // new nodes at or before it << 16
    // (two, so that one is cleared while the other is read)
    uint32_t off[2][kMergeTile];
};

__global__ void __launch_bounds__(kThreads, 4) k_merge(RebuildArgs a, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) uint8_t s_dyn[];
    MergeSmem& S = *reinterpret_cast<MergeSmem*>(s_dyn);
    __shared__ __align__(8) uint64_t s_bar[kStages];
    __shared__ uint32_t s_cut[kCuts + 1], s_cnt[2][kLevelSlots], s_warp[kThreads / 32], s_new[kThreads / 32];
    __shared__ uint32_t s_cta, s_pref, s_last;
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DevMeta* m = a.m;
    if (!merge_needed(a.bm)) {  // the storage layer stays: this only ends the batch
        if (blockIdx.x == 0 && warp == 0) {
            level_layout(a, false);
            post_batch(a);
        }
        return;
    }
    if (tid == 0) {
        s_cta = atomicAdd(&a.bm->tile_ctr[kCtrMerge], 1u);
        s_fail = 0;
        for (int k = 0; k < kStages; ++k) mbar_init(&s_bar[k], 1);
    }
    if (tid < 2 * kLevelSlots) (&s_cnt[0][0])[tid] = 0;
    // A CTA that stops for an error is not counted as finished, so no other may be the last: each
    // of them posts, or the host would read whatever the slot held before.
    if (block_sees_error(&m->error)) {
        if (warp == 0) post_batch(a);
        return;
    }
    const uint32_t size = m->size, src = m->cur, dst = src ^ 1u;
    const uint32_t newc = a.bm->new_count, cta = s_cta, G = gridDim.x;
    const bool flagged = (int32_t)m->tombs + a.bm->tomb_delta != 0;
    const uint64_t* K0 = a.st.keys[src];
    const uint64_t* V0 = a.st.vals[src];
    const uint8_t* M0 = a.st.meta[src];
    uint64_t* K1 = a.st.keys[dst];
    uint64_t* V1 = a.st.vals[dst];
    uint8_t* M1 = a.st.meta[dst];
    const uint32_t W = size + newc;  // at most PI_MAX_KEYS plus a batch
    const uint32_t nch = (W + kChunk - 1) / kChunk;
    const uint32_t c0 = (uint32_t)((uint64_t)nch * cta / G), c1 = (uint32_t)((uint64_t)nch * (cta + 1u) / G);
    const uint32_t d0 = min(c0 * kChunk, W), d1 = min(c1 * kChunk, W);
    const uint32_t lmin = a.min_lb > 2u ? a.min_lb : 2u;
    // clear the counts of the output tiles that start in [d0, d1)
    {
        const uint32_t t0 = (d0 + kNodes - 1) / kNodes, t1 = (d1 + kNodes - 1) / kNodes;
        for (uint32_t l = lmin + (uint32_t)warp; l < (uint32_t)kLevelSlots; l += kThreads / 32)
            for (uint32_t t = t0 + (uint32_t)lane; t < t1; t += 32u) a.lcnt[(size_t)(l - 2) * a.lstride + t] = 0u;
    }
    // cuts: new nodes before diagonal d
    auto find_cuts = [&](uint32_t c, uint32_t count) {
        for (uint32_t k = (uint32_t)warp; k < count; k += kThreads / 32) {
            const uint32_t d = min((c + k) * kChunk, W);
            uint32_t lo = d > size ? d - size : 0u, hi = min(newc, d);  // the count lies in [lo, hi]
            while (lo < hi) {
                const uint32_t step = (hi - lo + 31u) / 32u, p = lo + (uint32_t)lane * step;
                const bool before = p < hi && a.nn.loc[p] + p < d;
                const uint32_t n = (uint32_t)__popc(__ballot_sync(0xffffffffu, before));  // a prefix
                if (n == 0) break;
                if (n < 32u) hi = min(hi, lo + n * step);
                lo += (n - 1u) * step + 1u;
            }
            if (lane == 0) s_cut[k] = lo;
        }
    };
    // one thread: the old nodes of chunk c, whose cut is s_cut[k], into its stage
    auto fetch = [&](uint32_t c, uint32_t k) {
        const uint32_t xal = (min(c * kChunk, W) - s_cut[k]) & ~15u;
        MergeStage& T = S.st[(c - c0) % kStages];
        uint64_t* bar = &s_bar[(c - c0) % kStages];
        mbar_arrive_expect_tx(bar, kMergeTile * 17u);
        // the storage arrays are padded by more than a tile past the last node
        bulk_g2s(T.keys, K0 + xal, kMergeTile * 8u, bar);
        bulk_g2s(T.vals, V0 + xal, kMergeTile * 8u, bar);
        bulk_g2s(T.meta, M0 + xal, kMergeTile, bar);
    };
    uint32_t live = 0;
    if (c1 > c0) {
        // the CTA's old positions [x0, x1)
        const uint32_t nc = min(kCuts, c1 - c0);
        find_cuts(c0, nc + 1u);
        __syncthreads();
        const uint32_t x0 = d0 - s_cut[0];
        uint32_t x1 = d1 - s_cut[nc];
        if (c1 - c0 > kCuts) {  // the last cut lies past the first group
            const uint32_t first = s_cut[0];
            __syncthreads();
            find_cuts(c1, 1u);
            __syncthreads();
            x1 = d1 - s_cut[0];
            __syncthreads();
            if (tid == 0) s_cut[0] = first;
            __syncthreads();
        }
        if (tid == 0)  // the first chunks arrive while the CTA counts and looks back
            for (uint32_t k = 0; k < (uint32_t)kStages && c0 + k < c1; ++k) fetch(c0 + k, k);
        if (flagged) {
            for (uint32_t b = (x0 & ~15u) + 16u * (uint32_t)tid; b < x1; b += 64u * kThreads) {
                uint4 mw[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {  // (bytes past x1 count as flagged)
                    const uint32_t p = b + 16u * kThreads * (uint32_t)u;
                    mw[u] = p < x1 ? *reinterpret_cast<const uint4*>(M0 + p) : make_uint4(~0u, ~0u, ~0u, ~0u);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t p = b + 16u * kThreads * (uint32_t)u;
                    const uint32_t words[4] = {mw[u].x, mw[u].y, mw[u].z, mw[u].w};
                    if (p >= x0 && p + 16u <= x1) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) live += (uint32_t)__popc(~words[k] & 0x80808080u);
                    } else {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const uint32_t mt = (words[k >> 2] >> (8 * (k & 3))) & 0xFFu;
                            live += (p + k >= x0 && p + k < x1 && !(mt & kTomb)) ? 1u : 0u;
                        }
                    }
                }
            }
        } else if (tid == 0) {
            live = x1 - x0;
        }
    }
    live = __reduce_add_sync(0xffffffffu, live);
    if (lane == 0) s_warp[warp] = live;
    __syncthreads();  // (also orders every thread's clears before warp 0's fence)
    live = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) live += s_warp[w];
    if (warp == 0) {
        __threadfence();
        bool ok = true;
        const uint32_t ex = lookback_warp_wide<8>(a.desc, cta, epoch, live, a.err, &ok);
        __threadfence();
        if (lane == 0) {
            s_pref = ex;
            if (!ok) s_fail = 1;
        }
    }
    __syncthreads();
    uint32_t lbase = s_pref;  // live old nodes before the chunk
    uint32_t landed = 0;      // chunks whose copies have been waited for
#pragma unroll
    for (int k = 0; k < kMergePer; ++k) S.off[0][(uint32_t)tid + k * kThreads] = 0u;
    __syncthreads();
    uint32_t fl_tile = 0;
    bool fl = false;
    auto flush = [&]() {  // the counts of the last chunk's two output tiles
        if (!fl || tid >= 2 * kLevelSlots) return;
        const uint32_t side = tid >= kLevelSlots ? 1u : 0u, l = (uint32_t)tid - side * kLevelSlots;
        const uint32_t v = s_cnt[side][l];
        if (v) {
            atomicAdd(&a.lcnt[(size_t)(l - 2) * a.lstride + fl_tile + side], v);
            s_cnt[side][l] = 0;
        }
    };
    for (uint32_t c = c0; c < c1 && !s_fail; ++c) {
        const uint32_t ck = (c - c0) % kCuts;
        if (ck == 0 && c != c0) {  // the next group's cuts; nothing is in flight here
            __syncthreads();
            find_cuts(c, min(kCuts, c1 - c) + 1u);
            __syncthreads();
            if (tid == 0)
                for (uint32_t k = 0; k < (uint32_t)kStages && c + k < c1; ++k) fetch(c + k, k);
        }
        uint32_t* off = S.off[(c - c0) & 1u];
        uint32_t* off_next = S.off[((c - c0) & 1u) ^ 1u];
        MergeStage& T = S.st[(c - c0) % kStages];
        const uint32_t da = c * kChunk, db = min(da + kChunk, W);
        const uint32_t ja = s_cut[ck], jb = s_cut[ck + 1], xa = da - ja, xb = db - jb;
        const uint32_t xal = xa & ~15u, sh = xa - xal, end = xb - xal;  // positions [sh, end) of the tile at xal
        // the chunk's new nodes, kMergePer per thread: their insertion points, and whether each is
        // the last one there
        uint32_t nx[kMergePer], last = 0;
#pragma unroll
        for (int k = 0; k < kMergePer; ++k) {
            const uint32_t j = ja + (uint32_t)tid + k * kThreads;
            nx[k] = j < jb ? a.nn.loc[j] - xal : ~0u;
            if (j < jb && (j + 1u == jb || a.nn.loc[j + 1u] - xal != nx[k])) last |= 1u << k;
            if (j < jb && (nx[k] < sh || nx[k] > end)) {
                atomicOr(a.err, kErrBounds);
                nx[k] = ~0u;
            }
        }
        if (!mbar_wait_bounded(&s_bar[(c - c0) % kStages], ((c - c0) / kStages) & 1u, a.err)) s_fail = 1;
#pragma unroll
        for (int k = 0; k < kMergePer; ++k)
            if (((last >> k) & 1u) && nx[k] != ~0u) off[nx[k]] = (uint32_t)tid + k * kThreads + 1u;
        __syncthreads();
        if (s_fail) break;
        ++landed;
        // every thread has left the chunk before: its stage and offsets are free
        if (tid == 0 && ck > 0 && c + 1u < c1 && ck + 1u < kCuts) fetch(c + 1u, ck + 1u);
#pragma unroll
        for (int k = 0; k < kMergePer; ++k) off_next[(uint32_t)tid + k * kThreads] = 0u;
        flush();  // the chunk before's counts; this one's are added two barriers later
        const uint32_t b0 = (uint32_t)tid * kMergePer;
        uint32_t live_bits = 0, nat[kMergePer], lc = 0, nm = 0;
#pragma unroll
        for (int k = 0; k < kMergePer; ++k) {
            const bool lv = b0 + k >= sh && b0 + k < end && !(T.meta[b0 + k] & kTomb);
            live_bits |= (lv ? 1u : 0u) << k;
            lc += lv ? 1u : 0u;
            nm = max(nm, off[b0 + k]);
            nat[k] = nm;
        }
        uint32_t il = lc, in = nm;  // sums of live nodes, maxima of the new nodes' numbers
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, il, o), z = __shfl_up_sync(0xffffffffu, in, o);
            if (lane >= o) {
                il += y;
                in = max(in, z);
            }
        }
        if (lane == 31) {
            s_warp[warp] = il;
            s_new[warp] = in;
        }
        uint32_t el = il - lc, en = __shfl_up_sync(0xffffffffu, in, 1);
        if (lane == 0) en = 0;
        __syncthreads();
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            if (w < warp) {
                el += s_warp[w];
                en = max(en, s_new[w]);
            }
            tot += s_warp[w];
        }
#pragma unroll
        for (int k = 0; k < kMergePer; ++k) {
            off[b0 + k] = el | (max(en, nat[k]) << 16);
            el += (live_bits >> k) & 1u;
        }
        __syncthreads();
        const uint32_t out = lbase + ja, tile0 = out / kNodes;
        lbase += tot;
        auto count = [&](uint32_t h, uint32_t o) {  // a node of a built level, at output o
            const uint32_t side = o / kNodes - tile0;  // a chunk's outputs lie in two tiles
            for (uint32_t l = lmin; l <= h; ++l) atomicAdd(&s_cnt[side & 1u][l], 1u);
        };
#pragma unroll
        for (int k = 0; k < kMergePer; ++k) {
            const uint32_t p = (uint32_t)tid + k * kThreads;
            const uint32_t mt = T.meta[p];
            if (p < sh || p >= end || (mt & kTomb)) continue;
            const uint32_t v = off[p];
            const uint32_t o = out + (v & 0xFFFFu) + (v >> 16);
            if (o >= a.st_cap) {
                atomicOr(a.err, kErrBounds);
                continue;
            }
            K1[o] = T.keys[p];
            V1[o] = T.vals[p];
            M1[o] = (uint8_t)mt;
            if (mt >= lmin) count(mt, o);
        }
        // the chunk's new nodes, before the old node at their position, their loads issued together
        if (jb > ja) {
            uint64_t kv[kMergePer], vv[kMergePer];
            uint32_t hv[kMergePer];
#pragma unroll
            for (int k = 0; k < kMergePer; ++k) {
                const uint32_t j = ja + (uint32_t)tid + k * kThreads;
                const bool in = nx[k] != ~0u;
                kv[k] = in ? a.nn.keys[j] : 0ull;
                vv[k] = in ? a.nn.vals[j] : 0ull;
                hv[k] = in ? a.nn.height[j] : 0u;
            }
#pragma unroll
            for (int k = 0; k < kMergePer; ++k) {
                if (nx[k] == ~0u) continue;
                const uint32_t o = out + (off[nx[k]] & 0xFFFFu) + (uint32_t)tid + k * kThreads;
                if (o >= a.st_cap) {
                    atomicOr(a.err, kErrBounds);
                    continue;
                }
                K1[o] = kv[k];
                V1[o] = vv[k];
                M1[o] = (uint8_t)hv[k];
                if (hv[k] >= lmin) count(hv[k], o);
            }
        }
        // (s_cnt's adds: flushed after the next chunk's first barrier)
        fl_tile = tile0;
        fl = true;
    }
    __syncthreads();
    flush();
    if (s_fail) {  // nor is this one; its copies land first
        if (tid == 0)
            for (uint32_t k = 0; k < (uint32_t)kStages && c0 + landed + k < c1; ++k) {
                const uint32_t f = landed + k;
                mbar_wait_bounded(&s_bar[f % kStages], (f / kStages) & 1u, a.err);
            }
        if (warp == 0) post_batch(a);
        return;
    }
    if (tid == 0 && c1 > c0 && lbase - s_pref != live) atomicOr(a.err, kErrBounds);  // the two counts agree
    __syncthreads();  // every store of the CTA before its arrival is counted
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.bm->tile_ctr[kCtrMergeDone], 1u) == G - 1u ? 1u : 0u;
        if (s_last) __threadfence();
    }
    __syncthreads();
    if (s_last && warp == 0) {
        level_layout(a, true);
        post_batch(a);
    }
}

// The level layout of a bulk build (a batch's is done by the kernel that ends the batch).
__global__ void __launch_bounds__(32) k_level_layout(RebuildArgs a) {
    pdl_wait();
    pdl_trigger();
    level_layout(a, false);
}

// ---------------------------------------------------------------------------------
// Index-layer rebuild over tiles of 4096 storage nodes.
//   lcnt[(l - 2) * stride + tile] = live nodes of height >= l in the tile, for every
//   level l >= 2. The apply kernel keeps these counts current (its owners add or
//   remove one node per liveness change) and a merge counts what it writes, so they are
//   recounted from the state bytes only at create or after a capacity change;
//   prep:  per level, the exclusive prefix of the counts over tiles, in chunks, into
//          loff[(l - Lb) * ntiles + tile] (scan_counts);
//   write: the levels (k_rebuild_write).
__global__ void __launch_bounds__(256) k_rebuild_count(RebuildArgs a) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DevMeta* m = a.m;
    if (*(volatile const uint32_t*)&m->error) return;  // no barrier in this kernel
    if (!a.bm->rebuild || a.bm->merged || !a.force_rebuild) return;  // the merge counts what it writes
    const uint32_t size = m->size, cur = m->cur;
    const uint32_t ntiles = (size + kNodes - 1) / kNodes;
    for (uint32_t tile = blockIdx.x * 8u + (uint32_t)warp; tile < ntiles; tile += gridDim.x * 8u) {
    const uint32_t ts = tile * kNodes;
    const uint32_t cnt = min((uint32_t)kNodes, size - ts);
    const uint8_t* SM = a.st.meta[cur] + ts;
    uint32_t c = 0;  // lane i: nodes of height >= 2 + i
    for (uint32_t it = 0; it < kNodes / 512; ++it) {
        const uint32_t off = it * 512u + (uint32_t)lane * 16u;
        const uint4 w = *reinterpret_cast<const uint4*>(SM + off);  // padded past the end
        const uint32_t words[4] = {w.x, w.y, w.z, w.w};
        uint32_t hs[16];
        uint32_t hm = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t mt = (words[k >> 2] >> (8 * (k & 3))) & 0xFFu;
            hs[k] = (off + k < cnt && !(mt & kTomb)) ? (mt & kHeightMask) : 0u;
            hm = max(hm, hs[k]);
        }
        const uint32_t wm = __reduce_max_sync(0xffffffffu, hm);
        for (uint32_t l = 2; l <= wm; ++l) {
            uint32_t loc = 0;
#pragma unroll
            for (int k = 0; k < 16; ++k) loc += hs[k] >= l ? 1u : 0u;
            const uint32_t tot = __reduce_add_sync(0xffffffffu, loc);
            if ((uint32_t)lane == l - 2) c += tot;
        }
    }
    if (lane < 32 && lane + 2 < kLevelSlots) a.lcnt[(size_t)lane * a.lstride + tile] = c;
    }
}

// Exclusive scan, over tiles, of the tile counts of level Lb + row, in chunks of kScanChunk tiles
// (four per thread of a kB-thread CTA): a chunk gets the sum of the chunks before it by a look-back (the chain is a
// few chunks long). The level's last chunk checks the total against the level size.
template <int kB>
__device__ void scan_counts(const RebuildArgs& a, uint32_t row, uint32_t chunk, uint32_t epoch, uint32_t* s_tmp) {
    __shared__ uint32_t s_prefix;
    __shared__ int s_fine;
    const DevMeta* m = a.m;
    constexpr uint32_t kScanChunk = 4 * kB;
    const uint32_t Lb = m->Lb, l = Lb + row;
    const uint32_t ntiles = (m->size + kNodes - 1) / kNodes;
    const uint32_t nchunks = (ntiles + kScanChunk - 1) / kScanChunk;
    const uint32_t* c = a.lcnt + (size_t)(l - 2) * a.lstride;
    uint32_t* o = a.loff + (size_t)row * ntiles;
    const uint32_t t0 = chunk * kScanChunk + threadIdx.x * 4u;
    uint32_t v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = t0 + k < ntiles ? c[t0 + k] : 0u;
        sum += v[k];
    }
    uint32_t tot;
    uint32_t run = block_excl_sum<kB>(sum, s_tmp, &tot);
    if (threadIdx.x < 32) {
        bool ok;
        // descriptors: a row of nchunks words per level
        const uint32_t ex = lookback_warp(a.desc + (size_t)row * nchunks, chunk, epoch, tot, a.err, &ok);
        if (threadIdx.x == 0) {
            s_prefix = ex;
            s_fine = ok ? 1 : 0;
        }
    }
    __syncthreads();
    if (!s_fine) return;
    run += s_prefix;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (t0 + k < ntiles) o[t0 + k] = run;
        run += v[k];
    }
    if (chunk == nchunks - 1 && threadIdx.x == 0 && s_prefix + tot != m->n[l])
        atomicOr(a.err, kErrBounds);  // counts disagree with the level size
}

// What the writers need first: the scans of the tile counts, or, in an incremental rebuild, a
// change list per level. CTAs of kB threads take these units in turn, each until none is left.
// Returns how many there are.
template <int kB>
__device__ uint32_t prepare_units(const RebuildArgs& a, uint32_t epoch) {
    __shared__ uint32_t s_tmp[33], s_unit;
    const DevMeta* m = a.m;
    BatchMeta* bm = a.bm;
    const bool inc = bm->inc != 0;
    const uint32_t Lb = m->Lb, H = inc && bm->old_H > m->H ? bm->old_H : m->H;
    const uint32_t levels = H >= Lb && m->size ? H - Lb + 1u : 0u;
    const uint32_t ntiles = (m->size + kNodes - 1) / kNodes;
    const uint32_t units = inc ? levels : levels * ((ntiles + 4u * kB - 1u) / (4u * kB));
    for (;;) {
        if (threadIdx.x == 0) s_unit = atomicAdd(&bm->tile_ctr[kCtrRebuild], 1u);
        __syncthreads();
        const uint32_t u = s_unit;
        if (u >= units) return units;
        if (inc) relevel::lists<kB>(a, u, s_tmp);
        else scan_counts<kB>(a, u % levels, u / levels, epoch, s_tmp);  // a level's chunks in order
        __syncthreads();  // the barrier and thread 0's fence release the unit's results
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&bm->tile_ctr[kCtrPrep], 1u);
        }
    }
}

__global__ void __launch_bounds__(1024) k_rebuild_prep(RebuildArgs a, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    if (!a.bm->rebuild) return;
    if (block_sees_error(&a.m->error)) return;
    prepare_units<1024>(a, epoch);
}

// The same inside the writer (kFused): every CTA waits until all units are done, only for units
// that running CTAs have taken, so the wait ends however many CTAs fit the chip at once. It is
// bounded all the same, and an error ends it.
// For small batches, which are bound by their launches: one less (28.1 -> 27.0 us a batch of 1000
// look-ups, 47.7 -> 40.4 of 6000 mixed queries), with a grid that leaves half of each SM to the
// next batch. Larger batches keep k_rebuild_prep: the waiting CTAs would hold the SMs that the
// next batch's sort runs on (2^20 queries on 2^24 keys 359 -> 368 us a batch, 2^22 on 2^27 2% more).
__device__ bool prepare_write(const RebuildArgs& a, uint32_t epoch) {
    __shared__ int s_ready;
    const uint32_t units = prepare_units<kThreads>(a, epoch);
    if (threadIdx.x == 0) {
        uint32_t spins = 0;
        bool ok = true;
        while (ok && ld_relaxed32(&a.bm->tile_ctr[kCtrPrep]) < units) {
            ++spins;
            if (spins > kSpinLimit) {
                atomicOr(a.err, kErrTimeout);
                ok = false;
            }
            if ((spins & 1023u) == 0 && *(volatile uint32_t*)a.err) ok = false;
            if (spins > 32) __nanosleep(100);
        }
        __threadfence();  // the results are visible to the CTA past the barrier
        s_ready = ok ? 1 : 0;
    }
    __syncthreads();
    return s_ready != 0;
}

// Byte-wise arithmetic on a meta word holding four nodes (height in bits 0-5, delete
// flag in bit 7). live_heights clears the bytes of delete-flagged nodes; members(h, l)
// leaves bit 7 set in exactly the bytes whose height is >= l: 0x80 + h - l is >= 0x80
// iff h >= l, and never borrows from the next byte because h - l >= -33.
__device__ __forceinline__ uint32_t live_heights(uint32_t metaw) {
    const uint32_t t = (metaw >> 7) & 0x01010101u;  // 1 in the low bit of flagged bytes
    return metaw & ~(t * 0xFFu);
}
__device__ __forceinline__ uint32_t members(uint32_t hw, uint32_t l) {
    return ((hw | 0x80808080u) - l * 0x01010101u) & 0x80808080u;
}

constexpr uint32_t kMetaBytes = kNodes + 16;
constexpr uint32_t kWarpNodes = kNodes / 8;  // 512 nodes per warp

// One tile of 4096 nodes per CTA: the tile's meta arrives in shared memory by TMA bulk
// copy; keys are read from global memory only for the nodes that enter the index layer
// (about a quarter of them at p = 1/4, so key sectors holding none are never read).
// Warp w owns nodes [512 w, 512 w + 512); lane t holds nodes 16t..16t+15 of them.
//  1. per lane, a byte-wise membership test of its nodes for every level gives the
//     warp's count per level (lane i accumulates level Lb + i); the warps' counts are
//     prefixed across the tile (one barrier);
//  2. the lanes' level-Lb members (node indices) are placed in a per-warp list in
//     node order by one warp prefix sum;
//  3. the whole warp emits level Lb from the list, 32 consecutive entries per step
//     (coalesced stores), and compacts the list in place to the members of level
//     Lb + 1, keeping each one's index in level Lb for its down pointer; the next
//     levels repeat step 3 on the shrinking list.
// An incremental rebuild writes from the previous levels instead (relevel.cuh). One kernel
// for both, since the host cannot know which a batch needs and a launch that only exits costs
// it 3 us. Six CTAs per SM at 40 registers measured best over both kinds.
union WriteSmem {
    struct {
        uint8_t meta[kMetaBytes];
        uint32_t list[8 * kWarpNodes];
        uint32_t wcnt[8][32];
    } full;
    relevel::WriteSmem inc;
};

template <bool kFused>
__global__ void __launch_bounds__(kThreads, 6) k_rebuild_write(RebuildArgs a, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    __shared__ __align__(16) WriteSmem s_u;
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_base[kLevelSlots], s_n[kLevelSlots];
    __shared__ int s_ok;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DevMeta* m = a.m;
    if (!a.bm->rebuild) return;
    if (block_sees_error(&m->error)) return;
    if (!a.bm->inc && (m->H < m->Lb || m->size == 0)) return;
    if (kFused && !prepare_write(a, epoch)) return;
    if (a.bm->inc) {
        relevel::write(a, blockIdx.x, gridDim.x, s_u.inc);
        return;
    }
    uint8_t* s_meta = s_u.full.meta;
    uint32_t* s_list = s_u.full.list;
    auto& s_wcnt = s_u.full.wcnt;
    const uint32_t H = m->H, Lb = m->Lb, size = m->size, cur = m->cur;
    uint64_t* LK = m->lcur ? a.lkeys1 : a.lkeys;  // the index layer's buffer in use
    uint32_t* LD = m->lcur ? a.ldown1 : a.ldown;
    const uint32_t ntiles = (size + kNodes - 1) / kNodes;
    if (tid < kLevelSlots) {
        s_base[tid] = m->base[tid];
        s_n[tid] = m->n[tid];
    }
    if (tid == 0) mbar_init(&s_bar, 1);
    // A persistent loop over the tiles: the barrier's phase flips with every tile's copy.
    uint32_t phase = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1u) {
    const uint32_t ts = tile * kNodes;
    const uint32_t cnt = min((uint32_t)kNodes, size - ts);
    __syncthreads();  // the previous tile is done with shared memory
    if (tid == 0) {
        s_ok = 1;
        const uint32_t bm_ = ((cnt + 15u) / 16u) * 16u;
        mbar_arrive_expect_tx(&s_bar, bm_);
        bulk_g2s(s_meta, a.st.meta[cur] + ts, bm_, &s_bar);
    }
    const uint64_t* TK = a.st.keys[cur] + ts;  // this tile's keys
    __syncthreads();
    if (!mbar_wait_bounded(&s_bar, phase, a.err)) s_ok = 0;
    const uint32_t w0 = (uint32_t)warp * kWarpNodes;
    const uint32_t nb = w0 + (uint32_t)lane * 16u;
    uint32_t hw[4];
    {
        const uint4 v = *reinterpret_cast<const uint4*>(s_meta + nb);
        const uint32_t raw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t h = live_heights(raw[k]);
            const uint32_t first = nb + 4u * k;  // nodes past the storage layer's end are absent
            if (first + 4u > cnt) {
                const uint32_t keep = first >= cnt ? 0u : (cnt - first);
                h &= keep ? (0xFFFFFFFFu >> (8u * (4u - keep))) : 0u;
            }
            hw[k] = h;
        }
    }
    // 1. the warp's count per level
    uint32_t mine = 0;  // this lane's member count at level Lb
    {
        uint32_t c = 0;
        for (uint32_t l = Lb; l <= H; ++l) {
            uint32_t nl = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) nl += __popc(members(hw[k], l));
            if (l == Lb) mine = nl;
            const uint32_t tot = __reduce_add_sync(0xffffffffu, nl);
            if ((uint32_t)lane == l - Lb) c = tot;
            if (tot == 0) break;
        }
        s_wcnt[warp][lane] = c;
    }
    __syncthreads();
    if (!s_ok) {
        if (tid == 0) mbar_wait_bounded(&s_bar, phase, a.err);  // let the copy land
        return;
    }
    uint32_t wbase = 0;  // first position of this warp in level Lb + lane
    if (Lb + (uint32_t)lane <= H) {
        wbase = a.loff[(size_t)lane * ntiles + tile];
        for (int w = 0; w < warp; ++w) wbase += s_wcnt[w][lane];
    }
    // 2. level-Lb members in node order
    uint32_t* list = s_list + warp * kWarpNodes;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    uint32_t nlist = __shfl_sync(0xffffffffu, incl, 31);
    {
        uint32_t w = incl - mine;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t mk = members(hw[k], Lb);
            while (mk) {
                const uint32_t bit = __ffs(mk) - 1;
                list[w++] = nb + 4u * k + (bit >> 3);  // node within the tile
                mk &= mk - 1;
            }
        }
    }
    __syncwarp();
    // 3. emit level after level from the list, compacting it in place
    const uint32_t lt = lanemask_lt();
    uint32_t prev_base = 0;
    for (uint32_t l = Lb; l <= H && nlist > 0; ++l) {
        const uint32_t base = __shfl_sync(0xffffffffu, wbase, (int)(l - Lb));
        uint32_t nnext = 0;
        for (uint32_t j0 = 0; j0 < nlist; j0 += 32u) {
            const uint32_t j = j0 + (uint32_t)lane;
            const bool in = j < nlist;
            const uint32_t e = in ? list[j] : 0u;  // node | index in level l - 1 << 16
            const uint32_t node = e & 0xFFFFu;
            const uint32_t h = in ? (uint32_t)(s_meta[node] & kHeightMask) : 0u;
            const uint32_t up = __ballot_sync(0xffffffffu, in && h > l);
            __syncwarp();  // every lane has read its entry before the list is overwritten
            if (in) {
                const uint32_t p = base + j;
                if (p < s_n[l]) {
                    const uint32_t g = s_base[l] + p;
                    LK[g] = TK[node];
                    LD[g] = (l == Lb) ? ts + node : prev_base + (e >> 16);
                } else {
                    atomicOr(a.err, kErrBounds);
                }
                if (h > l) list[nnext + __popc(up & lt)] = node | (j << 16);
            }
            nnext += __popc(up);
            __syncwarp();
        }
        nlist = nnext;
        prev_base = base;
    }
    }  // tiles
}

// ---------------------------------------------------------------------------------
// Compaction of a tile of kNodes elements in rows of kThreads, for the bulk build and the export:
// row k holds elements [k kThreads, (k + 1) kThreads) of the tile, so loads are coalesced, and
// an element's place is its (row, warp)'s offset plus the kept lanes before it. (With 16
// consecutive elements per thread, neither loads nor stores were coalesced: 10^7 pairs took 445
// us to place and 236 to export.)
constexpr int kRowWarps = kPer * (kThreads / 32);  // 128 (row, warp) counts

struct Rows {
    uint32_t off[kRowWarps];
    uint32_t tile, prefix, total;
    int ok;
};

// Turns the counts in R.off into offsets, and finds the tile's first place by a look-back (tile
// numbers in the order CTAs take them). Returns false when the look-back gave up.
__device__ __forceinline__ bool place_rows(Rows& R, uint64_t* desc, uint32_t epoch, uint32_t* err) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x;
        uint32_t c[kRowWarps / 32], sum = 0;
#pragma unroll
        for (int k = 0; k < kRowWarps / 32; ++k) {
            c[k] = R.off[lane * (kRowWarps / 32) + k];
            sum += c[k];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= (uint32_t)o) x += y;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, x, 31);
        x -= sum;
#pragma unroll
        for (int k = 0; k < kRowWarps / 32; ++k) {
            R.off[lane * (kRowWarps / 32) + k] = x;
            x += c[k];
        }
        bool ok;
        const uint32_t ex = lookback_warp_wide<4>(desc, R.tile, epoch, tot, err, &ok);
        if (lane == 0) {
            R.prefix = ex;
            R.total = tot;
            R.ok = ok ? 1 : 0;
        }
    }
    __syncthreads();
    return R.ok != 0;
}

// Bulk build: keep the last query of every key run of the sorted input (the last
// occurrence of a key wins), with its value and tower height; count level sizes.
__global__ void __launch_bounds__(kThreads) k_create_storage(CreateArgs a, uint32_t epoch) {
    pdl_wait();
    pdl_trigger();
    __shared__ Rows R;
    __shared__ uint32_t s_ge[32];  // nodes of height >= 1 + i
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t n = a.n, ntiles = (n + kNodes - 1) / kNodes;
    if (tid < 32) s_ge[tid] = 0;
    uint32_t ge = 0, kept = 0;  // lane i: this warp's nodes of height >= 1 + i; thread 0: the CTA's nodes
    for (;;) {
        __syncthreads();
        if (tid == 0) R.tile = atomicAdd(&a.bm->tile_ctr[kCtrCreate], 1u);
        __syncthreads();
        const uint32_t tile = R.tile;
        if (tile >= ntiles) break;
        const uint32_t ts = tile * kNodes;
        uint64_t key[kPer];
        uint32_t at[kPer], keep = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = ts + (uint32_t)k * kThreads + (uint32_t)tid;
            key[k] = i < n ? a.sk[i] : kMaxKey;
            at[k] = i < n ? a.sp[i] & ((1u << 30) - 1u) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = ts + (uint32_t)k * kThreads + (uint32_t)tid;
            uint64_t next = __shfl_down_sync(0xffffffffu, key[k], 1);
            if (lane == 31) next = i + 1u < n ? a.sk[i + 1u] : kMaxKey;
            const bool kp = i < n && key[k] != kMaxKey && (i + 1u == n || next != key[k]);
            const uint32_t b = __ballot_sync(0xffffffffu, kp);
            keep |= (kp ? 1u : 0u) << k;
            if (lane == 0) R.off[k * (kThreads / 32) + warp] = (uint32_t)__popc(b);
        }
        if (!place_rows(R, a.desc, epoch, a.err)) break;
        if (tid == 0) kept += R.total;
#pragma unroll 4
        for (int k = 0; k < kPer; ++k) {
            const bool kp = (keep >> k) & 1u;
            const uint32_t b = __ballot_sync(0xffffffffu, kp);
            const uint32_t o = R.prefix + R.off[k * (kThreads / 32) + warp] + (uint32_t)__popc(b & lt);
            const uint32_t h = kp ? tower_height(key[k], a.hp) : 0u;
            for (uint32_t l = 1;; ++l) {
                const uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, h >= l));
                if (c == 0) break;
                if ((uint32_t)lane == l - 1u) ge += c;
            }
            if (!kp) continue;
            if (o >= a.st_cap) {
                atomicOr(a.err, kErrBounds);
                continue;
            }
            a.st.keys[0][o] = key[k];
            a.st.vals[0][o] = a.uvals[at[k]];
            a.st.meta[0][o] = (uint8_t)h;
        }
    }
    if (ge) atomicAdd(&s_ge[lane], ge);
    __syncthreads();
    if (tid == 0 && kept) atomicAdd(&a.m->size, kept);
    if (tid < 32 && s_ge[tid]) atomicAdd(&a.m->cnt[tid + 1], s_ge[tid]);
}

// Live pairs of the storage layer, in key order.
__global__ void __launch_bounds__(kThreads) k_export_live(Storage st, const DevMeta* m, uint64_t* ko,
                                                          uint64_t* vo, uint64_t cap, uint32_t* count,
                                                          uint64_t* desc, uint32_t* tile_ctr, uint32_t epoch,
                                                          uint32_t* err) {
    pdl_wait();
    pdl_trigger();
    __shared__ Rows R;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t size = m->size, cur = m->cur;
    const uint32_t ntiles = (size + kNodes - 1) / kNodes;
    for (;;) {
        __syncthreads();
        if (tid == 0) R.tile = atomicAdd(tile_ctr, 1u);
        __syncthreads();
        const uint32_t tile = R.tile;
        if (tile >= ntiles) break;
        const uint32_t ts = tile * kNodes;
        uint32_t live = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = ts + (uint32_t)k * kThreads + (uint32_t)tid;
            live |= (i < size && !(st.meta[cur][i] & kTomb) ? 1u : 0u) << k;
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t b = __ballot_sync(0xffffffffu, (live >> k) & 1u);
            if (lane == 0) R.off[k * (kThreads / 32) + warp] = (uint32_t)__popc(b);
        }
        if (!place_rows(R, desc, epoch, err)) break;
        if (tid == 0 && tile == ntiles - 1) *count = R.prefix + R.total;
#pragma unroll 8
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = ts + (uint32_t)k * kThreads + (uint32_t)tid;
            const bool lv = (live >> k) & 1u;
            const uint32_t b = __ballot_sync(0xffffffffu, lv);
            const uint64_t o = (uint64_t)R.prefix + R.off[k * (kThreads / 32) + warp] + (uint32_t)__popc(b & lt);
            if (lv && o < cap) {
                ko[o] = st.keys[cur][i];
                vo[o] = st.vals[cur][i];
            }
        }
    }
}

// Failure-path self-test: tile 1 waits for tile 0, which never publishes, so the
// bounded look-back must give up, record kErrTimeout and return.
__global__ void k_wait_selftest(uint64_t* desc, uint32_t* err) {
    bool ok = true;
    lookback_warp(desc, 1u, 1u, 0u, err, &ok);
}

}  // namespace

cudaError_t launch_merge(const RebuildArgs& a, uint32_t& epoch, cudaStream_t s, int num_sms) {
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(k_merge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MergeSmem));
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const uint32_t chunks = a.size_ub / kChunk + 1;
    const uint32_t cap = (uint32_t)num_sms * 4u;  // the CTAs resident at once
    launch_dep(k_merge, chunks < cap ? chunks : cap, kThreads, sizeof(MergeSmem), s, a, ++epoch);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_level_layout(const RebuildArgs& a, cudaStream_t s) {
    launch_dep(k_level_layout, 1, 32, 0, s, a);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_rebuild_count(const RebuildArgs& a, cudaStream_t s, int num_sms) {
    const uint32_t tiles = (a.size_ub + kNodes - 1) / kNodes + 1;
    const uint32_t cb = (tiles + 7) / 8, ccap = (uint32_t)num_sms * 4u;
    launch_dep(k_rebuild_count, cb < ccap ? cb : ccap, 256, 0, s, a);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_rebuild_write(const RebuildArgs& a, bool fused, uint32_t& epoch, cudaStream_t s, int num_sms) {
    // per tile of the storage layer, or of the levels and their changes (fewer but for change
    // lists, which a batch's queries bound); at most the CTAs resident at once
    const uint32_t nodes = (a.size_ub + kNodes - 1) / kNodes + 1;
    const uint32_t tiles = nodes + a.lst_cap / (2u * 256u) + kLevelSlots, cap = (uint32_t)num_sms * (fused ? 3u : 6u);
    const uint32_t grid = tiles < cap ? tiles : cap;
    ++epoch;
    if (fused) {
        launch_dep(k_rebuild_write<true>, grid, kThreads, 0, s, a, epoch);
    } else {
        const uint32_t units = (nodes + 4095) / 4096 * (kLevelSlots - 2), most = (uint32_t)num_sms;
        launch_dep(k_rebuild_prep, units < most ? units : most, 1024, 0, s, a, epoch);
        ++g_launches;
        launch_dep(k_rebuild_write<false>, grid, kThreads, 0, s, a, epoch);
    }
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_create_storage(const CreateArgs& a, uint32_t& epoch, cudaStream_t s, int num_sms) {
    if (a.n == 0) return cudaSuccess;
    const uint32_t tiles = (a.n + kNodes - 1) / kNodes;
    const uint32_t cap = (uint32_t)num_sms * 4u;
    launch_dep(k_create_storage, (int)(tiles < cap ? tiles : cap), kThreads, 0, s, a, ++epoch);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_export_live(const Storage& st, const DevMeta* m, uint64_t* keys_out, uint64_t* vals_out,
                               uint64_t cap, uint32_t* count, uint64_t* desc, uint32_t* tile_ctr,
                               uint32_t& epoch, uint32_t* err, cudaStream_t s, int num_sms, uint32_t size_ub) {
    const uint32_t tiles = size_ub / kNodes + 1;
    const uint32_t c = (uint32_t)num_sms * 4u;
    launch_dep(k_export_live, (int)(tiles < c ? tiles : c), kThreads, 0, s, st, m, keys_out, vals_out, cap, count, desc,
                                                                   tile_ctr, ++epoch, err);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(uint64_t* desc, uint32_t* err, cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(desc, err);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace pi
