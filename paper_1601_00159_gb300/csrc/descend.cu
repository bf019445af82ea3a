// Descend the index layer to each query's interception (Algorithm 2,
// Definition 4), then locate the query's key in the storage layer (Algorithm 4's
// getNode), for every distinct key of the sorted batch.
//
// Layout (built by the rebuild): all index levels live in one key array and one down
// array, top level first; level l is [base[l], base[l] + n[l]) followed by a sentinel
// entry with key 2^64-1. down[i] is the position of the same key in the level below
// (for the lowest built level: its storage-layer position), so the keys of level l-1
// that lie between two consecutive keys of level l are exactly
// [down[r], down[r + 1]).
//
// The descent works on the whole batch -- the paper's group query processing (Section 4.4.3)
// with the group being every distinct key of the batch. One kernel takes a tile of the sorted
// batch per CTA: it collects the tile's local run heads (a query whose key differs from the
// previous one, or the first query of a 128-query block), finds each head's place on the lowest
// built level (which holds every key of the levels above it) and, in the gap below, the storage
// node with the largest key <= q and its state, which it leaves in the tile's part of the state
// arrays, head after head. No tile waits for another. For k_apply it also leaves each block's first
// head's number and largest ownership marker, and, per group of blocks, the largest marker of those
// whose last key fills the next block too: a look-back that has come past blocks without a marker
// ends at such a block. (The largest of every block cost 2^18 queries 4 us of contended atomics.)
// Large batches take windows: the keys of a tile are neighbours, so their places lie in one
// stretch of the level, which the CTA reads into shared memory once, with coalesced loads, and
// searches there; the level is then read about once per batch instead of a few random sectors
// per key and level. Batches sparse on their index search from the top, seven entries a round.

#include "search.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// Keys <= q in the sorted K[0, n), by a whole warp: 32 probes a round.
__device__ __forceinline__ uint32_t warp_count_le(const uint64_t* K, uint32_t n, uint64_t q) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t lo = 0, hi = n;  // the count lies in [lo, hi]
    while (lo < hi) {
        const uint32_t step = (hi - lo + 31u) / 32u, p = lo + lane * step;
        const uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, p < hi && K[p] <= q));  // a prefix
        if (c == 0) break;
        if (c < 32u) hi = min(hi, lo + c * step);
        lo += (c - 1u) * step + 1u;
    }
    return lo;
}

// The array that gives a key its storage gap: the lowest built level, or the storage layer
// itself when no level is built (down is then null).
struct GapLevel {
    const uint64_t* keys;
    const uint32_t* down;
    uint32_t n;
};
__device__ __forceinline__ GapLevel gap_level(const DescendArgs& a) {
    const DevMeta* m = a.m;
    const uint32_t Lb = m->Lb;
    GapLevel g;
    if (Lb <= m->H) {
        g.keys = (m->lcur ? a.lkeys1 : a.lkeys) + m->base[Lb];
        g.down = (m->lcur ? a.ldown1 : a.ldown) + m->base[Lb];
        g.n = m->n[Lb];
    } else {
        g.keys = a.st.keys[m->cur];
        g.down = nullptr;
        g.n = m->size;
    }
    return g;
}

// Writes the state of key q at position `at`: r is the storage node with the largest key <= q,
// kr its key. Without a delete-flagged node in the storage layer no state byte is read.
__device__ __forceinline__ void store_state(const DescendArgs& a, uint32_t at, uint64_t q, int32_t r, uint64_t kr,
                                            const uint8_t* SM, const uint64_t* SV, bool flagged) {
    const bool exists = r >= 0 && kr == q;
    // the value is read with the meta byte, not after it, so both requests are in
    // flight together (a delete-flagged node's value is read and dropped)
    const uint8_t meta = exists && flagged ? SM[r] : (uint8_t)0;
    const uint64_t v = exists ? SV[r] : 0ull;
    const bool live = exists && !(meta & kTomb);
    a.loc[at] = (uint32_t)(r + 1);
    a.flags[at] = (uint8_t)((exists ? 1u : 0u) | (live ? 2u : 0u));
    a.val0[at] = live ? v : 0ull;
}

// What the end of the batch compares with, before anything changes it.
__device__ __forceinline__ void note_sizes(const DescendArgs& a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.bm->size0 = a.m->size;
        a.bm->tombs0 = a.m->tombs;
    }
}

// kWindow entries of the gap level fit a CTA's shared memory beside its heads, four CTAs to an
// SM. Two more warps find the places of the tile's first and last key while the others collect
// the heads. Bound by HBM's random 64-byte accesses (a line of storage keys or two, a value and a
// state byte per key), about half of the kernel's time; collecting the heads and searching the
// window take the rest. Measured, 2^22 skewed queries on 2^27 keys (1.5 M distinct): collecting
// the heads, walking the levels and locating took three kernels and 186 us, this one 157. 2^18
// appended keys on 4 M: 46 us in three kernels, 18 without windows.
constexpr uint32_t kWindow = 2560;

template <bool kWin>
struct LocateSmem {
    static constexpr uint32_t kT = kWin ? kApplyTile : kThreads;  // sorted queries per CTA
    uint64_t hk[kT];  // each warp's heads
    uint64_t wk[kWin ? kWindow : 1];
    uint32_t wd[kWin ? kWindow : 1];
    uint32_t x[kWin ? kT : 1];  // their places in the tile's stretch of the level
};

template <bool kWin>
__global__ void __launch_bounds__(kWin ? kThreads + 64 : kThreads, kWin ? 4 : 6) k_locate(DescendArgs a) {
    pdl_wait();
    pdl_trigger();
    constexpr uint32_t kT = LocateSmem<kWin>::kT;
    constexpr int kR = (int)(kT / kThreads);  // rows of 32 per warp
    extern __shared__ __align__(16) uint8_t s_dyn[];
    LocateSmem<kWin>& S = *reinterpret_cast<LocateSmem<kWin>*>(s_dyn);
    __shared__ uint32_t s_cnt[kWarps], s_half[kWarps], s_max[kWarps], s_c[2];
    __shared__ bool s_more[kWarps];
    const DevMeta* m = a.m;
    if (block_sees_error(&m->error)) return;
    note_sizes(a);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = a.n, qv = n - a.bm->invalid, tb = blockIdx.x * kT;
    const uint32_t lt = lanemask_lt();
    GapLevel g{};
    if (kWin) g = gap_level(a);
    if (warp < kWarps) {
        const uint32_t w0 = tb + (uint32_t)warp * 32u * kR;
        uint64_t kk[kR];
        uint32_t op[kR];
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            const uint32_t i = w0 + (uint32_t)k * 32u + (uint32_t)lane;
            kk[k] = i < qv ? a.sk[i] : kMaxKey;
            op[k] = i < qv ? (a.sp[i] >> 30) : 0u;
        }
        uint64_t carry = (w0 > 0 && w0 - 1 < qv) ? a.sk[w0 - 1] : kMaxKey;  // key before the element
        const uint32_t beyond = w0 + 32u * kR - 1u + kApplyBlock;  // a block past the warp's last query
        const uint64_t kb = beyond < qv ? a.sk[beyond] : 0ull;
        uint32_t nq = 0, half = 0, most = 0;
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            const uint32_t i = w0 + (uint32_t)k * 32u + (uint32_t)lane;
            const bool valid = i < qv;
            const uint64_t q = kk[k];
            uint64_t prev = __shfl_up_sync(0xffffffffu, q, 1);
            if (lane == 0) prev = carry;
            carry = __shfl_sync(0xffffffffu, q, 31);
            const bool head = valid && (i == 0 || q != prev);
            const bool local = valid && (head || i % kApplyBlock == 0);
            const uint32_t e = (valid && (op[k] == 1u || op[k] == 2u)) ? 2u * i + 3u : (head ? 2u * i + 2u : 0u);
            most = max(most, e);
            const uint32_t b = __ballot_sync(0xffffffffu, local);
            if (local) S.hk[(uint32_t)warp * 32u * kR + nq + (uint32_t)__popc(b & lt)] = q;
            nq += (uint32_t)__popc(b);
            if (kWin && k == kR / 2 - 1) half = nq;
            if (kWin && (k + 1) % (int)(kApplyBlock / 32u) == 0) {  // a block ends
                const uint32_t mk = __reduce_max_sync(0xffffffffu, most);
                const uint32_t bs = i / kApplyBlock * kApplyBlock;
                const uint64_t kn = k + 1 < kR ? __shfl_sync(0xffffffffu, kk[kR - 1], 31) : kb;
                if (lane == 0 && bs < n) {
                    const bool any = mk >= 2u * bs + 2u;
                    a.blk_mark[bs / kApplyBlock] = any ? mk : 0u;
                    if (any && bs + 2u * kApplyBlock - 1u < qv && kn == carry) atomicMax(&a.grp_mark[bs / kMarkGroup], mk);
                }
            }
        }
        const uint32_t mk = __reduce_max_sync(0xffffffffu, most);
        const bool more = beyond < qv && kb == carry;
        if (lane == 0) {
            s_cnt[warp] = nq;
            s_half[warp] = half;
            s_max[warp] = mk;
            s_more[warp] = more;
        }
    } else if (tb < qv) {  // the places of the tile's first and last key
        const uint32_t last = min(tb + kT, qv) - 1u;
        const uint32_t c = warp_count_le(g.keys, g.n, a.sk[warp == kWarps ? tb : last]);
        if (lane == 0) s_c[warp - kWarps] = c;
    }
    __syncthreads();
    if (kWin) {
        if (tid < kWarps) {  // a warp's two blocks
            uint32_t h = 0;
            for (int w = 0; w < tid; ++w) h += s_cnt[w];
            reinterpret_cast<uint2*>(a.blk_head)[tb / kT * kWarps + (uint32_t)tid] = make_uint2(h, h + s_half[tid]);
        }
    } else if (tid < (int)(kT / kApplyBlock)) {
        uint32_t mk = 0;
#pragma unroll
        for (int w = 0; w < (int)(kApplyBlock / 32u); ++w) mk = max(mk, s_max[tid * (int)(kApplyBlock / 32u) + w]);
        uint32_t h = 0;
        for (int w = 0; w < tid * (int)(kApplyBlock / 32u); ++w) h += s_cnt[w];
        if (tb + (uint32_t)tid * kApplyBlock < n) {
            a.blk_mark[tb / kApplyBlock + (uint32_t)tid] = mk;
            a.blk_head[tb / kApplyBlock + (uint32_t)tid] = h;
            if (mk && s_more[(tid + 1) * (int)(kApplyBlock / 32u) - 1]) atomicMax(&a.grp_mark[tb / kMarkGroup], mk);
        }
    }
    if (tb >= qv) return;
    uint32_t c0 = 0, span = 0, first = 0;
    bool staged = false;
    if (kWin) {
        c0 = s_c[0];
        const uint32_t c1 = s_c[1];
        first = c0 ? c0 - 1u : 0u;
        const uint32_t len = c1 - first + 1u;  // entry c1 <= n: at most the sentinel
        span = c1 - c0;
        staged = len <= kWindow;
        if (staged) {
            for (uint32_t x = (uint32_t)tid; x < len; x += blockDim.x) {
                S.wk[x] = g.keys[first + x];
                S.wd[x] = g.down ? g.down[first + x] : 0u;
            }
        }
        __syncthreads();
    }
    const uint32_t size = m->size, cur = m->cur;
    const bool flagged = m->tombs != 0;
    const uint64_t* SK = a.st.keys[cur];
    const uint8_t* SM = a.st.meta[cur];
    const uint64_t* SV = a.st.vals[cur];
    uint32_t off[kWarps], tot = 0;  // heads before each warp's
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        off[w] = tot;
        tot += s_cnt[w];
    }
    auto head_slot = [&](uint32_t h) {  // where head h of the tile lies in S.hk
        uint32_t at = h;
#pragma unroll
        for (int w = 1; w < kWarps; ++w)
            if (h >= off[w]) at = (uint32_t)w * 32u * kR + (h - off[w]);
        return at;
    };
    if (!kWin) {
        for (uint32_t h = (uint32_t)tid; h < tot; h += blockDim.x) {
            const uint64_t q = S.hk[head_slot(h)];
            uint64_t kr = 0;
            const int32_t r = storage_search(m, SK, a.lkeys, a.ldown, a.lkeys1, a.ldown1, q, kr, a.err);
            store_state(a, tb + h, q, r, kr, SM, SV, flagged);
        }
        return;
    }
    // Each head's gap: entries of the level <= q, searched in the window or between its ends
    const uint32_t step0 = span ? 1u << (31 - __clz(span)) : 0u;
    const uint32_t o = c0 - first;
    struct Gap {
        uint32_t c, lo, dn;
        uint64_t klo, kn;
    };
    auto gap_of = [&](uint32_t x) {  // x = c - c0
        Gap p;
        p.c = c0 + x;
        if (staged) {
            p.kn = S.wk[o + x];
            p.dn = S.wd[o + x];
            p.klo = p.c ? S.wk[o + x - 1u] : 0ull;
            p.lo = p.c ? S.wd[o + x - 1u] : 0u;
        } else {
            p.kn = g.keys[p.c];
            p.klo = p.c ? g.keys[p.c - 1u] : 0ull;
            p.dn = g.down ? g.down[p.c] : 0u;
            p.lo = p.c && g.down ? g.down[p.c - 1u] : 0u;
        }
        return p;
    };
    // First the places of all of the thread's heads, with the storage line of each asked for
    // from L2, so that the reads of a head below find it there.
    for (uint32_t h = (uint32_t)tid; h < tot; h += blockDim.x) {
        const uint32_t at = head_slot(h);
        const uint64_t q = S.hk[at];
        uint32_t x = 0;
        if (staged) {
            for (uint32_t step = step0; step > 0; step >>= 1)
                if (x + step <= span && S.wk[o + x + step - 1u] <= q) x += step;
        } else {
            x = count_le(g.keys + c0, span, q);
        }
        S.x[at] = x;
        if (g.down) {
            const Gap p = gap_of(x);
            const uint64_t* line = SK + gap_line(p.lo, p.dn, p.klo, p.kn, q);
            prefetch_l2(line);
        }
    }
    // Then the nodes; a node's value and state byte are asked for one head before they are read.
    uint32_t ph = 0xffffffffu;
    int32_t pr = -1;
    uint64_t pq = 0, pk = 0;
    for (uint32_t h = (uint32_t)tid; h < tot; h += blockDim.x) {
        const uint32_t at = head_slot(h);
        const uint64_t q = S.hk[at];
        const Gap p = gap_of(S.x[at]);
        int32_t r = (int32_t)p.c - 1;
        uint64_t kr = p.klo;
        if (g.down) r = gap_search(SK, p.lo, p.dn, p.klo, p.kn, q, size, kr, a.err);
        if (r >= 0 && kr == q) {
            prefetch_l2(SV + r);
            if (flagged) prefetch_l2(SM + r);
        }
        if (ph != 0xffffffffu) store_state(a, tb + ph, pq, pr, pk, SM, SV, flagged);
        ph = h;
        pr = r;
        pq = q;
        pk = kr;
    }
    if (ph != 0xffffffffu) store_state(a, tb + ph, pq, pr, pk, SM, SV, flagged);
}

// Small batches: the place of every query among the sorted tiles, and its storage node, for 32
// queries per CTA (consecutive ones of a sorted tile, one per lane). An element's place is its
// place in its tile, plus the keys of every earlier tile that are <= its own and of every later
// tile that are smaller: one warp per other tile counts those, while the last warp searches the
// lowest built level (it holds every key of the levels above) and the storage gap. The kernel
// is bound by dependent reads of L2, so the chains run side by side in warps of their own and
// every search reads seven entries a round; the lanes' keys are neighbours, so their probes
// share sectors. Every query is looked up, equal keys as often as they come: below kSmallSort
// queries the passes that would collect the distinct keys cost more than the look-ups they save.
constexpr uint32_t kRankWarps = 8;
constexpr int kRankThreads = 32 * (kRankWarps + 1);

__global__ void __launch_bounds__(kRankThreads) k_rank_locate(DescendArgs a, const uint64_t* __restrict__ tk,
                                                              const uint32_t* __restrict__ tp,
                                                              uint64_t* __restrict__ ok, uint32_t* __restrict__ op) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_pos[kRankWarps][32];
    const DevMeta* m = a.m;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t n = a.n, i = blockIdx.x * 32u + lane;
    const uint64_t q = i < n ? tk[i] : kMaxKey;
    note_sizes(a);
    int32_t r = -1;
    uint64_t v = 0;
    bool exists = false, live = false;
    if (warp < kRankWarps) {
        const uint32_t own = i / kRunTile, tiles = (n + kRunTile - 1) / kRunTile;
        uint32_t c = 0;
        for (uint32_t t = warp; t < tiles; t += kRankWarps) {
            if (t == own) {
                c += i - own * kRunTile;
                continue;
            }
            // keys <= q are keys < q + 1; invalid queries (2^64-1) stay behind every key
            const uint64_t* T = tk + t * kRunTile;
            const uint32_t len = min(kRunTile, n - t * kRunTile);
            if (t < own) c += count_le(T, len, q);
            else c += q ? count_le(T, len, q - 1u) : 0u;
        }
        s_pos[warp][lane] = c;
    } else if (q != kMaxKey && *(volatile const uint32_t*)&m->error == 0) {
        const uint32_t cur = m->cur;
        uint64_t kr = 0;
        r = storage_search(m, a.st.keys[cur], a.lkeys, a.ldown, a.lkeys1, a.ldown1, q, kr, a.err);
        exists = r >= 0 && kr == q;
        const uint8_t meta = exists && m->tombs ? a.st.meta[cur][r] : (uint8_t)0;
        v = exists ? a.st.vals[cur][r] : 0ull;
        live = exists && !(meta & kTomb);
    }
    __syncthreads();
    if (i >= n || (warp != 0 && warp != kRankWarps)) return;
    uint32_t pos = 0;
#pragma unroll
    for (uint32_t w = 0; w < kRankWarps; ++w) pos += s_pos[w][lane];
    if (pos >= n) {
        atomicOr(a.err, kErrBounds);
    } else if (warp == 0) {
        ok[pos] = q;
        op[pos] = tp[i];
    } else {
        a.loc[pos] = (uint32_t)(r + 1);
        a.flags[pos] = (uint8_t)((exists ? 1u : 0u) | (live ? 2u : 0u));
        a.val0[pos] = live ? v : 0ull;
    }
}

}  // namespace

cudaError_t launch_rank_locate(const DescendArgs& a, const uint64_t* tk, const uint32_t* tp, uint64_t* ok, uint32_t* op,
                               cudaStream_t s) {
    if (a.n == 0 || a.n > kSmallSort) return cudaErrorInvalidValue;
    launch_dep(k_rank_locate, (a.n + 31u) / 32u, kRankThreads, 0, s, a, tk, tp, ok, op);
    ++g_launches;
    return cudaGetLastError();
}

bool descend_windows(uint64_t n, uint64_t entries) {
    return n >= kWindowBatch && entries / (n / kApplyTile) <= kWindow * 3u / 4u;
}

cudaError_t launch_descend(const DescendArgs& a, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    if (a.windows) {
        static bool attr_set = false;
        constexpr int smem = (int)sizeof(LocateSmem<true>);
        if (!attr_set) {
            cudaError_t e = cudaFuncSetAttribute(k_locate<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
        launch_dep(k_locate<true>, (a.n + kApplyTile - 1) / kApplyTile, kThreads + 64, smem, s, a);
    } else {
        launch_dep(k_locate<false>, (a.n + kThreads - 1) / kThreads, kThreads, sizeof(LocateSmem<false>), s, a);
    }
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace pi
