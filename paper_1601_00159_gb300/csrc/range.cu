// Range search (Section 3.2.5): for every query [lo, hi], the live pairs with
// lo <= key <= hi in key order, packed query after query (offsets in CSR form).
//
// The paper sorts range queries by their lower bound, finds the interceptions like
// point queries, splits a range that crosses into the next thread's part and walks the
// storage layer up to the upper bound. Here a query's range is the slice [start, end) of the
// storage layer between the places of its bounds:
//   k_range_find   the slices, the live nodes of each, and their running sum over the CTAs (by
//                  the CTA that finishes last);
//   k_range_write  offsets[i] and, when the query's pairs fit in the caller's capacity,
//                  its keys and values.
// A lane per bound searches the index; sorting the bounds first, as a batch's keys are, took
// twelve launches and gained nothing back: with 2^16 ranges on 2^24 keys 173 us of kernels
// against 70, with 2^20 ranges 465 us a call against 272.
// A warp takes up to 32 consecutive queries as one run of nodes, so that its lanes are busy
// whatever the slices' lengths, its loads are consecutive nodes and its stores consecutive
// pairs; fewer queries per warp when the queries would not fill the chip. (A warp per query, each
// lane copying 16 consecutive nodes, took 182 us for 2^16 ranges of 100 keys, a call 399 us; the
// call now takes 110.) The CSR offsets fix every query's output place, so no query waits for
// another.

#include "search.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;

// Block-wide exclusive sum of 64-bit values (kThreads threads); total in *total.
__device__ __forceinline__ uint64_t block_excl_sum64(uint64_t v, uint64_t* tmp, uint64_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const uint64_t w = lane < kThreads / 32 ? tmp[lane] : 0ull;
        uint64_t s = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kThreads / 32) tmp[lane] = s - w;
        if (lane == kThreads / 32 - 1) tmp[32] = s;
    }
    __syncthreads();
    const uint64_t r = tmp[warp] + x - v;
    if (total) *total = tmp[32];
    __syncthreads();
    return r;
}

// Live nodes of the 16-byte meta chunk c, read as w, that lie in [s, e).
__device__ __forceinline__ uint32_t live_count(const uint4& w, uint64_t c, uint32_t s, uint32_t e) {
    const uint32_t words[4] = {w.x, w.y, w.z, w.w};
    const uint64_t b0 = c * 16u;
    const uint32_t lo = s > b0 ? (uint32_t)(s - b0) : 0u, hi = e < b0 + 16u ? (uint32_t)(e - b0) : 16u;
    uint32_t n = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
        uint32_t live = ~words[k] & 0x80808080u;  // the delete flag is bit 7
        const uint32_t from = lo > 4u * k ? lo - 4u * k : 0u, to = hi > 4u * k ? hi - 4u * k : 0u;
        live = from >= 4u ? 0u : (live >> (8u * from)) << (8u * from);
        live = to >= 4u ? live : live & ((1u << (8u * to)) - 1u);
        n += (uint32_t)__popc(live);
    }
    return n;
}

// Live nodes in [s, e), a long slice, by the whole warp: every lane keeps four loads in flight.
// (Chunk by chunk, the way of short slices, a warp waits for each load: one slice of 2^23 nodes took
// 6570 us, now 1910.) A call of its own, so that the kernel keeps six CTAs per SM.
constexpr uint32_t kLongSlice = 256;  // chunks
__device__ __noinline__ uint32_t long_live_count(const uint8_t* meta, uint32_t s, uint32_t e) {
    constexpr int kU = 4;
    const uint4* M = reinterpret_cast<const uint4*>(meta);
    const uint32_t c1 = (e - 1u) / 16u + 1u;
    uint32_t n = 0;
    for (uint32_t c0 = s / 16u + (threadIdx.x & 31u); c0 < c1; c0 += 32u * kU) {
        uint4 w[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {  // (bytes of ones count as flagged)
            const uint32_t c = c0 + 32u * (uint32_t)u;
            w[u] = c < c1 ? M[c] : make_uint4(~0u, ~0u, ~0u, ~0u);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) n += live_count(w[u], c0 + 32u * (uint32_t)u, s, e);
    }
    return __reduce_add_sync(0xffffffffu, n);
}

// Exclusive sum over the warp's lanes.
__device__ __forceinline__ uint64_t warp_excl_sum64(uint64_t v, uint64_t* total) {
    const uint32_t lane = threadIdx.x & 31u;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}

// The lane whose part of a run holds element x: the last one whose exclusive prefix is <= x
// (an empty part shares its prefix with the next, so it is never the last).
__device__ __forceinline__ uint32_t part_of(uint32_t pre, uint32_t x) {
    uint32_t j = 0;
#pragma unroll
    for (uint32_t st = 16; st > 0; st >>= 1) {
        const uint32_t p = __shfl_sync(0xffffffffu, pre, (int)(j + st));
        if (p <= x) j += st;
    }
    return j;
}

// Storage nodes below (lo) or up to (hi) a bound.
__device__ __forceinline__ uint32_t bound_place(const RangeArgs& a, uint64_t q, bool is_lo) {
    if (q == kMaxKey) return a.m->size;  // the bound 2^64-1 lies past every stored key
    uint64_t key = 0;
    const int32_t r =
        storage_search(a.m, a.st.keys[a.m->cur], a.lkeys, a.ldown, a.lkeys1, a.ldown1, q, key, a.err);
    return is_lo && r >= 0 && key == q ? (uint32_t)r : (uint32_t)(r + 1);
}

// Slices and live nodes of every query; per-CTA totals and, by the last CTA, their exclusive
// prefix and the grand total. qw: queries per warp.
__global__ void __launch_bounds__(kThreads, 6) k_range_find(RangeArgs a, uint32_t qw) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint64_t s_tmp[33], s_sum[kThreads / 32];
    __shared__ uint32_t s_cnt[kThreads];
    __shared__ uint32_t s_last;
    const DevMeta* m = a.m;
    if (block_sees_error(&m->error)) return;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint8_t* SM = a.st.meta[m->cur];
    const bool flagged = m->tombs != 0;
    const uint32_t q0 = (blockIdx.x * (kThreads / 32) + warp) * qw, i = q0 + lane;
    const bool mine = lane < qw && i < a.n;
    uint32_t s = 0, e = 0;
    // a lane per bound: 16 queries per round
    for (uint32_t r0 = 0; r0 < qw; r0 += 16u) {
        const uint32_t x = r0 + (lane >> 1), j = q0 + x;
        uint32_t place = 0;
        if (x < qw && j < a.n) place = bound_place(a, lane & 1u ? a.hi[j] : a.lo[j], !(lane & 1u));
        const uint32_t from = (lane - r0) & 15u;  // this lane's query's pair of lanes
        const uint32_t ps = __shfl_sync(0xffffffffu, place, (int)(2u * from));
        const uint32_t pe = __shfl_sync(0xffffffffu, place, (int)(2u * from + 1u));
        if (lane >= r0 && lane < r0 + 16u) {
            s = ps;
            e = pe;
        }
    }
    if (mine) {
        a.start[i] = s;
        a.end[i] = e;
    }
    const uint32_t len = mine && e > s ? e - s : 0u;
    uint32_t cnt = len;
    if (flagged) {
        s_cnt[threadIdx.x] = 0;
        __syncwarp();
        uint32_t chunks = len ? (e - 1u) / 16u - s / 16u + 1u : 0u;
        uint32_t nlong = 0;
        for (uint32_t rest = __ballot_sync(0xffffffffu, chunks >= kLongSlice); rest; rest &= rest - 1u) {
            const int j = __ffs((int)rest) - 1;
            const uint32_t c = long_live_count(SM, __shfl_sync(0xffffffffu, s, j), __shfl_sync(0xffffffffu, e, j));
            if ((int)lane == j) nlong = c;
        }
        if (chunks >= kLongSlice) chunks = 0;
        uint64_t total;
        const uint32_t pre = (uint32_t)warp_excl_sum64(chunks, &total);
        for (uint32_t x0 = 0; x0 < (uint32_t)total; x0 += 32u) {
            const uint32_t x = x0 + lane, j = part_of(pre, x);
            const uint32_t js = __shfl_sync(0xffffffffu, s, (int)j), je = __shfl_sync(0xffffffffu, e, (int)j);
            const uint32_t jp = __shfl_sync(0xffffffffu, pre, (int)j);
            if (x < (uint32_t)total) {
                const uint32_t at = js / 16u + (x - jp);
                const uint32_t c = live_count(reinterpret_cast<const uint4*>(SM)[at], at, js, je);
                if (c) atomicAdd(&s_cnt[warp * 32u + j], c);
            }
        }
        __syncwarp();
        cnt = s_cnt[threadIdx.x] + nlong;
    }
    if (mine) a.cnt[i] = cnt;
    uint64_t wsum;
    warp_excl_sum64(mine ? cnt : 0u, &wsum);
    if (lane == 0) s_sum[warp] = wsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t t = 0;
        for (int w = 0; w < kThreads / 32; ++w) t += s_sum[w];
        a.bsum[blockIdx.x] = t;
        __threadfence();
        s_last = atomicAdd(a.done, 1u) == gridDim.x - 1u ? 1u : 0u;
        if (s_last) __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    // every CTA has arrived: exclusive prefix of their sums in place
    uint64_t carry = 0;
    for (uint32_t b0 = 0; b0 < gridDim.x; b0 += kThreads) {
        const uint32_t b = b0 + threadIdx.x;
        const uint64_t v = b < gridDim.x ? __ldcg(&a.bsum[b]) : 0ull;
        uint64_t tot;
        const uint64_t ex = block_excl_sum64(v, s_tmp, &tot);
        if (b < gridDim.x) a.bsum[b] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        a.offsets[a.n] = carry;
        *a.done = 0;  // for the next call
    }
}

// Copies the live nodes of a warp's slices (lane j: `len` nodes from s, at `pre` in the run of
// `total` nodes) to consecutive places from o on; returns the place after the last.
__device__ __forceinline__ uint64_t copy_run(const RangeArgs& a, const uint64_t* SK, const uint64_t* SV,
                                             const uint8_t* SM, uint32_t s, uint32_t pre, uint32_t total, uint64_t o) {
    constexpr int kU = 4;  // nodes per lane and round, their loads issued together
    const uint32_t lane = threadIdx.x & 31u, lt = lanemask_lt();
    const uint32_t shift = s - pre;  // node = place in the run + shift
    for (uint32_t x0 = 0; x0 < total; x0 += 32u * kU) {
        uint64_t kv[kU], vv[kU];
        bool live[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint32_t x = x0 + 32u * (uint32_t)u + lane;
            const uint32_t p = x + __shfl_sync(0xffffffffu, shift, (int)part_of(pre, x));
            const bool in = x < total;
            live[u] = in && !(SM[in ? p : 0u] & kTomb);
            kv[u] = in ? SK[p] : 0ull;
            vv[u] = in ? SV[p] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint32_t b = __ballot_sync(0xffffffffu, live[u]);
            if (live[u]) {
                const uint64_t w = o + (uint32_t)__popc(b & lt);
                a.keys_out[w] = kv[u];
                a.vals_out[w] = vv[u];
            }
            o += (uint32_t)__popc(b);
        }
    }
    return o;
}

// Offsets and pairs. A query whose pairs do not fit below cap gets its offset only; the queries
// that fit are the first ones, so a warp's pairs are consecutive.
__global__ void __launch_bounds__(kThreads) k_range_write(RangeArgs a, uint32_t qw) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint64_t s_sum[kThreads / 32];
    const DevMeta* m = a.m;
    if (block_sees_error(&m->error)) return;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t cur = m->cur;
    const uint32_t i = (blockIdx.x * (kThreads / 32) + warp) * qw + lane;
    const bool mine = lane < qw && i < a.n;
    const uint32_t cnt = mine ? a.cnt[i] : 0u;
    uint64_t wsum;
    const uint64_t ex = warp_excl_sum64(cnt, &wsum);
    if (lane == 0) s_sum[warp] = wsum;
    __syncthreads();
    uint64_t wbase = a.bsum[blockIdx.x];
    for (uint32_t w = 0; w < warp; ++w) wbase += s_sum[w];
    if (mine) a.offsets[i] = wbase + ex;
    const bool fits = mine && wbase + ex + cnt <= a.cap;
    const uint32_t s = fits ? a.start[i] : 0u, e = fits ? a.end[i] : 0u;
    const uint32_t len = e > s && cnt ? e - s : 0u;
    uint64_t total;
    const uint64_t pre = warp_excl_sum64(len, &total);
    const uint64_t* SK = a.st.keys[cur];
    const uint64_t* SV = a.st.vals[cur];
    const uint8_t* SM = a.st.meta[cur];
    if (total < a.run_most) {
        copy_run(a, SK, SV, SM, s, (uint32_t)pre, (uint32_t)total, wbase);
    } else {  // slices that overlap many times over: one at a time
        uint64_t o = wbase;
        for (uint32_t j = 0; j < qw; ++j) {
            const uint32_t js = __shfl_sync(0xffffffffu, s, (int)j), jl = __shfl_sync(0xffffffffu, len, (int)j);
            o = copy_run(a, SK, SV, SM, js, lane ? jl : 0u, jl, o);
        }
    }
}

}  // namespace

// Queries per warp: 32, or fewer while the warps would not fill every SM.
static uint32_t range_warp_queries(uint32_t n, int num_sms) {
    uint32_t qw = 32;
    while (qw > 1u && n / qw < (uint32_t)num_sms * 32u) qw >>= 1;
    return qw;
}

uint32_t range_blocks(uint32_t n, int num_sms) {
    const uint32_t per = range_warp_queries(n, num_sms) * (kThreads / 32);
    return (n + per - 1) / per;
}

cudaError_t launch_range(const RangeArgs& a, cudaStream_t s, int num_sms) {
    if (a.n == 0) return cudaSuccess;
    const uint32_t qw = range_warp_queries(a.n, num_sms), blocks = range_blocks(a.n, num_sms);
    launch_dep(k_range_find, blocks, kThreads, 0, s, a, qw);
    ++g_launches;
    launch_dep(k_range_write, blocks, kThreads, 0, s, a, qw);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace pi
