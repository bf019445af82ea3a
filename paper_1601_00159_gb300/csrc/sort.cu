// Sorts a query set by key (Definition 3: the queries of a query set are ordered by key;
// Section 4.2: the sort can use data parallelism); invalid queries go to its end.
//
// LSD radix sort with 8-bit digits over tiles of 2048 or 4096 elements. A tile ranks its elements
// stably and writes them staged in shared memory, so each digit's run is written
// contiguously. Where a tile's digits go comes, up to kSweepMost queries, from a decoupled
// look-back inside the pass (Merrill and Garland 2016; Adinets and Merrill, "Onesweep", 2022): one
// launch per pass, the digit counts over the whole batch having been counted by the kernel
// before. Larger batches count each tile's digits in a kernel of its own before each pass, whose
// last CTAs scan the counts, so that no tile waits for another.
// A pass whose byte is the same in every key is skipped (byte-wise min/max in the scan). The
// sort is stable, so equal keys stay in arrival order: the order is (key, arrival index), the
// reading of Definition 3 for duplicate keys.
//
// Prefix passes. When more bytes vary than the caller's pass budget (4 for batches),
// only the most significant varying bytes get passes. Keys that agree on those bytes
// then form contiguous segments, still in arrival order. Distinct keys share a segment
// only when they collide on those bytes: about D^2 / 2^33 pairs for D distinct uniform
// keys under 4 bytes, a few hundred at D = 1.2 M. Two kernels finish the order:
//   find: marks the start of every segment that holds two different keys;
//   fix:  orders each marked segment by (key, position). A warp does segments of up to
//         32 queries by counting ranks. A CTA does longer ones (a hot key that collides)
//         with a stable LSD pass per remaining byte, through buffer B.
//
// Payload word: op << 30 | arrival index. Invalid queries (op > 2 or the reserved key)
// get the sort key 2^64-1 and so gather at the end of the sorted batch.

#include "common.cuh"

namespace pi {
namespace {

constexpr int kThreads = 256;             // of the count, the scatter and the fix-up
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;
constexpr int kWarps = kThreads / 32;
constexpr int kWarpSpan = 32 * kItems;    // 256 consecutive elements per warp
static_assert(kTile == kSortTile, "tile size shared with the host's sizing");

// The first digit of a full-width batch: its four most significant bytes vary, and the passes
// start at the lowest of them. The scan counts this byte; other plans count theirs
// in the plan kernel.
constexpr uint32_t kUsualByte = 4;
constexpr uint32_t kUsualRow = 8;         // its row of the counts (rows 0 .. 7: the passes')
constexpr uint32_t kLargeTiles = 1u << 19;  // from here on, their tiles hold 4096 elements instead of 2048

// Above kSweepMost: tiles per CTA of the counting kernel, elements per warp.
constexpr uint32_t kCountTiles = 4;
constexpr uint32_t kCountSpan = kTile * kCountTiles / kWarps;
static_assert(kScanGroup % kCountTiles == 0 && kTile % kCountSpan == 0, "a CTA's tiles lie in one group");

__device__ __forceinline__ uint32_t usual_digit(uint64_t k) { return (uint32_t)(k >> (8u * kUsualByte)) & 255u; }

// Adds the digits of a thread's nv <= kN consecutive elements to the block's counts, each run
// of equal digits with one shared-memory atomic, and one per warp when the whole warp holds
// one digit, so that a hot key's run costs no contention. The whole warp calls it.
template <int kN>
__device__ __forceinline__ void count_digits(const uint32_t (&d)[kN], uint32_t nv, uint32_t* h) {
    uint32_t cur = d[0], run = nv ? 1u : 0u;
    bool single = true;
#pragma unroll
    for (int k = 1; k < kN; ++k) {
        if ((uint32_t)k >= nv) break;
        if (d[k] == cur) {
            ++run;
        } else {
            single = false;
            atomicAdd(&h[cur], run);
            cur = d[k];
            run = 1;
        }
    }
    const uint32_t d0 = __shfl_sync(0xffffffffu, cur, 0);
    if (__all_sync(0xffffffffu, single && cur == d0)) {  // the warp holds one digit
        const uint32_t tot = __reduce_add_sync(0xffffffffu, run);
        if ((threadIdx.x & 31u) == 0 && tot) atomicAdd(&h[d0], tot);
    } else if (run) {
        atomicAdd(&h[cur], run);
    }
}

// One read of the caller's queries that finds, per key byte, whether it is the same in every
// valid key (byte-wise min and max), which decides the radix passes that can be skipped, and
// counts the invalid queries. Nothing is written: the first pass reads the caller's arrays again
// and packs as it goes (writing the packed queries here and reading them back cost 12 us of 2^22
// queries). Four consecutive queries per thread and step (16-byte key loads, one 4-byte load of
// their op codes) when the arrays are aligned for it, so that every thread keeps several loads
// in flight; the byte-wise extremes are kept four bytes to a word with SIMD min/max. It also
// clears what the passes start from, the first pass's look-back words or the counts' arrivals, and the
// descent's group marks.
struct ScanAcc {
    uint32_t invalid = 0;
    uint32_t mxl = 0, mxh = 0;                  // byte-wise max of the valid keys (low, high word)
    uint32_t mnl = 0xFFFFFFFFu, mnh = 0xFFFFFFFFu;  // byte-wise min
    __device__ __forceinline__ uint64_t take(uint64_t k, uint32_t op) {
        const bool valid = op <= 2u && k != kMaxKey;
        invalid += valid ? 0u : 1u;
        if (!valid) return kMaxKey;
        mxl = __vmaxu4(mxl, (uint32_t)k);
        mxh = __vmaxu4(mxh, (uint32_t)(k >> 32));
        mnl = __vminu4(mnl, (uint32_t)k);
        mnh = __vminu4(mnh, (uint32_t)(k >> 32));
        return k;
    }
};

template <bool kSweep>
__global__ void __launch_bounds__(256) k_scan(const uint8_t* __restrict__ ops, const uint64_t* __restrict__ keys,
                                              uint32_t n, uint32_t* __restrict__ fixmap, uint32_t* __restrict__ clear,
                                              uint32_t nclear, uint32_t* __restrict__ marks, uint32_t nmarks,
                                              uint32_t* __restrict__ hist, BatchMeta* bm) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_hist[256];
    if (kSweep) {
        s_hist[threadIdx.x] = 0;
        __syncthreads();
    }
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x, gs = gridDim.x * blockDim.x;
    for (uint32_t w = gt; w < nclear; w += gs) clear[w] = 0;
    for (uint32_t w = gt; w < nmarks; w += gs) marks[w] = 0;
    for (uint32_t w = gt; w < (n + 31u) / 32u; w += gs) fixmap[w] = 0;  // segment marks of the prefix fix-up
    ScanAcc acc;
    const bool vec = ((reinterpret_cast<uintptr_t>(keys) & 15u) | (reinterpret_cast<uintptr_t>(ops) & 3u)) == 0;
    uint32_t tail = 0;  // first query left to the scalar loop
    if (vec) {
        const uint32_t n4 = n / 4u;
        for (uint32_t g0 = gt - (threadIdx.x & 31u); g0 < n4; g0 += gs) {  // whole warps
            const uint32_t g = g0 + (threadIdx.x & 31u), i = 4u * g;
            uint32_t dg[4] = {0, 0, 0, 0};
            if (g < n4) {
                const ulonglong2 k01 = reinterpret_cast<const ulonglong2*>(keys + i)[0];
                const ulonglong2 k23 = reinterpret_cast<const ulonglong2*>(keys + i)[1];
                const uint32_t o4 = ops ? *reinterpret_cast<const uint32_t*>(ops + i) : 0u;
                const uint32_t o0 = o4 & 255u, o1 = (o4 >> 8) & 255u, o2 = (o4 >> 16) & 255u, o3 = o4 >> 24;
                dg[0] = usual_digit(acc.take(k01.x, o0));
                dg[1] = usual_digit(acc.take(k01.y, o1));
                dg[2] = usual_digit(acc.take(k23.x, o2));
                dg[3] = usual_digit(acc.take(k23.y, o3));
            }
            if (kSweep) count_digits(dg, g < n4 ? 4u : 0u, s_hist);
        }
        tail = 4u * n4;
    }
    for (uint32_t i = tail + gt; i < n; i += gs) {
        const uint32_t op = ops ? ops[i] : 0u;
        const uint64_t k = acc.take(keys[i], op);
        if (kSweep) atomicAdd(&s_hist[usual_digit(k)], 1u);
    }
    uint32_t invalid = acc.invalid;
    uint32_t mx[8], mn[8];  // mn holds max of (255 - byte), so zero is the identity
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        mx[d] = (acc.mxl >> (8 * d)) & 255u;
        mx[4 + d] = (acc.mxh >> (8 * d)) & 255u;
        mn[d] = 255u - ((acc.mnl >> (8 * d)) & 255u);
        mn[4 + d] = 255u - ((acc.mnh >> (8 * d)) & 255u);
    }
    __shared__ uint32_t s_red[17];
    if (threadIdx.x < 17) s_red[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        mx[d] = __reduce_max_sync(0xffffffffu, mx[d]);
        mn[d] = __reduce_max_sync(0xffffffffu, mn[d]);
    }
    invalid = __reduce_add_sync(0xffffffffu, invalid);
    if ((threadIdx.x & 31) == 0) {
        if (invalid) atomicAdd(&s_red[16], invalid);
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            atomicMax(&s_red[d], mx[d]);
            atomicMax(&s_red[8 + d], mn[d]);
        }
    }
    __syncthreads();
    if (kSweep && s_hist[threadIdx.x]) atomicAdd(&hist[kUsualRow * 256u + threadIdx.x], s_hist[threadIdx.x]);
    // one global atomic per byte per CTA
    if (threadIdx.x < 8) atomicMax(&bm->bmax[threadIdx.x], s_red[threadIdx.x]);
    else if (threadIdx.x < 16) atomicMax(&bm->bnmin[threadIdx.x - 8], s_red[threadIdx.x]);
    else if (threadIdx.x == 16 && s_red[16]) atomicAdd(&bm->invalid, s_red[16]);
}

// Query i of the caller, as the sort takes it: invalid queries get the key 2^64-1.
__device__ __forceinline__ void load_query(const SortBuffers& sb, uint32_t i, uint64_t& key, uint32_t& pay) {
    const uint32_t op = sb.ops ? sb.ops[i] : 0u;
    const uint64_t k = sb.keys[i];
    key = op <= 2u ? k : kMaxKey;
    pay = ((op & 3u) << 30) | i;
}

// Digits of the caller's queries i0 .. i0 + nv - 1 (nv <= 8, i0 a multiple of 8), with 16-byte key
// loads and an 8-byte load of the op codes when the arrays are aligned for them.
__device__ __forceinline__ void query_digits(const SortBuffers& sb, uint32_t i0, uint32_t nv, uint32_t shift,
                                             uint32_t (&dg)[8]) {
    const bool vec = ((reinterpret_cast<uintptr_t>(sb.keys) & 15u) | (reinterpret_cast<uintptr_t>(sb.ops) & 7u)) == 0;
    if (vec && nv == 8u) {
        const ulonglong2* p = reinterpret_cast<const ulonglong2*>(sb.keys + i0);
        const uint2 o = sb.ops ? *reinterpret_cast<const uint2*>(sb.ops + i0) : make_uint2(0u, 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const ulonglong2 v = p[k];
            const uint32_t w = (k < 2 ? o.x : o.y) >> (16 * (k & 1));
            dg[2 * k] = (w & 255u) <= 2u ? (uint32_t)(v.x >> shift) & 255u : 255u;
            dg[2 * k + 1] = ((w >> 8) & 255u) <= 2u ? (uint32_t)(v.y >> shift) & 255u : 255u;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            uint64_t key = 0;
            uint32_t pay;
            if ((uint32_t)k < nv) load_query(sb, i0 + k, key, pay);
            dg[k] = (uint32_t)(key >> shift) & 255u;
        }
    }
}

// Pass plan. The digit bytes D are the bytes that vary among the valid keys. Invalid
// queries carry the sort key 2^64-1 and must follow every valid key: when there are
// some, D also holds the highest byte p whose maximum over the valid keys is below 0xFF
// (every invalid key is larger there; with no such byte D is every byte). Passes
// ping-pong so that the last one writes buffer A.
// With more than max_passes bytes in D, the passes take the most significant
// max_passes of them (the prefix). The fix-up then orders each segment of equal prefix
// bytes by the full key; its long-segment path sorts by every other byte that can
// differ inside a segment (rdig).
// This kernel plans for the passes with a look-back, and counts the first pass's digits when they are
// not those that the scan has counted.
__global__ void __launch_bounds__(256) k_sort_plan(uint32_t n, SortBuffers sb, BatchMeta* bm, uint32_t max_passes) {
    pdl_wait();
    pdl_trigger();
    __shared__ SortPlan s_plan;
    __shared__ uint32_t s_hist[256];
    if (threadIdx.x == 0) {
        plan_digits(bm->bmax, bm->bnmin, bm->invalid, n, max_passes, s_plan);
        if (blockIdx.x == 0) bm->plan = s_plan;
    }
    s_hist[threadIdx.x] = 0;
    __syncthreads();
    if (s_plan.digit[0] == kUsualByte) return;  // counted by the scan
    const uint32_t shift = 8u * s_plan.digit[0];
    for (uint32_t base = blockIdx.x * 2048u; base < n; base += gridDim.x * 2048u) {
        const uint32_t i0 = base + threadIdx.x * 8u;
        const uint32_t nv = i0 < n ? min(8u, n - i0) : 0u;
        uint32_t dg[8];
        query_digits(sb, i0, nv, shift, dg);
        count_digits(dg, nv, s_hist);
    }
    __syncthreads();
    if (s_hist[threadIdx.x]) atomicAdd(&sb.hist[threadIdx.x], s_hist[threadIdx.x]);
}

// Look-back word of one digit of one tile: flag (2 bits) | count (30). 0: not published yet.
// Words are cleared between uses: a pass clears its tiles' words of the other buffer for the
// next pass, and the scan those of the first.
constexpr uint32_t kWordAgg = 1u << 30, kWordPrefix = 2u << 30, kWordMask = kWordAgg - 1u;

// Sum of one digit's counts over the tiles before `tile`: 16 tiles' words per round, which the
// threads of the digits read as rows. A wait that gives up records kErrTimeout and returns
// false.
__device__ __forceinline__ bool digit_lookback(const uint32_t* words, uint32_t tile, uint32_t* err, uint32_t& sum) {
    constexpr int kWin = 16;
    uint32_t excl = 0, spins = 0;
    int64_t t = (int64_t)tile - 1;
    while (t >= 0) {
        uint32_t w[kWin];
#pragma unroll
        for (int i = 0; i < kWin; ++i) w[i] = t - i >= 0 ? ld_relaxed32(words + (size_t)(t - i) * 256) : kWordPrefix;
        bool stop = false, stall = false;
        int used = 0;
#pragma unroll
        for (int i = 0; i < kWin; ++i) {
            if (stop || stall) continue;
            if (w[i] == 0) {
                stall = true;
                continue;
            }
            excl += w[i] & kWordMask;
            ++used;
            stop = (w[i] & kWordPrefix) != 0;
        }
        if (stop) break;
        t -= used;
        if (stall) {
            ++spins;
            if (spins > kSpinLimit) {
                atomicOr(err, kErrTimeout);
                return false;
            }
            if ((spins & 1023u) == 0 && *(volatile uint32_t*)err) return false;
            if (spins > 32) __nanosleep(100);
        }
    }
    sum = excl;
    return true;
}

// One pass: tiles of kPassThreads x kI elements. Bound by issue slots and shared memory in the
// ranking (nine ballots and an atomic per element row); the look-back's wait overlaps the
// other CTA of the SM. Larger tiles mean fewer look-backs in flight, smaller ones more CTAs for
// batches that would leave SMs idle.
constexpr int kPassThreads = 512;
constexpr int kPassWarps = kPassThreads / 32;
template <int kI>
constexpr int pass_smem() {
    return kPassThreads * kI * (int)(sizeof(uint64_t) + sizeof(uint32_t)) + kPassWarps * 256 * 4;
}

template <int kI>
__global__ void __launch_bounds__(kPassThreads, 2) k_sort_pass(uint32_t j, uint32_t n, SortBuffers sb, BatchMeta* bm,
                                                               uint32_t* err) {
    pdl_wait();
    pdl_trigger();
    constexpr uint32_t kT = kPassThreads * kI;
    const SortPlan& P = bm->plan;
    if (j >= P.npass) return;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    uint64_t* s_key = reinterpret_cast<uint64_t*>(s_dyn);
    uint32_t* s_pay = reinterpret_cast<uint32_t*>(s_dyn + kT * sizeof(uint64_t));
    uint32_t(*s_whist)[256] = reinterpret_cast<uint32_t(*)[256]>(s_dyn + kT * 12u);
    __shared__ uint32_t s_gbase[256], s_tstart[256], s_next[256];
    __shared__ uint32_t s_tmp[33], s_tile;
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_tile = atomicAdd(&bm->tile_ctr[j], 1u);
        s_fail = 0;
    }
    for (int i = tid; i < kPassWarps * 64; i += kPassThreads)
        reinterpret_cast<uint4*>(&s_whist[0][0])[i] = make_uint4(0, 0, 0, 0);
    if (tid < 256) s_next[tid] = 0;
    const uint32_t shift = 8u * P.digit[j];
    const bool caller = P.src[j] == 0;  // the first pass reads the caller's queries
    const uint64_t* src_k = P.src[j] == 1 ? sb.a_k : sb.b_k;
    const uint32_t* src_p = P.src[j] == 1 ? sb.a_p : sb.b_p;
    uint64_t* dst_k = P.dst[j] == 1 ? sb.a_k : sb.b_k;
    uint32_t* dst_p = P.dst[j] == 1 ? sb.a_p : sb.b_p;
    const uint32_t row = j == 0 && P.digit[0] == kUsualByte ? kUsualRow : j;
    const uint32_t all = tid < 256 ? sb.hist[row * 256u + (uint32_t)tid] : 0u;  // the batch's count of digit tid
    uint32_t* words = j & 1u ? sb.desc[1] : sb.desc[0];
    uint32_t* other = j & 1u ? sb.desc[0] : sb.desc[1];
    __syncthreads();
    const uint32_t tile = s_tile, tbase = tile * kT, tn = min(kT, n - tbase);

    uint64_t key[kI];
    uint32_t pay[kI], dig[kI], rank[kI];
#pragma unroll
    for (int k = 0; k < kI; ++k) {
        const uint32_t li = (uint32_t)(warp * 32 * kI + k * 32 + lane);
        const bool v = li < tn;
        key[k] = 0ull;
        pay[k] = 0u;
        if (v) {
            if (caller) {
                load_query(sb, tbase + li, key[k], pay[k]);
            } else {
                key[k] = src_k[tbase + li];
                pay[k] = src_p[tbase + li];
            }
        }
        dig[k] = v ? (uint32_t)((key[k] >> shift) & 255u) : 256u;
    }
    const uint32_t dbase = block_excl_sum<kPassThreads>(all, s_tmp, nullptr);  // the digit's first output slot
    warp_digit_ranks<kI, 8>(dig, rank, s_whist[warp]);
    __syncthreads();
    // Thread d < 256 owns digit d: the tile's count is published, and each warp's first rank.
    uint32_t total = 0;
    if (tid < 256) {
#pragma unroll
        for (int w = 0; w < kPassWarps; ++w) {
            const uint32_t c = s_whist[w][tid];
            s_whist[w][tid] = total;
            total += c;
        }
        atomicExch(&words[(size_t)tile * 256 + tid], (tile == 0 ? kWordPrefix : kWordAgg) | total);
        other[(size_t)tile * 256 + tid] = 0;  // for the next pass
    }
    const uint32_t tstart = block_excl_sum<kPassThreads>(total, s_tmp, nullptr);
    if (tid < 256) s_tstart[tid] = tstart;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kI; ++k) {
        const uint32_t d = dig[k];
        if (d < 256u) {
            const uint32_t pos = s_tstart[d] + s_whist[warp][d] + rank[k];
            s_key[pos] = key[k];
            s_pay[pos] = pay[k];
        }
    }
    if (tid < 256) {
        uint32_t before = 0;
        if (tile > 0) {
            if (!digit_lookback(words + tid, tile, err, before)) s_fail = 1;
            atomicExch(&words[(size_t)tile * 256 + tid], kWordPrefix | (before + total));
        }
        s_gbase[tid] = dbase + before - tstart;  // output slot = this + place in the tile
    }
    __syncthreads();
    if (s_fail) return;
    const bool next = j + 1 < P.npass;
    const uint32_t nshift = next ? 8u * P.digit[j + 1] : 0u;
    for (uint32_t s0 = 0; s0 < tn; s0 += kPassThreads) {
        const uint32_t s = s0 + (uint32_t)tid;
        const bool in = s < tn;
        const uint64_t k = in ? s_key[s] : 0ull;
        if (in) {
            const uint32_t g = s_gbase[(uint32_t)(k >> shift) & 255u] + s;
            if (g < n) {
                dst_k[g] = k;
                dst_p[g] = s_pay[s];
            } else {
                atomicOr(err, kErrBounds);
            }
        }
        if (next) {  // the next pass's digit counts; a hot key's run is one atomic per warp
            const uint32_t nd = in ? (uint32_t)(k >> nshift) & 255u : 256u;
            const uint32_t d0 = __shfl_sync(0xffffffffu, nd, 0);
            if (__all_sync(0xffffffffu, nd == d0)) {
                if (lane == 0 && d0 < 256u) atomicAdd(&s_next[d0], 32u);
            } else if (in) {
                atomicAdd(&s_next[nd], 1u);
            }
        }
    }
    if (next) {
        __syncthreads();
        if (tid < 256 && s_next[tid]) atomicAdd(&sb.hist[(j + 1u) * 256u + (uint32_t)tid], s_next[tid]);
    }
}

// ---------------------------------------------------------------------------------
// Batches above kSweepMost: a counting and a scattering kernel per pass. With hundreds of tiles
// in flight the look-back costs more than a launch that reads one digit byte per element:
// 2^22 queries on 2^27 keys took 571 us a batch with k_sort_pass and 544 with these two; at 2^20
// queries k_sort_pass is ahead (428 against 432), and at 10^5 by 21 of 99 us.

// Exclusive running sum, per digit (thread d), over `rows` rows of 256 counters starting
// at `in`: writes each row's prefix to `out` (may equal `in`) and returns the total.
__device__ __forceinline__ uint32_t scan_rows(const uint32_t* in, uint32_t* out, uint32_t rows) {
    const uint32_t d = threadIdx.x;
    constexpr int kRows = 32;
    uint32_t run = 0;
    for (uint32_t t = 0; t < rows; t += kRows) {
        uint32_t c[kRows];
#pragma unroll
        for (int k = 0; k < kRows; ++k) c[k] = (t + (uint32_t)k < rows) ? __ldcg(&in[(size_t)(t + k) * 256 + d]) : 0u;
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            if (t + (uint32_t)k < rows) {
                out[(size_t)(t + k) * 256 + d] = run;
                run += c[k];
            }
        }
    }
    return run;
}

// Digit histogram of every tile for pass j, then its scan, by the CTAs that finish
// last (no CTA waits for another): the last CTA of each group of kScanGroup tiles turns
// the group's counts into offsets within the group (toff) and the group's digit totals
// (gsum); the last group to finish turns those totals into the groups' offsets, in
// place, and the digit totals into digit bases (dofs). A tile's first output slot for
// digit d is then dofs[d] + gsum[group][d] + toff[tile][d]. Pass 0 (kFirst) plans the digits,
// in every CTA, and reads the caller's keys; later passes read the digit bytes the previous
// scatter wrote beside its output. A thread takes 8 consecutive elements a step and adds each
// run of equal digits with one shared-memory atomic (one per warp when the whole warp holds
// one digit), so a run of a hot key costs no atomic contention.
// The kernel is bound by its chain of dependent round trips, not by the bytes: so a CTA counts
// four tiles (2^22 queries are then one wave of 512 CTAs, not three of 2048 with one tile
// each), with every load of digit bytes in flight, and the scans load 32 rows per round trip.
// 2^22 queries on 2^27 keys took 504 us a batch with one tile per CTA, 16 rows and a kernel of
// its own for the plan, and take 497. Tiles of 4096 elements, which need half the rows, left the
// counts as they were and cost the scatter 8 us.
template <bool kFirst>
__global__ void __launch_bounds__(kThreads, 4) k_sort_count(uint32_t j, uint32_t n, SortBuffers sb, BatchMeta* bm,
                                                            uint32_t max_passes) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t h[kCountTiles][256];
    __shared__ uint32_t s_tmp[33];
    __shared__ uint32_t s_last;
    __shared__ SortPlan s_plan;
    if (!kFirst && j >= bm->plan.npass) return;
    if (kFirst && threadIdx.x == 0) {
        plan_digits(bm->bmax, bm->bnmin, bm->invalid, n, max_passes, s_plan);
        if (blockIdx.x == 0) bm->plan = s_plan;
    }
#pragma unroll
    for (uint32_t t = 0; t < kCountTiles; ++t) h[t][threadIdx.x] = 0;
    __syncthreads();
    // A warp reads kCountSpan consecutive elements of one tile, 8 per lane and step.
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t* ht = h[warp / (kTile / kCountSpan)];
    const uint32_t wbase = (blockIdx.x * kWarps + warp) * kCountSpan + lane * 8u;
    if (kFirst) {
        const uint32_t shift = 8u * s_plan.digit[0];
#pragma unroll 1
        for (uint32_t i0 = wbase; i0 < wbase + kCountSpan; i0 += 256u) {
            const uint32_t nv = i0 < n ? min(8u, n - i0) : 0u;
            uint32_t dg[8];
            query_digits(sb, i0, nv, shift, dg);
            count_digits(dg, nv, ht);
        }
    } else {
        constexpr int kSteps = kCountSpan / 256u;
        uint2 v[kSteps];
#pragma unroll
        for (int u = 0; u < kSteps; ++u) {  // 8 digit bytes a load, every load in flight
            const uint32_t i0 = wbase + (uint32_t)u * 256u;
            v[u] = i0 < n ? *reinterpret_cast<const uint2*>(sb.ndig + i0) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kSteps; ++u) {
            const uint32_t i0 = wbase + (uint32_t)u * 256u;
            uint32_t dg[8];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                dg[k] = (v[u].x >> (8 * k)) & 255u;
                dg[4 + k] = (v[u].y >> (8 * k)) & 255u;
            }
            count_digits(dg, i0 < n ? min(8u, n - i0) : 0u, ht);
        }
    }
    __syncthreads();
    const uint32_t d = threadIdx.x;
    const uint32_t tile = blockIdx.x * kCountTiles, ntiles = (n + kTile - 1) / kTile;
#pragma unroll
    for (uint32_t t = 0; t < kCountTiles; ++t)
        if (tile + t < ntiles) sb.tcnt[(size_t)(tile + t) * 256 + d] = h[t][d];
    const uint32_t g = tile / kScanGroup, ngroups = (ntiles + kScanGroup - 1) / kScanGroup;
    const uint32_t t0 = g * kScanGroup, t1 = min(t0 + kScanGroup, ntiles);
    uint32_t* ctr = sb.gctr + (size_t)j * (ngroups + 1);
    // Arrival: the block barrier orders every thread's counts before thread 0's fence,
    // which (being cumulative) releases them all before its atomic; the last CTA's
    // thread 0 fences after the atomic and the barrier passes that on to its threads.
    __syncthreads();
    if (d == 0) {
        __threadfence();
        s_last = atomicAdd(&ctr[g], 1u) == (t1 - t0 + kCountTiles - 1u) / kCountTiles - 1u;
        if (s_last) __threadfence();  // every CTA of the group has arrived: their counts are visible
    }
    __syncthreads();
    if (!s_last) return;
    sb.gsum[(size_t)g * 256 + d] = scan_rows(sb.tcnt + (size_t)t0 * 256, sb.toff + (size_t)t0 * 256, t1 - t0);
    __syncthreads();
    if (d == 0) {
        __threadfence();
        s_last = atomicAdd(&ctr[ngroups], 1u) == ngroups - 1u;
        if (s_last) __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    const uint32_t run = scan_rows(sb.gsum, sb.gsum, ngroups);
    sb.dofs[d] = block_excl_sum<kThreads>(run, s_tmp, nullptr);  // digit bases of this pass
}


__global__ void __launch_bounds__(kThreads, 4) k_sort_scatter(uint32_t j, uint32_t n, SortBuffers sb,
                                                           BatchMeta* bm, uint32_t* err) {
    pdl_wait();
    pdl_trigger();
    const SortPlan& P = bm->plan;
    if (j >= P.npass) return;
    const uint32_t shift = 8u * P.digit[j];
    const bool caller = P.src[j] == 0;  // the first pass reads the caller's queries
    const uint64_t* src_k = P.src[j] == 1 ? sb.a_k : sb.b_k;
    const uint32_t* src_p = P.src[j] == 1 ? sb.a_p : sb.b_p;
    uint64_t* dst_k = P.dst[j] == 1 ? sb.a_k : sb.b_k;
    uint32_t* dst_p = P.dst[j] == 1 ? sb.a_p : sb.b_p;

    extern __shared__ __align__(16) uint8_t s_dyn[];
    uint64_t* s_key = reinterpret_cast<uint64_t*>(s_dyn);
    uint32_t* s_pay = reinterpret_cast<uint32_t*>(s_dyn + kTile * sizeof(uint64_t));
    __shared__ uint32_t s_whist[kWarps][256];
    __shared__ uint32_t s_gbase[256];
    __shared__ uint32_t s_tstart[256];
    __shared__ uint32_t s_tmp[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < kWarps * 256; i += kThreads) (&s_whist[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = blockIdx.x;
    const uint32_t tbase = tile * kTile;
    const uint32_t tn = min((uint32_t)kTile, n - tbase);

    uint64_t key[kItems];
    uint32_t pay[kItems];
    uint32_t dig[kItems];
    uint32_t rank[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        uint32_t li = warp * kWarpSpan + k * 32 + lane;
        bool v = li < tn;
        key[k] = 0ull;
        pay[k] = 0u;
        if (v) {
            if (caller) {
                load_query(sb, tbase + li, key[k], pay[k]);
            } else {
                key[k] = src_k[tbase + li];
                pay[k] = src_p[tbase + li];
            }
        }
        dig[k] = v ? (uint32_t)((key[k] >> shift) & 255u) : 256u;
    }
    warp_digit_ranks<kItems, 8>(dig, rank, s_whist[warp]);
    __syncthreads();
    // Thread tid owns digit tid: tile total and per-warp exclusive prefix.
    uint32_t total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        uint32_t c = s_whist[w][tid];
        s_whist[w][tid] = total;
        total += c;
    }
    s_gbase[tid] = sb.dofs[tid] + sb.gsum[(size_t)(tile / kScanGroup) * 256 + tid] +
                   sb.toff[(size_t)tile * 256 + tid];
    s_tstart[tid] = block_excl_sum<kThreads>(total, s_tmp, nullptr);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        uint32_t d = dig[k];
        if (d < 256u) {
            uint32_t pos = s_tstart[d] + s_whist[warp][d] + rank[k];
            s_key[pos] = key[k];
            s_pay[pos] = pay[k];
        }
    }
    __syncthreads();
    const bool next = j + 1 < P.npass;
    const uint32_t nshift = next ? 8u * P.digit[j + 1] : 0u;
    for (uint32_t s = tid; s < tn; s += kThreads) {
        uint64_t k = s_key[s];
        uint32_t d = (uint32_t)((k >> shift) & 255u);
        uint32_t g = s_gbase[d] + (s - s_tstart[d]);
        if (g < n) {
            dst_k[g] = k;
            dst_p[g] = s_pay[s];
            if (next) sb.ndig[g] = (uint8_t)(k >> nshift);  // the next pass's digit
        } else {
            atomicOr(err, kErrBounds);
        }
    }
}

// ---------------------------------------------------------------------------------
// Prefix fix-up. After the prefix passes buffer A is sorted by key & pmask ("the
// prefix"), and positions with equal prefix hold their queries in arrival order.

// Marks (in fixmap) the first position of every segment of equal prefix that holds two
// different keys. A position i whose key differs from key i-1 but whose prefix does not
// lies inside such a segment; the segment's start is found by a galloping search back
// from i followed by a binary search, both over the prefix order.
__global__ void __launch_bounds__(256) k_sort_find(uint32_t n, SortBuffers sb, const BatchMeta* bm, bool sweep) {
    pdl_wait();
    pdl_trigger();
    const SortPlan& P = bm->plan;
    if (sweep && blockIdx.x == 0)  // the passes are done with the counts: zero for the next sort
        for (uint32_t w = threadIdx.x; w < kSortHist; w += 256u) sb.hist[w] = 0;
    if (!P.fix) return;
    const uint64_t pm = P.pmask;
    const uint64_t* __restrict__ ak = sb.a_k;
    const uint32_t lane = threadIdx.x & 31u;
    constexpr int kU = 4;  // positions per thread and step, loaded together
    for (uint32_t base = blockIdx.x * 256u * kU; base < n; base += gridDim.x * 256u * kU) {
        uint64_t k1[kU], k0[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint32_t i = base + (uint32_t)u * 256u + threadIdx.x;
            k1[u] = i < n ? ak[i] : 0ull;
            k0[u] = (lane == 0 && i > 0 && i < n) ? ak[i - 1] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint32_t i = base + (uint32_t)u * 256u + threadIdx.x;
            uint64_t kp = __shfl_up_sync(0xffffffffu, k1[u], 1);
            if (lane == 0) kp = k0[u];
            if (i == 0 || i >= n || kp == k1[u] || ((kp ^ k1[u]) & pm) != 0) continue;
            const uint64_t mk = k1[u] & pm;
            uint32_t in = i - 1;  // ak[in] is in the segment
            uint64_t d = 1;
            while (d <= in && (ak[in - d] & pm) == mk) {
                in -= (uint32_t)d;
                d <<= 1;
            }
            uint32_t lo = d <= in ? in - (uint32_t)d + 1 : 0u, hi = in;  // the start lies in [lo, hi]
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if ((ak[mid] & pm) == mk) hi = mid;
                else lo = mid + 1;
            }
            atomicOr(&sb.fixmap[lo >> 5], 1u << (lo & 31u));
        }
    }
}

constexpr int kFixSlice = kThreads * 32;  // positions per fix-up CTA: one fixmap word per thread

// Stable LSD sort of the segment [s, e) of buffer A by the bytes P.rdig (ascending),
// by the whole CTA, through the same range of buffer B. The segment is in arrival
// order, so the result is in (key, arrival) order.
__device__ void cta_segment_lsd(uint32_t s, uint32_t e, const SortPlan& P, const SortBuffers& sb,
                                uint32_t (*s_whist)[256], uint32_t* s_base, uint32_t* s_tmp) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t* src_k = sb.a_k;
    uint32_t* src_p = sb.a_p;
    uint64_t* dst_k = sb.b_k;
    uint32_t* dst_p = sb.b_p;
    for (uint32_t r = 0; r < P.nr; ++r) {
        const uint32_t shift = 8u * P.rdig[r];
        for (int w = 0; w < kWarps; ++w) s_whist[w][tid] = 0;
        s_base[tid] = 0;
        __syncthreads();
        for (uint32_t i = s + tid; i < e; i += kThreads) atomicAdd(&s_base[(uint32_t)(src_k[i] >> shift) & 255u], 1u);
        __syncthreads();
        const uint32_t cnt = s_base[tid];
        __syncthreads();
        s_base[tid] = s + block_excl_sum<kThreads>(cnt, s_tmp, nullptr);
        __syncthreads();
        for (uint32_t c = s; c < e; c += kTile) {
            uint64_t key[kItems];
            uint32_t pay[kItems], dig[kItems], rank[kItems];
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                const uint32_t i = c + warp * kWarpSpan + k * 32 + lane;
                const bool v = i < e;
                key[k] = v ? src_k[i] : 0ull;
                pay[k] = v ? src_p[i] : 0u;
                dig[k] = v ? (uint32_t)((key[k] >> shift) & 255u) : 256u;
            }
            warp_digit_ranks<kItems, 8>(dig, rank, s_whist[warp]);
            __syncthreads();
            uint32_t total = 0;  // thread tid owns digit tid: per-warp exclusive prefix
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t cc = s_whist[w][tid];
                s_whist[w][tid] = total;
                total += cc;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                const uint32_t d = dig[k];
                if (d < 256u) {
                    const uint32_t pos = s_base[d] + s_whist[warp][d] + rank[k];
                    if (pos >= s && pos < e) {
                        dst_k[pos] = key[k];
                        dst_p[pos] = pay[k];
                    }
                }
            }
            __syncthreads();
            s_base[tid] += total;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) s_whist[w][tid] = 0;
            __syncthreads();
        }
        uint64_t* tk = src_k; src_k = dst_k; dst_k = tk;
        uint32_t* tp = src_p; src_p = dst_p; dst_p = tp;
    }
    if (src_k != sb.a_k) {  // an odd number of passes left the result in B
        for (uint32_t i = s + tid; i < e; i += kThreads) {
            sb.a_k[i] = src_k[i];
            sb.a_p[i] = src_p[i];
        }
    }
    __syncthreads();
}

// Orders the segment [s, e) of buffer A by the bytes the prefix passes skipped, for a
// segment of at most one tile: it is read into registers once, every pass ranks it and
// places it in shared memory (s_k, s_p: kTile entries) in digit order, the next pass
// reads it back from there, and the result is written to A once. Stable.
__device__ void cta_segment_smem(uint32_t s, uint32_t e, const SortPlan& P, const SortBuffers& sb,
                                 uint64_t* s_k, uint32_t* s_p, uint32_t (*s_whist)[256], uint32_t* s_base,
                                 uint32_t* s_tmp) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t L = e - s;
    uint64_t key[kItems];
    uint32_t pay[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t li = (uint32_t)(warp * kWarpSpan + k * 32 + lane);
        key[k] = li < L ? sb.a_k[s + li] : 0ull;
        pay[k] = li < L ? sb.a_p[s + li] : 0u;
    }
    for (int w = 0; w < kWarps; ++w) s_whist[w][tid] = 0;
    __syncthreads();
    for (uint32_t r = 0; r < P.nr; ++r) {
        const uint32_t shift = 8u * P.rdig[r];
        uint32_t dig[kItems], rank[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t li = (uint32_t)(warp * kWarpSpan + k * 32 + lane);
            dig[k] = li < L ? (uint32_t)((key[k] >> shift) & 255u) : 256u;
        }
        warp_digit_ranks<kItems, 8>(dig, rank, s_whist[warp]);
        __syncthreads();
        uint32_t total = 0;  // thread tid owns digit tid: per-warp exclusive prefix
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t cc = s_whist[w][tid];
            s_whist[w][tid] = total;
            total += cc;
        }
        s_base[tid] = block_excl_sum<kThreads>(total, s_tmp, nullptr);  // the digit's first slot
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t d = dig[k];
            if (d < 256u) {
                const uint32_t pos = s_base[d] + s_whist[warp][d] + rank[k];
                s_k[pos] = key[k];
                s_p[pos] = pay[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t li = (uint32_t)(warp * kWarpSpan + k * 32 + lane);
            if (li < L) {
                key[k] = s_k[li];
                pay[k] = s_p[li];
            }
        }
        for (int w = 0; w < kWarps; ++w) s_whist[w][tid] = 0;
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const uint32_t li = (uint32_t)(warp * kWarpSpan + k * 32 + lane);
        if (li < L) {
            sb.a_k[s + li] = key[k];
            sb.a_p[s + li] = pay[k];
        }
    }
    __syncthreads();
}

// Orders every marked segment. Each CTA reads kThreads fixmap words (kFixSlice
// positions) and takes the segments that start there. A warp orders a segment of at
// most 32 queries: rank = queries with a smaller key, or the same key and an earlier
// position. Longer segments are queued for the whole CTA.
__global__ void __launch_bounds__(kThreads) k_sort_fix(uint32_t n, SortBuffers sb, BatchMeta* bm, bool long_too) {
    pdl_wait();
    pdl_trigger();
    const SortPlan& P = bm->plan;
    if (!P.fix) return;
    // segment starts (a segment holds >= 2 queries); then the keys of a long segment
    // ordered in shared memory
    __shared__ __align__(16) uint32_t s_list[kFixSlice / 2];
    __shared__ uint32_t s_pay[kTile];
    static_assert(kFixSlice / 2 * sizeof(uint32_t) >= kTile * sizeof(uint64_t), "a tile's keys fit s_list");
    __shared__ uint32_t s_big[kFixSlice / 32 + 1];  // starts of segments of more than 32
    __shared__ uint32_t s_nbig, s_end;
    __shared__ uint32_t s_tmp[33];
    __shared__ uint32_t s_whist[kWarps][256];
    __shared__ uint32_t s_base[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nwords = (n + 31u) / 32u;
    const uint32_t wi = blockIdx.x * kThreads + tid;
    uint32_t w = wi < nwords ? sb.fixmap[wi] : 0u;
    uint32_t total;
    uint32_t off = block_excl_sum<kThreads>((uint32_t)__popc(w), s_tmp, &total);
    while (w) {
        const uint32_t b = (uint32_t)(__ffs(w) - 1);
        w &= w - 1;
        if (off < kFixSlice / 2) s_list[off] = wi * 32u + b;  // starts are >= 2 apart: always true
        ++off;
    }
    if (tid == 0) s_nbig = 0;
    __syncthreads();
    if (total == 0) return;
    if (total > kFixSlice / 2) total = kFixSlice / 2;
    const uint64_t pm = P.pmask;
    const uint64_t* ak = sb.a_k;
    for (uint32_t x = warp; x < total; x += kWarps) {
        const uint32_t s = s_list[x];
        const uint64_t mk = ak[s] & pm;
        const uint32_t i = s + lane;
        // The segment's queries are the lanes of a prefix of the warp (prefix order).
        const uint64_t key = i < n ? ak[i] : 0ull;
        const bool in = i < n && (key & pm) == mk;
        const uint32_t m = (uint32_t)__popc(__ballot_sync(0xffffffffu, in));
        const bool longer = m == 32u && s + 32u < n && (ak[s + 32u] & pm) == mk;
        if (longer) {
            if (lane == 0) {
                const uint32_t slot = atomicAdd(&s_nbig, 1u);
                if (slot < kFixSlice / 32 + 1) s_big[slot] = s;  // starts are > 32 apart: always true
            }
            continue;
        }
        const uint32_t pay = in ? sb.a_p[i] : 0u;
        uint32_t rank = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const uint64_t kj = __shfl_sync(0xffffffffu, key, j);
            rank += ((uint32_t)j < m && (kj < key || (kj == key && j < lane))) ? 1u : 0u;
        }
        __syncwarp();
        if (in) {
            sb.a_k[s + rank] = key;
            sb.a_p[s + rank] = pay;
        }
    }
    __syncthreads();
    const uint32_t nbig = min(s_nbig, (uint32_t)(kFixSlice / 32 + 1));
    for (uint32_t x = 0; x < nbig; ++x) {
        const uint32_t s = s_big[x];
        if (warp == 0) {
            // End of the segment, by the first warp: lane l probes s + 32 + 2^l - 1 (a
            // gallop in one round), then 32-way rounds narrow the bracket. The segment's
            // positions are a prefix of [s + 32, n), so each round's hits are a prefix.
            const uint64_t mk = ak[s] & pm;
            const uint32_t base = s + 32u;  // in the segment
            const uint64_t off = (1ull << lane) - 1ull;
            const bool hit = base + off < n && (ak[base + off] & pm) == mk;
            const uint32_t hm = __ballot_sync(0xffffffffu, hit);  // lane 0 always hits
            const int top = 31 - __clz(hm);
            uint32_t lo = base + ((1u << top) - 1u) + 1u;  // past the last position known in it
            const uint64_t qn = (uint64_t)base + (2ull << top) - 1ull;  // the first probe past it
            uint32_t hi = (top < 31 && qn < (uint64_t)n) ? (uint32_t)qn : n;  // not in it (or n)
            while (hi > lo) {  // the end lies in [lo, hi]
                const uint32_t step = (hi - lo + 31u) / 32u;
                const uint32_t p = lo + lane * step;
                const bool in = p < hi && (ak[p] & pm) == mk;
                const uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, in));
                if (c == 0) break;  // lo itself is past the segment
                const uint32_t nlo = lo + (c - 1u) * step + 1u;
                const uint32_t nhi = lo + c * step;
                lo = nlo;
                hi = nhi < hi ? nhi : hi;
            }
            if (lane == 0) {
                s_end = lo;
                atomicAdd(&bm->fix_big, lo - s);
            }
        }
        __syncthreads();
        if (!long_too) continue;
        if (s_end - s <= (uint32_t)kTile)
            cta_segment_smem(s, s_end, P, sb, reinterpret_cast<uint64_t*>(s_list), s_pay, s_whist, s_base, s_tmp);
        else
            cta_segment_lsd(s, s_end, P, sb, s_whist, s_base, s_tmp);
    }
}

// ---------------------------------------------------------------------------------
// Small batches (at most kSmallSort queries): instead of the radix pipeline's chain of
// dependent launches, every CTA sorts one tile of kRunTile consecutive queries by
// (key, arrival) in shared memory and leaves it sorted in in_k / in_p; the descent's
// k_rank_locate then finds each query's place among the other tiles. Such a batch is bound
// by launches and dependent latency, not by memory. A warp orders runs of 8 by counting,
// then the runs merge pairwise: an element's place is its place in its own run plus the count
// of the sibling run's smaller keys (or equal ones, when the sibling is the earlier run, which
// keeps arrival order). Consecutive lanes hold consecutive keys, so a merge's probes mostly
// share shared-memory wavefronts. The kernel is bound by issue slots: the levels are unrolled
// (a probe is a load, a 64-bit compare and an add), the levels inside a warp's 64 elements need
// no block barrier, and a tile that is not full stops merging at its length.
// Measured, 2^14 searches on 2^16 keys: sort and look-up took 15 launches and 89 us between
// events, as two launches 29; the batch went from 98 to 56 us by this (28 with the launches and
// host work around it cut since). 2^10 queries on 50,021 keys: 92 to 54 us a batch (26 since).
constexpr int kRunThreads = kRunTile / 2;  // two elements per thread, 64 consecutive ones per warp

// Keys of the sorted run[0, kLen) below x.
template <uint32_t kLen>
__device__ __forceinline__ uint32_t count_below(const uint64_t* run, uint64_t x) {
    uint32_t c = 0;
#pragma unroll
    for (uint32_t step = kLen / 2; step > 0; step >>= 1)
        if (run[c + step - 1] < x) c += step;
    return run[c] < x ? c + 1u : c;
}

struct RunBuffers {
    uint64_t k[2][kRunTile];
    uint16_t i[2][kRunTile];  // op << 11 | position in the tile
};
static_assert(kRunTile <= 2048, "11 position bits");

// Merges the runs of kLen elements of buffer kSrc, and so on up to the tile's length tn; the
// result is in the buffer whose number it returns.
template <uint32_t kLen, int kSrc>
__device__ __forceinline__ int merge_runs(RunBuffers& s, uint32_t tn) {
    if constexpr (kLen >= kRunTile) {
        return kSrc;
    } else {
        if (kLen >= 64 && kLen >= tn) return kSrc;
        const uint32_t p0 = (threadIdx.x >> 5) * 64u + (threadIdx.x & 31u);
#pragma unroll
        for (uint32_t u = 0; u < 2; ++u) {
            const uint32_t p = p0 + u * 32u;
            const uint64_t k = s.k[kSrc][p];
            const bool later = (p & kLen) != 0;  // this run is the later one of its pair
            // keys <= k are keys < k + 1; the sentinel 2^64-1 follows every key
            uint32_t c = count_below<kLen>(&s.k[kSrc][(p ^ kLen) & ~(kLen - 1u)], later ? k + 1u : k);
            if (later && k == kMaxKey) c = kLen;
            const uint32_t dst = (p & ~kLen) + c;
            s.k[kSrc ^ 1][dst] = k;
            s.i[kSrc ^ 1][dst] = s.i[kSrc][p];
        }
        if (kLen < 32) __syncwarp();
        else __syncthreads();
        return merge_runs<2 * kLen, (kSrc ^ 1)>(s, tn);
    }
}

__global__ void __launch_bounds__(kRunThreads) k_tile_sort(const uint8_t* __restrict__ ops,
                                                           const uint64_t* __restrict__ keys, uint32_t n,
                                                           uint64_t* __restrict__ tk, uint32_t* __restrict__ tp,
                                                           BatchMeta* bm) {
    pdl_wait();
    pdl_trigger();
    __shared__ __align__(16) RunBuffers s;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t tbase = blockIdx.x * kRunTile;
    const uint32_t tn = min((uint32_t)kRunTile, n - tbase);
    uint64_t key[2];
    uint32_t id[2], bad = 0;
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u) {
        const uint32_t e = warp * 64u + u * 32u + lane;
        const bool in = e < tn;
        const uint32_t op = in ? ops[tbase + e] : 0u;
        const uint64_t k = in ? keys[tbase + e] : kMaxKey;
        const bool valid = op <= 2u && k != kMaxKey;
        key[u] = valid ? k : kMaxKey;
        id[u] = ((op & 3u) << 11) | e;
        bad += in && !valid ? 1u : 0u;
        s.k[1][e] = key[u];
    }
    __syncwarp();
    // runs of 8: rank = smaller keys, or equal keys of earlier positions
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u) {
        const uint32_t r0 = warp * 64u + u * 32u + (lane & 24u), o = lane & 7u;
        uint32_t rank = 0;
#pragma unroll
        for (uint32_t j = 0; j < 8; j += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&s.k[1][r0 + j]);
            rank += (v.x < key[u] || (v.x == key[u] && j < o)) ? 1u : 0u;
            rank += (v.y < key[u] || (v.y == key[u] && j + 1u < o)) ? 1u : 0u;
        }
        s.k[0][r0 + rank] = key[u];
        s.i[0][r0 + rank] = (uint16_t)id[u];
    }
    __syncwarp();
    const int src = merge_runs<8, 0>(s, tn);
    for (uint32_t p = threadIdx.x; p < tn; p += kRunThreads) {
        const uint32_t x = s.i[src][p];
        tk[tbase + p] = s.k[src][p];
        tp[tbase + p] = ((x >> 11) << 30) | (tbase + (x & 2047u));
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0 && bad) atomicAdd(&bm->invalid, bad);
}

}  // namespace

cudaError_t launch_tile_sort(const uint8_t* ops, const uint64_t* keys, uint32_t n, const SortBuffers& sb,
                             BatchMeta* bm, cudaStream_t s) {
    if (n == 0 || n > kSmallSort) return cudaErrorInvalidValue;
    launch_dep(k_tile_sort, (n + kRunTile - 1) / kRunTile, kRunThreads, 0, s, ops, keys, n, sb.in_k, sb.in_p, bm);
    ++g_launches;
    return cudaGetLastError();
}

namespace {

template <int kI>
cudaError_t launch_passes(uint32_t n, const SortBuffers& sb, BatchMeta* bm, uint32_t* err, cudaStream_t s,
                          int max_passes) {
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(k_sort_pass<kI>, cudaFuncAttributeMaxDynamicSharedMemorySize, pass_smem<kI>());
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const uint32_t tiles = (n + kPassThreads * kI - 1) / (kPassThreads * kI);
    for (uint32_t j = 0; j < (uint32_t)max_passes; ++j) {
        launch_dep(k_sort_pass<kI>, tiles, kPassThreads, pass_smem<kI>(), s, j, n, sb, bm, err);
        ++g_launches;
    }
    return cudaSuccess;
}

}  // namespace

static cudaError_t launch_count_passes(uint32_t n, const SortBuffers& sb, BatchMeta* bm, uint32_t* err, cudaStream_t s,
                                       int max_passes) {
    static bool attr_set = false;
    const int dyn = kTile * (int)(sizeof(uint64_t) + sizeof(uint32_t));
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(k_sort_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const uint32_t tiles = (n + kTile - 1) / kTile;
    for (uint32_t j = 0; j < (uint32_t)max_passes; ++j) {
        const uint32_t ctas = (tiles + kCountTiles - 1) / kCountTiles;
        if (j == 0) launch_dep(k_sort_count<true>, ctas, kThreads, 0, s, j, n, sb, bm, (uint32_t)max_passes);
        else launch_dep(k_sort_count<false>, ctas, kThreads, 0, s, j, n, sb, bm, (uint32_t)max_passes);
        ++g_launches;
        launch_dep(k_sort_scatter, tiles, kThreads, dyn, s, j, n, sb, bm, err);
        ++g_launches;
    }
    return cudaSuccess;
}

cudaError_t launch_sort(const uint8_t* ops, const uint64_t* keys, uint32_t n, const SortBuffers& buffers,
                        BatchMeta* bm, uint32_t* err, cudaStream_t s, int num_sms, int max_passes, bool* hist_clear,
                        bool long_too) {
    if (n == 0) return cudaSuccess;
    if (max_passes < 1 || max_passes > 8) return cudaErrorInvalidValue;
    SortBuffers sb = buffers;
    sb.ops = ops;
    sb.keys = keys;
    const bool sweep = n <= kSweepMost, large = n >= kLargeTiles;
    const int grid = min((int)((n + 255) / 256), num_sms * 8);
    const uint32_t nmarks = sb.grp_mark ? (n + kMarkGroup - 1) / kMarkGroup : 0u;
    cudaError_t e = cudaSuccess;
    if (sweep) {
        if (!*hist_clear && (e = cudaMemsetAsync(sb.hist, 0, kSortHist * sizeof(uint32_t), s)) != cudaSuccess) return e;
        *hist_clear = false;
        const uint32_t tile = (uint32_t)kPassThreads * (large ? 8u : 4u), words = (n + tile - 1) / tile * 256u;
        launch_dep(k_scan<true>, grid, 256, 0, s, ops, keys, n, sb.fixmap, sb.desc[0], words, sb.grp_mark, nmarks, sb.hist, bm);
        launch_dep(k_sort_plan, min((int)((n + 2047) / 2048), num_sms * 4), 256, 0, s, n, sb, bm, (uint32_t)max_passes);
        g_launches += 2;
        e = large ? launch_passes<8>(n, sb, bm, err, s, max_passes) : launch_passes<4>(n, sb, bm, err, s, max_passes);
    } else {
        const uint32_t ngroups = ((n + kTile - 1) / kTile + kScanGroup - 1) / kScanGroup;
        launch_dep(k_scan<false>, grid, 256, 0, s, ops, keys, n, sb.fixmap, sb.gctr, 8u * (ngroups + 1u), sb.grp_mark,
                   nmarks, (uint32_t*)nullptr, bm);
        ++g_launches;
        e = launch_count_passes(n, sb, bm, err, s, max_passes);
    }
    if (e != cudaSuccess) return e;
    if (max_passes < 8) {  // with eight passes every byte is sorted: nothing to fix
        const int fgrid = min((int)((n + 1023) / 1024), num_sms * 8);
        launch_dep(k_sort_find, fgrid, 256, 0, s, n, sb, bm, sweep);
        ++g_launches;
        if (sweep) *hist_clear = true;
        launch_dep(k_sort_fix, (n + kFixSlice - 1) / kFixSlice, kThreads, 0, s, n, sb, bm, long_too);
        ++g_launches;
    }
    return cudaGetLastError();
}

cudaError_t launch_sort_long(uint32_t n, const SortBuffers& sb, BatchMeta* bm, cudaStream_t s) {
    // the short segments are in order already: ordering them again changes nothing
    launch_dep(k_sort_fix, (n + kFixSlice - 1) / kFixSlice, kThreads, 0, s, n, sb, bm, true);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace pi
