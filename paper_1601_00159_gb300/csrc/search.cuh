// Searches of the index and storage layers that one thread does for one key.
#pragma once

#include "common.cuh"

namespace pi {

// Keys <= q in the sorted K[0, n): each round reads seven evenly spaced entries at once, so
// that n entries take about log8(n) dependent reads.
__device__ __forceinline__ uint32_t count_le(const uint64_t* K, uint32_t n, uint64_t q) {
    uint32_t lo = 0, len = n;  // the count lies in [lo, lo + len]
    while (len >= 8u) {
        uint64_t v[7];
#pragma unroll
        for (uint32_t j = 0; j < 7; ++j) v[j] = K[lo + (uint32_t)(((uint64_t)len * (j + 1u)) >> 3)];
        uint32_t c = 0;  // pivots <= q: a prefix
#pragma unroll
        for (uint32_t j = 0; j < 7; ++j) c += v[j] <= q ? 1u : 0u;
        const uint32_t nlo = c ? (uint32_t)(((uint64_t)len * c) >> 3) + 1u : 0u;
        const uint32_t nhi = c < 7u ? (uint32_t)(((uint64_t)len * (c + 1u)) >> 3) : len;
        lo += nlo;
        len = nhi - nlo;
    }
    uint64_t v[7];
#pragma unroll
    for (uint32_t j = 0; j < 7; ++j) v[j] = j < len ? K[lo + j] : kMaxKey;
    uint32_t c = 0;
#pragma unroll
    for (uint32_t j = 0; j < 7; ++j) c += j < len && v[j] <= q ? 1u : 0u;
    return lo + c;
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// First node of the 64-byte line in which a storage gap's answer is looked for first (see
// gap_search); slo's line when there is nothing to interpolate with.
__device__ __forceinline__ uint32_t gap_line(uint32_t slo, uint32_t shi, uint64_t klo, uint64_t khi, uint64_t q) {
    uint32_t est = slo;
    if (khi != kMaxKey && khi > klo && shi > slo + 8u) {
        const float f = __ull2float_rz(q - klo) / __ull2float_rn(khi - klo);  // in [0, 1]
        est = slo + (uint32_t)(f * (float)(shi - slo));
        if (est >= shi) est = shi - 1u;
    }
    return est & ~7u;
}

// Largest p in [slo - 1, shi) with K[p] <= q, for a storage gap with K[shi] > q and,
// when slo > 0 or q is at least K[0], K[slo] <= q; -1 when q is below every key. The gap's keys
// lie between klo = K[slo] and khi = K[shi], so the answer is looked for first in the
// 64-byte line of 8 keys around the linear estimate slo + (q - klo) / (khi - klo) *
// (shi - slo), then line by line towards it: for keys spread evenly over the gap one of the
// first lines holds it. After four the rest of the gap is searched seven entries a round, so
// the search is exact and short for any distribution (the gap past the level's last key has no
// upper key to interpolate with; walking its lines made a batch of appended keys wait 30 reads).
__device__ __forceinline__ int32_t gap_search(const uint64_t* K, uint32_t slo, uint32_t shi, uint64_t klo,
                                              uint64_t khi, uint64_t q, uint32_t lim, uint64_t& k_out, uint32_t* err) {
    if (shi > lim || slo > shi) {
        atomicOr(err, kErrBounds);
        return -1;
    }
    uint32_t lo = slo, hi = shi;  // the answer plus one lies in [lo, hi]
    if (khi != kMaxKey && khi > klo && shi > slo + 8u) {
        uint32_t c = gap_line(slo, shi, klo, khi, q);
#pragma unroll 1
        for (int it = 0; it < 4; ++it) {
            uint64_t k0[4], k1[4];
            ld_256(K + c, k0);
            ld_256(K + c + 4u, k1);
            const uint64_t kk[8] = {k0[0], k0[1], k0[2], k0[3], k1[0], k1[1], k1[2], k1[3]};
            uint32_t gt = 0;  // bit j: K[c + j] > q; past the array's sentinel any key may follow
#pragma unroll
            for (int j = 0; j < 8; ++j) gt |= (kk[j] > q ? 1u : 0u) << j;
            const uint32_t le = gt ? (uint32_t)(__ffs((int)gt) - 1) : 8u;  // keys <= q in the line
            if (le > 0u && le < 8u) {
#pragma unroll
                for (int j = 0; j < 7; ++j)
                    if ((uint32_t)j + 1u == le) k_out = kk[j];
                return (int32_t)(c + le) - 1;
            }
            if (le == 0u) {  // the answer is before this line
                hi = c < hi ? c : hi;
                if (c <= lo) break;
                c -= 8u;
            } else {  // at its end or after it
                lo = c + 8u > lo ? c + 8u : lo;
                k_out = kk[7];
                if (c + 8u >= hi) break;
                c += 8u;
            }
            if (lo >= hi) break;
        }
    }
    if (lo < hi) lo += count_le(K + lo, hi - lo, q);
    if (lo > 0u) k_out = K[lo - 1u];
    return (int32_t)lo - 1;
}

// The storage node with the largest key <= q (-1: none) and its key: the lowest built level
// holds every key of the levels above it, so it is searched as one sorted array, which gives
// the storage gap of q. Without a built level the storage layer is searched itself.
__device__ __forceinline__ int32_t storage_search(const DevMeta* m, const uint64_t* SK, const uint64_t* lkeys,
                                                  const uint32_t* ldown, const uint64_t* lkeys1, const uint32_t* ldown1,
                                                  uint64_t q, uint64_t& key, uint32_t* err) {
    const uint32_t size = m->size, H = m->H, Lb = m->Lb;
    if (Lb > H) {
        const uint32_t c = count_le(SK, size, q);
        key = c ? SK[c - 1u] : 0ull;
        return (int32_t)c - 1;
    }
    const uint32_t base = m->base[Lb], lcur = m->lcur;
    const uint64_t* K = (lcur ? lkeys1 : lkeys) + base;
    const uint32_t* D = (lcur ? ldown1 : ldown) + base;
    const uint32_t c = count_le(K, m->n[Lb], q);  // the level's sentinel follows its entries
    const uint64_t kn = K[c], klo = c ? K[c - 1u] : 0ull;
    const uint32_t dn = D[c], lo = c ? D[c - 1u] : 0u;
    return gap_search(SK, lo, dn, klo, kn, q, size, key, err);
}

}  // namespace pi
