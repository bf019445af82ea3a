// Searches of the index and storage layers that one thread does for one key.
#pragma once

#include "common.cuh"

namespace pi {

// Largest p in [slo - 1, shi) with K[p] <= q, for a storage gap with K[shi] > q and,
// when slo > 0 or has_lo, K[slo] <= q; -1 when q is below every key. The gap's keys
// lie between klo = K[slo] and khi = K[shi], so the answer is looked for first in the
// 64-byte line of 8 keys around the linear estimate slo + (q - klo) / (khi - klo) *
// (shi - slo): for keys spread evenly over the gap that line usually holds it. From
// there the search moves line by line towards the answer, so it stays exact for any
// key distribution.
__device__ __forceinline__ int32_t gap_search(const uint64_t* K, uint32_t slo, uint32_t shi, uint64_t klo,
                                              uint64_t khi, uint64_t q, uint32_t lim, uint64_t& k_out, uint32_t* err) {
    uint32_t est = slo;
    if (shi > slo + 1u && khi != kMaxKey && khi > klo) {
        const float f = __ull2float_rz(q - klo) / __ull2float_rn(khi - klo);  // in [0, 1]
        est = slo + (uint32_t)(f * (float)(shi - slo));
        if (est >= shi) est = shi - 1u;
    }
    uint32_t c = est & ~7u;
    int dir = 0;
    const uint32_t max_lines = (shi - slo) / 8u + 3u;
    for (uint32_t it = 0;; ++it) {
        if (c > lim || it > max_lines) {
            atomicOr(err, kErrBounds);
            return -1;
        }
        const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(K + c);
        uint64_t kk[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const ulonglong2 v = kp[j];
            kk[2 * j] = v.x;
            kk[2 * j + 1] = v.y;
        }
        uint32_t gt = 0;  // bit j: K[c + j] > q (a suffix of the line, the keys being sorted)
#pragma unroll
        for (int j = 0; j < 8; ++j) gt |= (kk[j] > q ? 1u : 0u) << j;
        if (gt == 0xFFu) {  // the answer is before this line
            if (dir > 0) return (int32_t)c - 1;  // (k_out was set on the previous line)
            if (c == 0) return -1;
            dir = -1;
            c -= 8u;
        } else if (gt == 0u) {  // the answer is at the end of this line or after it
            k_out = kk[7];
            if (dir < 0) return (int32_t)c + 7;
            dir = 1;
            c += 8u;
        } else {
            const int f = __ffs(gt) - 1;  // >= 1
#pragma unroll
            for (int j = 1; j < 8; ++j)
                if (j == f) k_out = kk[j - 1];
            return (int32_t)c + f - 1;
        }
    }
}

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
