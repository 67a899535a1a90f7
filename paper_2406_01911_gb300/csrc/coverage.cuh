// Coverage of a seed set on an RR pool (Sec. 2.2): the RR sets with at least one member in S, counted
// per stratum. Shared by the library's coverage calls and hyperim_coverage_noalloc.
//
// What bounds it is one pass over the members (200,000 sets of 30: 26 MB, 4 us at the measured copy rate).
// A flag byte per vertex costs far more than that: clearing n of them, and a 32-byte sector read per
// member. Up to kCoverSeeds seeds therefore sit in every block's shared memory instead: a filter of
// 2^15 bits that passes a stranger with probability below 1 in 16 and a sorted list that decides.
// A warp streams the members of several consecutive sets (they are contiguous), and only a member that
// is a seed looks up which set it lies in. COVER_FIGURES
#pragma once
#include <cstdint>

#include "../../include/hyperim.h"
#include "mat.cuh"

namespace hyperim {

constexpr int kCoverThreads = 256;
constexpr int kCoverSeeds = 2048;         // seeds held on chip (power of two)
constexpr int kCoverFilterBits = 15;

struct CoverShared {
    uint32_t filter[1 << (kCoverFilterBits - 5)];
    uint32_t seeds[kCoverSeeds];
    unsigned int lam[HYPERIM_NSTRATA];
};

__device__ __forceinline__ uint32_t cover_hash(uint32_t v) { return (v * 0x9E3779B1u) >> (32 - kCoverFilterBits); }

// Whole block. seeds[0, k), k <= kCoverSeeds; ids outside [0, n) match nothing. skip(r): the set takes
// no part. per: consecutive sets per warp and step (1..32). Adds to lam[0..15].
template <typename Skip>
__device__ __forceinline__ void cover_sets(CoverShared& S, const int64_t* __restrict__ rr_off,
                                           const int32_t* __restrict__ mem, const uint8_t* __restrict__ rr_stratum,
                                           int64_t count, int32_t n, const int32_t* __restrict__ seeds, int32_t k,
                                           int per, unsigned long long* __restrict__ lam, Skip&& skip) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (1 << (kCoverFilterBits - 5)); i += kCoverThreads) S.filter[i] = 0;
    if (threadIdx.x < HYPERIM_NSTRATA) S.lam[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < k; i += kCoverThreads) S.seeds[i] = (uint32_t)seeds[i];
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += kCoverThreads) {
        const uint32_t h = cover_hash(S.seeds[i]);
        atomicOr(&S.filter[h >> 5], 1u << (h & 31));
    }
    group_sort<kCoverThreads>(S.seeds, k);  // synchronises
    __syncthreads();
    const int64_t warp = (blockIdx.x * (int64_t)kCoverThreads + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * kCoverThreads) >> 5;
    for (int64_t r0 = warp * per; r0 < count; r0 += nwarps * per) {
        const int sets = (int)min((int64_t)per, count - r0);
        // lane i: the end of set r0 + i
        const int64_t end = lane < sets ? rr_off[r0 + lane + 1] : INT64_MAX;
        const int64_t first = rr_off[r0], last = __shfl_sync(0xFFFFFFFFu, end, sets - 1);
        uint32_t hit = 0;  // bit i: set r0 + i holds a seed
        const uint32_t all = sets == 32 ? 0xFFFFFFFFu : (1u << sets) - 1u;
        constexpr int U = 4;
        for (int64_t base = first; base < last; base += 32 * U) {
            uint32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t x = base + u * 32 + lane;
                v[u] = x < last ? (uint32_t)mem[x] : 0xFFFFFFFFu;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t h = cover_hash(v[u]);
                bool f = v[u] < (uint32_t)n && (S.filter[h >> 5] >> (h & 31) & 1u);
                if (f) {
                    int lo = 0, hi = k;  // least seed >= v
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (S.seeds[mid] < v[u]) lo = mid + 1; else hi = mid;
                    }
                    f = lo < k && S.seeds[lo] == v[u];
                }
                for (uint32_t b = __ballot_sync(0xFFFFFFFFu, f); b; b &= b - 1) {
                    // the set of that member: the number of ends at or below its place
                    const int64_t x = base + u * 32 + (__ffs(b) - 1);
                    hit |= 1u << __popc(__ballot_sync(0xFFFFFFFFu, end <= x));
                }
            }
            if (hit == all) break;
        }
        if (lane < sets && (hit >> lane & 1u) && !skip(r0 + lane))
            atomicAdd(&S.lam[rr_stratum[r0 + lane] & (HYPERIM_NSTRATA - 1)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < HYPERIM_NSTRATA && S.lam[threadIdx.x])
        atomicAdd(&lam[threadIdx.x], (unsigned long long)S.lam[threadIdx.x]);
}

// sets per warp and step: a few steps for every resident warp, so that a pool of few large sets still
// spreads over the chip
inline int cover_per(int64_t count, int sm) {
    const int64_t per = count / ((int64_t)sm * 64);
    return (int)(per < 1 ? 1 : per > 32 ? 32 : per);
}

}  // namespace hyperim
