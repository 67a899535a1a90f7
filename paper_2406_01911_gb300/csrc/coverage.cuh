// Coverage of a seed set on an RR pool (Sec. 2.2): the RR sets with at least one member in S, counted
// per stratum. Shared by the library's coverage calls and hyperim_coverage_noalloc.
//
// What bounds it is one pass over the members (200,000 sets of 30: 26 MB, 4 us at the measured copy rate).
// A flag byte per vertex costs far more than that: clearing n of them, and a 32-byte sector read per
// member. Up to kCoverSeeds seeds therefore sit in every block's shared memory instead: a bit per hash value,
// which decides nearly every member by one read that waits for no other, and an open-addressing table at most
// half full for the rest. (With the table alone a warp waited for its longest probe chain: 20,000 sets of 60
// members on 4M vertices, 100 seeds, 94 us, with flags 71, now 27.)
// A warp streams the members of several consecutive sets (they are contiguous), and only a member that
// is a seed looks up which set it lies in; the rest of that set is passed over (large sets hold many
// seeds: without that the warps of the largest sets ran 15 times as long as the others).
// 200,000 sets of 30 members, 100 seeds: 48 us with flags, 36 with the table alone, 21 so.
#pragma once
#include <cstdint>

#include "../../include/hyperim.h"
#include "mat.cuh"

namespace hyperim {

constexpr int kCoverThreads = 512;
constexpr int kCoverSeeds = 2048;         // seeds held on chip

// log2 of the table's slots: at least twice the seeds
__host__ __device__ inline int cover_bits(int32_t k) {
    int b = 7;
    while ((1 << b) < 2 * k) ++b;
    return b;
}
// a bit per value of the hash's top kCoverFilter bits: a member whose bit is clear is no seed
constexpr int kCoverFilter = 16;
constexpr int kCoverFilterWords = 1 << (kCoverFilter - 5);
inline size_t cover_smem(int32_t k) { return (sizeof(uint32_t) << cover_bits(k)) + sizeof(uint32_t) * kCoverFilterWords; }

// Whole block; slot: cover_smem(k) bytes of shared memory (a seed or kSentinel each, then the hash bits).
// seeds[0, k), k <= kCoverSeeds; ids outside [0, n) match nothing. skip(r): the set takes no part. per: consecutive sets per warp and step (1..32). Adds to lam[0..15].
template <typename Skip>
__device__ __forceinline__ void cover_sets(uint32_t* slot, const int64_t* __restrict__ rr_off,
                                           const int32_t* __restrict__ mem, const uint8_t* __restrict__ rr_stratum,
                                           int64_t count, int32_t n, const int32_t* __restrict__ seeds, int32_t k,
                                           int per, unsigned long long* __restrict__ lam, Skip&& skip) {
    const int lane = threadIdx.x & 31;
    __shared__ unsigned int s_lam[HYPERIM_NSTRATA];
    const int bits = cover_bits(k);
    const uint32_t mask = (1u << bits) - 1;
    uint32_t* filter = slot + mask + 1;
    for (int i = threadIdx.x; i <= (int)mask; i += kCoverThreads) slot[i] = kSentinel;
    for (int i = threadIdx.x; i < kCoverFilterWords; i += kCoverThreads) filter[i] = 0;
    if (threadIdx.x < HYPERIM_NSTRATA) s_lam[threadIdx.x] = 0;
    __syncthreads();
    uint32_t mine[kCoverSeeds / kCoverThreads];  // this thread's seeds, all read before the first is entered
#pragma unroll
    for (int u = 0; u < kCoverSeeds / kCoverThreads; ++u) {
        const int i = u * kCoverThreads + threadIdx.x;
        mine[u] = i < k ? (uint32_t)seeds[i] : kSentinel;
    }
#pragma unroll
    for (int u = 0; u < kCoverSeeds / kCoverThreads; ++u) {
        const uint32_t v = mine[u];
        if (v >= (uint32_t)n) continue;
        const uint32_t hv = v * 0x9E3779B1u;
        atomicOr(&filter[hv >> (37 - kCoverFilter)], 1u << (hv >> (32 - kCoverFilter) & 31));
        for (uint32_t h = hv >> (32 - bits);; h = (h + 1) & mask) {  // half the slots stay empty
            const uint32_t old = atomicCAS(&slot[h], kSentinel, v);
            if (old == kSentinel || old == v) break;
        }
    }
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
        for (int64_t base = first; base < last;) {
            // a set that has its seed already is left at once
            const int at = __popc(__ballot_sync(0xFFFFFFFFu, end <= base));
            if (hit >> at & 1u) {
                base = __shfl_sync(0xFFFFFFFFu, end, at);
                continue;
            }
            uint32_t v[U], word[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t x = base + u * 32 + lane;
                v[u] = x < last ? (uint32_t)mem[x] : 0xFFFFFFFFu;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) word[u] = filter[v[u] * 0x9E3779B1u >> (37 - kCoverFilter)];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                bool f = false;
                const uint32_t hv = v[u] * 0x9E3779B1u;
                if ((word[u] >> (hv >> (32 - kCoverFilter) & 31) & 1u) && v[u] < (uint32_t)n) {
                    uint32_t h = hv >> (32 - bits), x = slot[h];
                    while (x != kSentinel && x != v[u]) {
                        h = (h + 1) & mask;
                        x = slot[h];
                    }
                    f = x == v[u];
                }
                uint32_t b = __ballot_sync(0xFFFFFFFFu, f);
                while (b) {
                    // the set of that member: the number of ends at or below its place
                    const int64_t x0 = base + u * 32;
                    const int i = __popc(__ballot_sync(0xFFFFFFFFu, end <= x0 + (__ffs(b) - 1)));
                    hit |= 1u << i;
                    const int64_t rest = __shfl_sync(0xFFFFFFFFu, end, i) - x0;  // the set's last place here
                    b = rest >= 32 ? 0u : b & ~((1u << rest) - 1u);
                }
            }
            base += 32 * U;
            if (hit == all) break;
        }
        if (lane < sets && (hit >> lane & 1u) && !skip(r0 + lane))
            atomicAdd(&s_lam[rr_stratum[r0 + lane] & (HYPERIM_NSTRATA - 1)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < HYPERIM_NSTRATA && s_lam[threadIdx.x])
        atomicAdd(&lam[threadIdx.x], (unsigned long long)s_lam[threadIdx.x]);
}

// sets per warp and step: a few steps for every resident warp, so that a pool of few large sets still
// spreads over the chip
inline int cover_per(int64_t count, int sm) {
    const int64_t per = (count + (int64_t)sm * 64 - 1) / ((int64_t)sm * 64);
    return (int)(per < 1 ? 1 : per > 32 ? 32 : per);
}

// blocks: a warp for every `per` sets, up to four blocks per SM, two where there are many seeds: every block
// enters them all, one atomic after another (200,000 sets of 2 members, 2,000 seeds: 29 us with eight blocks of 256
// threads per SM, with flags 27, now 16; 600 seeds and sets of 60: 31 us with two blocks, 42 with one)
inline int cover_blocks(int64_t count, int per, int32_t k, int sm) {
    const int64_t warps = (count + per - 1) / per;
    const int64_t want = (warps * 32 + kCoverThreads - 1) / kCoverThreads, most = (int64_t)sm * (k <= 512 ? 4 : 2);
    return (int)(want < most ? want : most);
}

}  // namespace hyperim
