// Greedy max coverage over an RR pool (Algorithm 1; marginal coverage of Eq. 2) on the device.
//
// Scores are integers: an RR set of stratum s weighs W_s = floor(|V_s| 2^32 / n_s) (1 with plain
// roots), so sums do not depend on the order of the atomic updates. Each round: argmax over the
// vertices not picked yet (ties to the lowest id), then the RR sets containing the winner that
// are not covered yet are retired: marked covered, counted in Lambda_s, and their weight is
// subtracted from the score of every member. The k rounds run inside one launch (k_greedy), whose
// blocks meet at a barrier between them.
#include <algorithm>
#include <cstddef>
#include <new>
#include <string>
#include <vector>

#include "coverage.cuh"
#include "internal.h"

namespace hyperim {
namespace {

constexpr int kArgThreads = 256;

struct Weights {
    unsigned long long w[HYPERIM_NSTRATA];
};

// A prefix view of a pool: only the RR sets (stratum s, index j) with j < lim[s] take part (the
// sets a pool grown to a smaller theta would hold). on = 0: every set of the pool.
struct Limits {
    uint32_t lim[HYPERIM_NSTRATA];
    int on;
    __device__ __forceinline__ bool skip(const uint8_t* rr_stratum, const uint32_t* rr_j, int64_t r) const {
        return on && rr_j[r] >= lim[rr_stratum[r]];
    }
};

// occurrences of each vertex over the RR sets of a prefix view; one warp per RR set
__global__ void k_count_occ_view(const int64_t* __restrict__ rr_off, const int32_t* __restrict__ mem,
                                 const uint8_t* __restrict__ rr_stratum, const uint32_t* __restrict__ rr_j,
                                 int64_t N, Limits L, uint32_t* __restrict__ cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = warp; r < N; r += nwarps) {
        if (L.skip(rr_stratum, rr_j, r)) continue;
        for (int64_t x = rr_off[r] + lane; x < rr_off[r + 1]; x += 32) atomicAdd(&cnt[mem[x]], 1u);
    }
}

__global__ void k_count_occ(const int32_t* __restrict__ mem, int64_t total, uint32_t* __restrict__ cnt) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[mem[x]], 1u);
}

// inverted index (vertex -> RR ids) and initial weighted scores; one warp per RR set
__global__ void k_scatter_inv(const int64_t* __restrict__ rr_off, const int32_t* __restrict__ mem,
                              const uint8_t* __restrict__ rr_stratum, const uint32_t* __restrict__ rr_j,
                              int64_t N, Limits L, const int64_t* __restrict__ inv_off,
                              uint32_t* __restrict__ cur, uint32_t* __restrict__ inv,
                              unsigned long long* __restrict__ score, Weights W) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = warp; r < N; r += nwarps) {
        if (L.skip(rr_stratum, rr_j, r)) continue;
        const int64_t b = rr_off[r], e = rr_off[r + 1];
        const unsigned long long w = W.w[rr_stratum[r]];
        for (int64_t x = b + lane; x < e; x += 32) {
            const int32_t v = mem[x];
            const uint32_t pos = atomicAdd(&cur[v], 1u);
            inv[inv_off[v] + pos] = (uint32_t)r;
            atomicAdd(&score[v], w);
        }
    }
}

__device__ __forceinline__ bool better(unsigned long long s1, uint32_t i1, unsigned long long s2,
                                       uint32_t i2) {
    return s1 > s2 || (s1 == s2 && i1 < i2);
}

// The best (score, id) among the unpicked vertices of [0, n) visited by one thread (first index
// t, stride T): four consecutive vertices per step, their flags and scores loaded together
// without depending on one another (vectorised: score and picked are 16- and 4-byte aligned).
// `load` reads a score (plain, or through L2 where other threads of the block change scores by
// atomics).
template <bool kL2Scores = false>
__device__ __forceinline__ void scan_unpicked(const unsigned long long* __restrict__ score,
                                              const uint8_t* __restrict__ picked, int64_t n, int64_t t, int64_t T,
                                              unsigned long long& bs, uint32_t& bi) {
    const int64_t n4 = n >> 2;
    for (int64_t q = t; q < n4; q += T) {
        const uchar4 pk = reinterpret_cast<const uchar4*>(picked)[q];
        ulonglong2 a, b;
        if (kL2Scores) {
            a = __ldcg(reinterpret_cast<const ulonglong2*>(score) + 2 * q);
            b = __ldcg(reinterpret_cast<const ulonglong2*>(score) + 2 * q + 1);
        } else {
            a = reinterpret_cast<const ulonglong2*>(score)[2 * q];
            b = reinterpret_cast<const ulonglong2*>(score)[2 * q + 1];
        }
        const uint32_t v = (uint32_t)(4 * q);
        if (!pk.x && better(a.x, v, bs, bi)) { bs = a.x; bi = v; }
        if (!pk.y && better(a.y, v + 1, bs, bi)) { bs = a.y; bi = v + 1; }
        if (!pk.z && better(b.x, v + 2, bs, bi)) { bs = b.x; bi = v + 2; }
        if (!pk.w && better(b.y, v + 3, bs, bi)) { bs = b.y; bi = v + 3; }
    }
    for (int64_t v = 4 * n4 + t; v < n; v += T) {
        if (picked[v]) continue;
        const unsigned long long sc = kL2Scores ? __ldcg(score + v) : score[v];
        if (better(sc, (uint32_t)v, bs, bi)) { bs = sc; bi = (uint32_t)v; }
    }
}

// argmax of score over unpicked vertices, lowest id on ties (the stepwise greedy, over a score vector
// of the caller's); the last block to finish reduces the per-block winners and marks the seed picked.
__global__ void __launch_bounds__(kArgThreads)
k_argmax(const unsigned long long* __restrict__ score, uint8_t* __restrict__ picked, int32_t n,
         unsigned long long* __restrict__ bscore, uint32_t* __restrict__ bid,
         unsigned int* __restrict__ ticket, int32_t* __restrict__ best) {
    __shared__ unsigned long long ss[kArgThreads / 32];
    __shared__ uint32_t si[kArgThreads / 32];
    __shared__ bool last;
    unsigned long long bs = 0;
    uint32_t bi = 0xFFFFFFFFu;
    scan_unpicked(score, picked, n, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                  (int64_t)gridDim.x * blockDim.x, bs, bi);
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
        const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { ss[wid] = bs; si[wid] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kArgThreads / 32; ++w)
            if (better(ss[w], si[w], bs, bi)) { bs = ss[w]; bi = si[w]; }
        bscore[blockIdx.x] = bs;
        bid[blockIdx.x] = bi;
        __threadfence();
        const unsigned int t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    bs = 0;
    bi = 0xFFFFFFFFu;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        const unsigned long long s = ((volatile unsigned long long*)bscore)[b];
        const uint32_t i = ((volatile uint32_t*)bid)[b];
        if (better(s, i, bs, bi)) { bs = s; bi = i; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
        const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
    }
    if (lane == 0) { ss[wid] = bs; si[wid] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kArgThreads / 32; ++w)
            if (better(ss[w], si[w], bs, bi)) { bs = ss[w]; bi = si[w]; }
        *best = (int32_t)bi;
        picked[bi] = 1;
        *ticket = 0;
    }
}

// retire the uncovered RR sets containing the round's winner; one warp per inverted entry
__global__ void k_retire(const int32_t* __restrict__ best, const int64_t* __restrict__ inv_off,
                         const uint32_t* __restrict__ inv, const int64_t* __restrict__ rr_off,
                         const int32_t* __restrict__ mem, const uint8_t* __restrict__ rr_stratum,
                         uint32_t* __restrict__ covered, unsigned long long* __restrict__ score,
                         unsigned long long* __restrict__ lam, Weights W) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int32_t v = *best;
    const int64_t b = inv_off[v], e = inv_off[v + 1];
    for (int64_t t = b + warp; t < e; t += nwarps) {
        const uint32_t r = inv[t];
        uint32_t old = 0;
        if (lane == 0) old = atomicExch(&covered[r], 1u);
        old = __shfl_sync(0xFFFFFFFFu, old, 0);
        if (old) continue;
        const int s = rr_stratum[r];
        const unsigned long long neg = 0ull - W.w[s];
        if (lane == 0) atomicAdd(&lam[s], 1ull);
        for (int64_t x = rr_off[r] + lane; x < rr_off[r + 1]; x += 32) atomicAdd(&score[mem[x]], neg);
    }
}

// ---- the k rounds in one launch -----------------------------------------------------------------
// What a round costs is not its arithmetic: with one launch for the argmax and one for the
// retirement, 2M vertices and 100 to 200 rounds, a round took 19 us for 1 us of score reads. So
//   - only vertices that some RR set of the view holds take part ("active": a tenth to a third of
//     2M), numbered 0..na-1, their scores side by side, the RR sets' members renumbered to match:
//     the argmax reads 8 bytes per active vertex;
//   - a picked vertex needs no flag, its score is 0 once its sets are retired; when the best score is
//     0 the rest of the seeds are the lowest ids not picked yet;
//   - all rounds run in one launch with two barriers a round; block winners are reduced by every block
//     for itself, so the winner needs no third one. Up to kGClusterMembers members in the pool the launch
//     is one cluster of kGCluster blocks: its barrier is the hardware's and the block winners go straight
//     into the other blocks' shared memory. Larger pools (a round may retire tens of millions of
//     members) take a block for every 16K members, resident together by the contract of a cooperative
//     launch, with a barrier in global memory whose wait is bounded (kErrSpin); the smallest pools one block
//     and no barrier at all;
//   - in a cluster the argmax looks at candidates only: the vertices whose score is at least that of the
//     kCand-th largest, found once by the radix select below, one per thread, which keeps its vertex and
//     its index range in registers: what is left of an argmax is one read of a score. Scores only
//     decrease, so while the best candidate still reaches that threshold it is the best of all (every
//     vertex at the threshold is a candidate, so ties are settled among them); when it does not, one
//     round looks at every active vertex and the candidates are chosen anew. Where more share the threshold
//     than fit, or fewer have a score, there are none, and the select (five passes) is tried again a round later,
//     then 2, 4, 8 .. rounds later. (A grid of 152 blocks loses more in the select's histograms than it gains:
//     106 -> 112 ms on the 100k query.)
// 100 seeds from sets of 1.2 members on 2M vertices, nearly all scores alike: 40,000 and 400,000 sets took 3.9 and
// 11.5 ms with a select every round and the id read after the score, 0.9 and 2.0 ms so (1.8 and 1.9 with two
// launches a round).
// 200 seeds chosen on the pools of 40,000 sets of that graph, with the estimate: 4.9 ms with two launches a
// round, 4.0 ms with a cooperative launch over 152 blocks and no candidates, 3.3 ms so (k_greedy itself 2.7
// and 2.2 ms: a round is still a chain of six or seven dependent L2 reads); the index build 0.42 -> 0.14 ms
// with long sets spread over blocks. The Eq. upper_2 bound took 17 launches a round (35 ms of a 100 ms
// query), now none of its own. Above 4M members a cluster's 16 SMs lose: a pool of 8M (608 sets of a third
// of 100k vertices) retires nearly all of them in its first round.
constexpr int kGThreads = 512;
constexpr int kGWarps = kGThreads / 32;
constexpr int64_t kGMembersPerBlock = 1 << 14;
constexpr int kGCluster = 16;
constexpr int64_t kGClusterMembers = 1 << 22;
constexpr int64_t kGClusterScan = 1 << 19;
constexpr unsigned int kCand = 4096, kCandCap = kGCluster * kGThreads;  // at most one per thread
constexpr int kTopBits = 11;
constexpr int kTopBins = 1 << kTopBits;

// active vertices: act[c] = v, cidx[v] = c (any order), score[c] = 0; the counts are cleared for
// the scatter. nact: one word, zeroed by the caller.
constexpr int kActThreads = 256, kActItems = 8;
__global__ void __launch_bounds__(kActThreads)
k_active(uint32_t* __restrict__ cnt, int32_t n, int32_t* __restrict__ act, uint32_t* __restrict__ cidx,
         unsigned long long* __restrict__ score, unsigned int* __restrict__ nact) {
    __shared__ int wsum[kActThreads / 32];
    __shared__ unsigned int base_s;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t v0 = (int64_t)blockIdx.x * (kActThreads * kActItems);
    uint32_t flags = 0;
    int mine[kActItems];
    int run = 0;  // active vertices of this warp so far
#pragma unroll
    for (int i = 0; i < kActItems; ++i) {
        const int64_t v = v0 + (wid * kActItems + i) * 32 + lane;
        const bool f = v < n && cnt[v] != 0;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, f);
        mine[i] = run + __popc(b & ((1u << lane) - 1u));
        run += __popc(b);
        if (f) {
            flags |= 1u << i;
            cnt[v] = 0;
        }
    }
    if (lane == 0) wsum[wid] = run;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kActThreads / 32; ++w) {
            const int c = wsum[w];
            wsum[w] = t;
            t += c;
        }
        base_s = t ? atomicAdd(nact, (unsigned int)t) : 0u;
    }
    __syncthreads();
    const uint32_t base = base_s + (uint32_t)wsum[wid];
#pragma unroll
    for (int i = 0; i < kActItems; ++i) {
        if (!(flags >> i & 1u)) continue;
        const int32_t v = (int32_t)(v0 + (wid * kActItems + i) * 32 + lane);
        const uint32_t c = base + (uint32_t)mine[i];
        act[c] = v;
        cidx[v] = c;
        score[c] = 0;
    }
}

// RR sets taken by blocks: a batch of kSetsPerWarp sets per warp; a warp does a set of up to kLongSet
// members alone, longer ones are left to the whole block after its warps are done. (Sets are tiny at the
// median and 10,000 members at the end of their tail: with one warp per set whatever its size, the longest
// set's 400 dependent steps were what a launch or a round waited for.)
// find(i, x0, x1, tag): whether item i takes part, its member range and a tag; body(x, tag).
constexpr int kLongSet = 256;
constexpr int kSetsPerWarp = 2;
struct LongSets {
    int64_t x0[kGWarps * kSetsPerWarp], x1[kGWarps * kSetsPerWarp];
    unsigned long long tag[kGWarps * kSetsPerWarp];
    int count;
};
template <typename Find, typename Body>
__device__ __forceinline__ void block_sets(LongSets& S, int64_t items, Find&& find, Body&& body) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // consecutive items go to different blocks: few long ones still spread over the grid
    const int64_t batch = (int64_t)gridDim.x * kGWarps * kSetsPerWarp;
    for (int64_t i0 = blockIdx.x; i0 < items; i0 += batch) {
        if (threadIdx.x == 0) S.count = 0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kSetsPerWarp; ++q) {
            const int64_t i = i0 + (int64_t)(q * kGWarps + wid) * gridDim.x;
            int64_t x0 = 0, x1 = 0;
            unsigned long long tag = 0;
            if (i >= items || !find(i, x0, x1, tag)) continue;
            if (x1 - x0 <= kLongSet) {
                for (int64_t x = x0 + lane; x < x1; x += 32) body(x, tag);
            } else if (lane == 0) {
                const int at = atomicAdd(&S.count, 1);
                S.x0[at] = x0;
                S.x1[at] = x1;
                S.tag[at] = tag;
            }
        }
        __syncthreads();
        const int todo = S.count;
        for (int q = 0; q < todo; ++q) {
            const int64_t x1 = S.x1[q];
            const unsigned long long tag = S.tag[q];
#pragma unroll 4
            for (int64_t x = S.x0[q] + threadIdx.x; x < x1; x += kGThreads) body(x, tag);
        }
        __syncthreads();
    }
}

// inverted index (vertex -> RR ids), the members' numbers and the initial scores (cidx null: a vertex's
// number is its id)
__global__ void __launch_bounds__(kGThreads)
k_scatter_active(const int64_t* __restrict__ rr_off, const int32_t* __restrict__ mem,
                 const uint8_t* __restrict__ rr_stratum, const uint32_t* __restrict__ rr_j,
                 int64_t N, Limits L, const int64_t* __restrict__ inv_off,
                 uint32_t* __restrict__ cur, uint32_t* __restrict__ inv,
                 const uint32_t* __restrict__ cidx, uint32_t* __restrict__ memc,
                 unsigned long long* __restrict__ score, Weights W) {
    __shared__ LongSets S;
    block_sets(
        S, N,
        [&](int64_t r, int64_t& x0, int64_t& x1, unsigned long long& tag) {
            if (L.skip(rr_stratum, rr_j, r)) return false;
            x0 = rr_off[r];
            x1 = rr_off[r + 1];
            tag = (unsigned long long)r << 4 | (unsigned long long)rr_stratum[r];
            return true;
        },
        [&](int64_t x, unsigned long long tag) {
            const int32_t v = mem[x];
            const uint32_t c = cidx ? cidx[v] : (uint32_t)v;
            inv[inv_off[v] + atomicAdd(&cur[v], 1u)] = (uint32_t)(tag >> 4);
            if (cidx) memc[x] = c;
            atomicAdd(&score[c], W.w[tag & 15]);
        });
}

struct GreedyOut {
    unsigned long long lam[HYPERIM_NSTRATA];
    unsigned long long best_lo, best_hi;  // Eq. upper_2: the least bound (prefix mode)
};

struct GreedyParams {
    const int32_t* act;          // by number (null: every vertex takes part, its number is its id)
    unsigned long long* score;   // by number
    const unsigned int* nact;
    const int64_t* inv_off;      // by vertex
    const uint32_t* inv;
    const int64_t* rr_off;
    const uint32_t* memc;
    const uint8_t* rr_stratum;
    uint8_t* covered;            // per RR set
    uint8_t* picked;             // per vertex
    int32_t* seeds;
    GreedyOut* out;
    Weights W;
    int32_t n, k;
    int prefix;                  // 1: also the Eq. upper_2 bound of every prefix of the seeds
    uint32_t* cand;              // kCandCap numbers
    unsigned int* ncand;
    unsigned long long* pscore;  // per block
    uint32_t* pid;               // per block: vertex, number
    unsigned long long* psum;    // per block: 128-bit partial sums
    unsigned int* hist;          // 3 x kTopBins, zeroed
    unsigned int* bar;           // zeroed
    DevStatus* st;
    int spin_limit;              // rounds of a barrier wait before it gives up
};

// All blocks of the launch meet; false when the bounded wait gave up here.
template <bool kCluster>
__device__ bool grid_meet(const GreedyParams& P, unsigned int& target) {
    __shared__ int ok_s;
    if (kCluster) {  // the cluster's barrier: what a block wrote before is seen by the others after
        // not .aligned: the lanes of a warp arrive here from loops of different lengths
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        return true;
    }
    __syncthreads();
    if (gridDim.x == 1) return true;
    if (threadIdx.x == 0) {
        __threadfence();
        target += gridDim.x;
        atomicAdd(P.bar, 1u);
        int it = 0;
        unsigned int seen;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(P.bar) : "memory");
        } while ((int)(seen - target) < 0 && ++it < P.spin_limit);
        ok_s = (int)(seen - target) >= 0;
        if (!ok_s && atomicCAS(&P.st->code, 0, (int32_t)kErrSpin) == 0) P.st->detail = -1;
        __threadfence();
    }
    __syncthreads();
    return ok_s != 0;
}

// a block's winner: score, vertex, its range of the index (end = 0: not known)
struct Winner {
    unsigned long long score;
    int64_t begin, end;
    uint32_t v, pad;
};

// w into block `rank`'s copy of the shared array `to`, at this block's place (one cluster)
__device__ __forceinline__ void send_winner(Winner* to, unsigned int rank, const Winner& w) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(to + blockIdx.x);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(ra), "l"(w.score) : "memory");
    asm volatile("st.shared::cluster.u64 [%0 + 8], %1;" ::"r"(ra), "l"(w.begin) : "memory");
    asm volatile("st.shared::cluster.u64 [%0 + 16], %1;" ::"r"(ra), "l"(w.end) : "memory");
    asm volatile("st.shared::cluster.u32 [%0 + 24], %1;" ::"r"(ra), "r"(w.v) : "memory");
}

__device__ __forceinline__ void add128(unsigned long long& lo, unsigned long long& hi, unsigned long long a_lo,
                                       unsigned long long a_hi) {
    const unsigned long long l = lo + a_lo;
    hi += a_hi + (l < lo ? 1ull : 0ull);
    lo = l;
}

// The want-th largest score `kth` and how many of its copies are among the want largest (kleft; fewer
// scores than want: kth = 0). A radix select over 11-bit digits below the largest score `top`, most
// significant first; a digit of 0 is never counted (most scores have it), it is what is left when the
// others hold too few. Three histograms rotate: the next one is cleared between the barriers that
// separate its last readers from its next writers.
template <bool kCluster>
__device__ bool kth_score(const GreedyParams& P, unsigned int na, unsigned long long top, unsigned int want,
                          unsigned int* h, int& turn, unsigned int& target, unsigned long long& kth,
                          unsigned int& kleft) {
    __shared__ unsigned int digit_s, left_s;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t t0 = blockIdx.x * (int64_t)kGThreads + threadIdx.x, T = (int64_t)gridDim.x * kGThreads;
    unsigned long long prefix = 0;
    kleft = want;
    const int bits = top ? 64 - __clzll((long long)top) : 0;
    for (int sh = ((bits + kTopBits - 1) / kTopBits - 1) * kTopBits; sh >= 0; sh -= kTopBits) {
        unsigned int* hist = P.hist + turn * kTopBins;
        const int next = turn == 2 ? 0 : turn + 1;
        for (int i = threadIdx.x; i < kTopBins; i += kGThreads) {
            h[i] = 0;
            if (blockIdx.x == 0) P.hist[next * kTopBins + i] = 0;
        }
        __syncthreads();
        for (int64_t c = t0; c < na; c += T) {
            const unsigned long long x = __ldcg(P.score + c);
            const unsigned long long above = sh + kTopBits >= 64 ? 0ull : x >> (sh + kTopBits);
            const unsigned int d = (unsigned int)(x >> sh) & (kTopBins - 1);
            if (above == prefix && d) atomicAdd(&h[d], 1u);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kTopBins; i += kGThreads)
            if (h[i]) atomicAdd(&hist[i], h[i]);
        if (!grid_meet<kCluster>(P, target)) return false;
        if (wid == 0) {  // lane i: digits [64 i, 64 i + 64), from the highest lane down
            constexpr int per = kTopBins / 32;
            unsigned int sum = 0;
            for (int i = 0; i < per; ++i) sum += __ldcg(hist + lane * per + i);
            unsigned int suf = sum;  // this lane's digits and all higher ones
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_down_sync(0xFFFFFFFFu, suf, o);
                if (lane + o < 32) suf += t;
            }
            const uint32_t reach = __ballot_sync(0xFFFFFFFFu, suf >= kleft);
            if (reach == 0) {
                if (lane == 0) {
                    digit_s = 0;
                    left_s = kleft - suf;
                }
            } else if (lane == 31 - __clz(reach)) {
                unsigned int cum = suf - sum;
                int i = per - 1;
                for (; i > 0; --i) {
                    const unsigned int v = __ldcg(hist + lane * per + i);
                    if (cum + v >= kleft) break;
                    cum += v;
                }
                digit_s = (unsigned int)(lane * per + i);
                left_s = kleft - cum;
            }
        }
        __syncthreads();
        prefix = (prefix << kTopBits) | digit_s;
        kleft = left_s;
        turn = next;
        __syncthreads();
    }
    kth = prefix;
    return true;
}

// Eq. upper_2 (p_max = 1) for the seeds so far: cover plus the sum of the k largest scores (a picked or
// inactive vertex counts 0), entered into block 0's running minimum.
template <bool kCluster>
__device__ bool topk_bound(const GreedyParams& P, unsigned int na, unsigned long long top, unsigned long long cover,
                           unsigned int* h, int& turn, unsigned int& target, unsigned long long& best_lo,
                           unsigned long long& best_hi) {
    __shared__ unsigned long long slo[kGWarps], shi[kGWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t t0 = blockIdx.x * (int64_t)kGThreads + threadIdx.x, T = (int64_t)gridDim.x * kGThreads;
    unsigned long long prefix = 0;
    unsigned int kleft = 0;
    if (!kth_score<kCluster>(P, na, top, (unsigned int)P.k, h, turn, target, prefix, kleft)) return false;
    unsigned long long lo = 0, hi = 0;
    for (int64_t c = t0; c < na; c += T) {
        const unsigned long long x = __ldcg(P.score + c);
        if (x > prefix) add128(lo, hi, x, 0ull);
    }
    for (int o = 16; o > 0; o >>= 1)
        add128(lo, hi, __shfl_xor_sync(0xFFFFFFFFu, lo, o), __shfl_xor_sync(0xFFFFFFFFu, hi, o));
    if (lane == 0) {
        slo[wid] = lo;
        shi[wid] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kGWarps; ++w) add128(lo, hi, slo[w], shi[w]);
        P.psum[2 * blockIdx.x] = lo;
        P.psum[2 * blockIdx.x + 1] = hi;
    }
    if (!grid_meet<kCluster>(P, target)) return false;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        lo = hi = 0;
        for (unsigned int b = 0; b < gridDim.x; ++b) add128(lo, hi, __ldcg(P.psum + 2 * b), __ldcg(P.psum + 2 * b + 1));
        add128(lo, hi, kleft * prefix, __umul64hi(kleft, prefix));
        add128(lo, hi, cover, 0ull);
        if (hi < best_hi || (hi == best_hi && lo < best_lo)) {
            best_lo = lo;
            best_hi = hi;
        }
    }
    return true;
}

template <bool kCluster>
__global__ void __launch_bounds__(kGThreads, 1) k_greedy(GreedyParams P) {
    __shared__ Winner winners[kGCluster];  // the blocks' winners (one cluster)
    __shared__ Winner mine_s;              // this block's
    __shared__ int64_t win_b, win_e;
    __shared__ unsigned long long s_lam[HYPERIM_NSTRATA];
    __shared__ unsigned long long ss[kGWarps];
    __shared__ uint32_t si[kGWarps];
    __shared__ unsigned long long win_s;
    __shared__ uint32_t win_v;
    __shared__ unsigned int h[kTopBins];
    __shared__ LongSets sets;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t t0 = blockIdx.x * (int64_t)kGThreads + threadIdx.x, T = (int64_t)gridDim.x * kGThreads;
    const unsigned int na = P.act ? *P.nact : (unsigned int)P.n;
    unsigned int target = 0;
    int turn = 0;
    unsigned long long cover = 0, best_lo = ~0ull, best_hi = ~0ull;
    if (threadIdx.x < HYPERIM_NSTRATA) s_lam[threadIdx.x] = 0;
    // in a cluster every block has to run before one writes into another's shared memory (send_winner)
    if (kCluster) grid_meet<kCluster>(P, target);
    else __syncthreads();
    int32_t round = 0;
    unsigned int nc = 0;            // candidates (0: none, every active vertex is looked at)
    unsigned long long floor = 0;   // every other vertex scores less than this
    int32_t next_try = 0, wait = 1;  // candidates are not looked for before this round
    uint32_t own_c = 0, own_v = 0xFFFFFFFFu;  // this thread's candidate: number, vertex, index range
    int64_t own_b = 0, own_e = 0;
    for (;; ++round) {
        if (round == P.k && !P.prefix) break;
        // the best (score, lowest id): per block, then over the blocks' winners by every block
        unsigned long long bs = 0;
        uint32_t bi = 0xFFFFFFFFu;
        auto take = [&](unsigned long long x, uint32_t v) {
            if (x && better(x, v, bs, bi)) { bs = x; bi = v; }
        };
        auto reduce = [&]() {  // over the block; the result is warp 0's
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
                const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
                if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
            }
            if (lane == 0) { ss[wid] = bs; si[wid] = bi; }
            __syncthreads();
            if (wid == 0) {
                bs = lane < kGWarps ? ss[lane] : 0ull;
                bi = lane < kGWarps ? si[lane] : 0xFFFFFFFFu;
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
                    const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
                    if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
                }
            }
        };
        auto share = [&]() {  // over the blocks; the result is every thread's, in win_s and win_v
            reduce();
            if (kCluster) {
                if (threadIdx.x == 0) mine_s = Winner{bs, 0, 0, bi, 0u};
                __syncthreads();
                if (own_e && own_v == mine_s.v) {
                    mine_s.begin = own_b;
                    mine_s.end = own_e;
                }
                __syncthreads();
                if (wid == 0 && lane < (int)gridDim.x) send_winner(winners, (unsigned int)lane, mine_s);
                if (!grid_meet<kCluster>(P, target)) return false;
                if (wid == 0) {
                    bs = lane < (int)gridDim.x ? winners[lane].score : 0ull;
                    bi = lane < (int)gridDim.x ? winners[lane].v : 0xFFFFFFFFu;
                    const uint32_t sent = bi;
                    for (int o = 16; o > 0; o >>= 1) {
                        const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
                        const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
                        if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
                    }
                    if (lane < (int)gridDim.x && sent == bi && bs) {  // the one block that sent the winner
                        win_b = winners[lane].begin;
                        win_e = winners[lane].end;
                    }
                }
            } else if (gridDim.x > 1) {
                if (threadIdx.x == 0) {
                    P.pscore[blockIdx.x] = bs;
                    P.pid[blockIdx.x] = bi;
                }
                if (!grid_meet<kCluster>(P, target)) return false;
                bs = 0;
                bi = 0xFFFFFFFFu;
                for (int b = threadIdx.x; b < (int)gridDim.x; b += kGThreads) {
                    const unsigned long long x = __ldcg(P.pscore + b);
                    const uint32_t v = __ldcg(P.pid + b);
                    if (better(x, v, bs, bi)) { bs = x; bi = v; }
                }
                reduce();
            }
            if (threadIdx.x == 0) {
                win_s = bs;
                win_v = bi;
            }
            __syncthreads();
            return true;
        };
        bool full = nc == 0;
        if (kCluster && !full) {
            if (own_e) {
                bs = __ldcg(P.score + own_c);
                if (bs) bi = own_v;
            }
            if (!share()) return;
            full = win_s < floor;
            bs = 0;
            bi = 0xFFFFFFFFu;
        }
        if (full) {
            // the blocks have read the winners above before any of them is written again
            if (nc && !grid_meet<kCluster>(P, target)) return;
            own_e = 0;
            own_v = 0xFFFFFFFFu;
            const int64_t na4 = na >> 2;
            for (int64_t q = t0; q < na4; q += T) {
                const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2*>(P.score) + 2 * q);
                const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2*>(P.score) + 2 * q + 1);
                // the ids with the scores, not after them: where nearly all scores are alike every one of them decides
                uint4 v = make_uint4((uint32_t)(4 * q), (uint32_t)(4 * q + 1), (uint32_t)(4 * q + 2), (uint32_t)(4 * q + 3));
                if (P.act) v = reinterpret_cast<const uint4*>(P.act)[q];
                take(a.x, v.x);
                take(a.y, v.y);
                take(b.x, v.z);
                take(b.y, v.w);
            }
            for (int64_t c = 4 * na4 + t0; c < na; c += T) take(__ldcg(P.score + c), P.act ? (uint32_t)P.act[c] : (uint32_t)c);
            if (!share()) return;
            nc = 0;
            if (kCluster && !P.prefix && na > 4 * kCand && P.k - round > 8 && win_s && round >= next_try) {
                unsigned int kleft;
                if (blockIdx.x == 0 && threadIdx.x == 0) *P.ncand = 0;
                if (!kth_score<kCluster>(P, na, win_s, kCand, h, turn, target, floor, kleft)) return;
                if (floor) {
                    for (int64_t c = t0; c < na; c += T)
                        if (__ldcg(P.score + c) >= floor) {
                            const unsigned int at = atomicAdd(P.ncand, 1u);
                            if (at < kCandCap) P.cand[at] = (uint32_t)c;
                        }
                    if (!grid_meet<kCluster>(P, target)) return;
                    nc = __ldcg(P.ncand);
                    if (nc > kCandCap) nc = 0;  // too many at the threshold: no candidates
                    if (t0 < nc) {
                        own_c = __ldcg(P.cand + t0);
                        own_v = P.act ? (uint32_t)P.act[own_c] : own_c;
                        own_b = P.inv_off[own_v];
                        own_e = P.inv_off[own_v + 1];
                    }
                }
                if (nc) {
                    wait = 1;
                } else {
                    next_try = round + wait;
                    wait *= 2;
                }
            }
        }
        const unsigned long long win = win_s;
        const uint32_t v = win_v;
        if (P.prefix && !topk_bound<kCluster>(P, na, win, cover, h, turn, target, best_lo, best_hi)) return;
        if (round == P.k || win == 0) break;
        cover += win;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            P.seeds[round] = (int32_t)v;
            P.picked[v] = 1;
        }
        // retire the winner's sets that are not covered yet (a set holds it once: one warp finds it)
        int64_t b, e;
        if (kCluster && win_e) {
            b = win_b;
            e = win_e;
        } else {
            b = P.inv_off[v];
            e = P.inv_off[v + 1];
        }
        block_sets(
            sets, e - b,
            [&](int64_t t, int64_t& x0, int64_t& x1, unsigned long long& tag) {
                const uint32_t r = P.inv[b + t];
                x0 = P.rr_off[r];
                x1 = P.rr_off[r + 1];
                const int s = P.rr_stratum[r];
                if (__ldcg(P.covered + r)) return false;
                __syncwarp();
                if (lane == 0) {
                    __stcg(P.covered + r, (uint8_t)1);
                    atomicAdd(&s_lam[s], 1ull);
                }
                tag = 0ull - P.W.w[s];
                return true;
            },
            [&](int64_t x, unsigned long long neg) { atomicAdd(&P.score[P.memc[x]], neg); });
        if (!grid_meet<kCluster>(P, target)) return;
    }
    __syncthreads();
    if (threadIdx.x < HYPERIM_NSTRATA && s_lam[threadIdx.x]) atomicAdd(&P.out->lam[threadIdx.x], s_lam[threadIdx.x]);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        P.out->best_lo = best_lo;
        P.out->best_hi = best_hi;
        // every set is covered: the lowest ids not picked yet
        for (int32_t v = 0; round < P.k; ++round, ++v) {
            while (P.picked[v]) ++v;
            P.seeds[round] = v;
        }
    }
}

// coverage of a seed set: RR sets with at least one member in S, per stratum; one warp per set
__global__ void k_coverage(const int64_t* __restrict__ rr_off, const int32_t* __restrict__ mem,
                           const uint8_t* __restrict__ rr_stratum, const uint32_t* __restrict__ rr_j,
                           int64_t N, Limits L, const uint8_t* __restrict__ in_s,
                           unsigned long long* __restrict__ lam) {
    __shared__ unsigned int s_lam[HYPERIM_NSTRATA];  // 16 words for every hit would queue at the L2
    if (threadIdx.x < HYPERIM_NSTRATA) s_lam[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = warp; r < N; r += nwarps) {
        if (L.skip(rr_stratum, rr_j, r)) continue;
        const int64_t b = rr_off[r], e = rr_off[r + 1];
        bool hit = false;
        for (int64_t base = b; base < e; base += 32) {
            const int64_t x = base + lane;
            if (__any_sync(0xFFFFFFFFu, x < e && in_s[mem[x]] != 0)) { hit = true; break; }
        }
        if (hit && lane == 0) atomicAdd(&s_lam[rr_stratum[r]], 1u);
    }
    __syncthreads();
    if (threadIdx.x < HYPERIM_NSTRATA && s_lam[threadIdx.x])
        atomicAdd(&lam[threadIdx.x], (unsigned long long)s_lam[threadIdx.x]);
}

__global__ void __launch_bounds__(kCoverThreads)
k_cover_sets(const int64_t* __restrict__ rr_off, const int32_t* __restrict__ mem, const uint8_t* __restrict__ rr_stratum,
             const uint32_t* __restrict__ rr_j, int64_t N, Limits L, int32_t n, const int32_t* __restrict__ seeds,
             int32_t k, int per, unsigned long long* __restrict__ lam) {
    extern __shared__ uint32_t cover_slots[];
    cover_sets(cover_slots, rr_off, mem, rr_stratum, N, n, seeds, k, per, lam,
               [&](int64_t r) { return L.skip(rr_stratum, rr_j, r); });
}

__global__ void k_mark(const int32_t* __restrict__ seeds, int32_t k, uint8_t* __restrict__ in_s) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x)
        in_s[seeds[i]] = 1;
}

// ---- batched form: greedy max coverage and the R2 coverage of many queries, one block each ----
// A query's block builds the inverted index of its R1 view, runs the k greedy rounds (argmax over
// the unpicked vertices, lowest id on ties; retirement of the covered sets) and counts the sets
// of its R2 view that hold a seed: the same integer arithmetic as the grid kernels above, so the
// seeds and coverages are identical. Scratch per block, sized for the batch's largest graph and
// view; queries are taken from a counter, so a block that finishes a small query takes the next.
constexpr int kGBThreads = 1024;
constexpr int kGBWarps = kGBThreads / 32;

struct GreedyBatchQuery {
    const int64_t* off1;
    const int32_t* mem1;
    const uint8_t* str1;
    const uint32_t* j1;
    int64_t count1;
    Limits L1;
    const int64_t* off2;
    const int32_t* mem2;
    const uint8_t* str2;
    const uint32_t* j2;
    int64_t count2;
    Limits L2;
    Weights W;
    int32_t n, k;
    int32_t* seeds;             // k entries
    unsigned long long* lam;    // lambda_r1[16], lambda_r2[16]
};

struct GreedyBatchParams {
    const GreedyBatchQuery* q;
    int nq;
    unsigned int* next;
    unsigned long long* score;  // per block: n_cap
    uint32_t* off;              // per block: n_cap + 1 (counts, then index ends)
    uint8_t* picked;            // per block: n_cap
    uint32_t* inv;              // per block: inv_cap
    uint32_t* covered;          // per block: cov_cap
    int64_t n_cap, inv_cap, cov_cap;
};

__global__ void __launch_bounds__(kGBThreads, 1) k_greedy_batch(GreedyBatchParams B) {
    __shared__ unsigned long long s_lam[2 * HYPERIM_NSTRATA];
    __shared__ unsigned long long ss[kGBWarps];
    __shared__ uint32_t si[kGBWarps];
    __shared__ uint32_t s_part[kGBWarps];
    __shared__ int s_q, s_best;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long* score = B.score + (int64_t)blockIdx.x * B.n_cap;
    uint32_t* off = B.off + (int64_t)blockIdx.x * (B.n_cap + 1);
    uint8_t* picked = B.picked + (int64_t)blockIdx.x * B.n_cap;
    uint32_t* inv = B.inv + (int64_t)blockIdx.x * B.inv_cap;
    uint32_t* covered = B.covered + (int64_t)blockIdx.x * B.cov_cap;
    for (;;) {
        if (threadIdx.x == 0) s_q = (int)atomicAdd(B.next, 1u);
        __syncthreads();
        if (s_q >= B.nq) break;
        const GreedyBatchQuery& Q = B.q[s_q];
        const int32_t n = Q.n;
        for (int64_t v = threadIdx.x; v < n; v += kGBThreads) {
            score[v] = 0;
            off[v] = 0;
            picked[v] = 0;
        }
        for (int64_t r = threadIdx.x; r < Q.count1; r += kGBThreads) covered[r] = 0;
        if (threadIdx.x < 2 * HYPERIM_NSTRATA) s_lam[threadIdx.x] = 0;
        __syncthreads();
        // occurrences of each vertex over the R1 view
        for (int64_t r = wid; r < Q.count1; r += kGBWarps) {
            if (Q.L1.skip(Q.str1, Q.j1, r)) continue;
            for (int64_t x = Q.off1[r] + lane; x < Q.off1[r + 1]; x += 32) atomicAdd(&off[Q.mem1[x]], 1u);
        }
        __syncthreads();
        // exclusive scan of the counts, in place: each thread one contiguous range
        {
            const int64_t per = ((int64_t)n + kGBThreads - 1) / kGBThreads;
            const int64_t b = (int64_t)threadIdx.x * per, e = min((int64_t)n, b + per);
            uint32_t sum = 0;
            for (int64_t v = b; v < e; ++v) sum += __ldcg(off + v);
            uint32_t incl = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) s_part[wid] = incl;
            __syncthreads();
            uint32_t base = 0;
            for (int w = 0; w < wid; ++w) base += s_part[w];
            uint32_t run = base + incl - sum;
            for (int64_t v = b; v < e; ++v) {
                const uint32_t c = __ldcg(off + v);
                off[v] = run;
                run += c;
            }
        }
        __syncthreads();
        // inverted index and initial scores; afterwards off[v] is the end of v's entries
        for (int64_t r = wid; r < Q.count1; r += kGBWarps) {
            if (Q.L1.skip(Q.str1, Q.j1, r)) continue;
            const unsigned long long w = Q.W.w[Q.str1[r]];
            for (int64_t x = Q.off1[r] + lane; x < Q.off1[r + 1]; x += 32) {
                const int32_t v = Q.mem1[x];
                inv[atomicAdd(&off[v], 1u)] = (uint32_t)r;
                atomicAdd(&score[v], w);
            }
        }
        __syncthreads();
        for (int round = 0; round < Q.k; ++round) {
            unsigned long long bs = 0;
            uint32_t bi = 0xFFFFFFFFu;
            scan_unpicked<true>(score, picked, n, threadIdx.x, kGBThreads, bs, bi);
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
                const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
                if (better(os, oi, bs, bi)) { bs = os; bi = oi; }
            }
            if (lane == 0) { ss[wid] = bs; si[wid] = bi; }
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < kGBWarps; ++w)
                    if (better(ss[w], si[w], bs, bi)) { bs = ss[w]; bi = si[w]; }
                s_best = (int)bi;
                Q.seeds[round] = (int32_t)bi;
                picked[bi] = 1;
            }
            __syncthreads();
            const int32_t v = s_best;
            const int64_t b = v ? (int64_t)__ldcg(off + v - 1) : 0, e = __ldcg(off + v);
            for (int64_t t = b + wid; t < e; t += kGBWarps) {
                const uint32_t r = inv[t];
                uint32_t old = 0;
                if (lane == 0) old = atomicExch(&covered[r], 1u);
                old = __shfl_sync(0xFFFFFFFFu, old, 0);
                if (old) continue;
                const int s = Q.str1[r];
                const unsigned long long neg = 0ull - Q.W.w[s];
                if (lane == 0) atomicAdd(&s_lam[s], 1ull);
                for (int64_t x = Q.off1[r] + lane; x < Q.off1[r + 1]; x += 32) atomicAdd(&score[Q.mem1[x]], neg);
            }
            __syncthreads();
        }
        // coverage of the seed set on the R2 view
        for (int64_t r = wid; r < Q.count2; r += kGBWarps) {
            if (Q.L2.skip(Q.str2, Q.j2, r)) continue;
            const int64_t b = Q.off2[r], e = Q.off2[r + 1];
            bool hit = false;
            for (int64_t base = b; base < e; base += 32) {
                const int64_t x = base + lane;
                if (__any_sync(0xFFFFFFFFu, x < e && picked[Q.mem2[x]] != 0)) { hit = true; break; }
            }
            if (hit && lane == 0) atomicAdd(&s_lam[HYPERIM_NSTRATA + Q.str2[r]], 1ull);
        }
        __syncthreads();
        if (threadIdx.x < 2 * HYPERIM_NSTRATA) Q.lam[threadIdx.x] = s_lam[threadIdx.x];
        __syncthreads();
    }
}

int grid_cap(int64_t items, int threads, int sm, int per_sm) {
    int64_t b = (items + threads - 1) / threads;
    const int64_t cap = (int64_t)sm * per_sm;
    if (b < 1) b = 1;
    return (int)std::min(b, cap);
}

}  // namespace

namespace {
// the view of p that lim names (nullptr: the whole pool); lim[s] <= p->n_s[s]
Limits make_limits(const hyperim_pool* p, const uint64_t* lim, uint64_t view_ns[HYPERIM_NSTRATA]) {
    Limits L{};
    for (int i = 0; i < HYPERIM_NSTRATA; ++i) {
        view_ns[i] = lim ? std::min<uint64_t>(lim[i], p->n_s[i]) : p->n_s[i];
        L.lim[i] = (uint32_t)std::min<uint64_t>(view_ns[i], 0xFFFFFFFFull);
        if (view_ns[i] < p->n_s[i]) L.on = 1;
    }
    return L;
}
}  // namespace

namespace {
// one launch of kGCluster blocks as one cluster
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, cudaStream_t s) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kGCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(kGCluster);
    cfg.blockDim = dim3(kGThreads);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

// whether the device takes such a cluster (16 blocks is more than the portable 8): asked once
bool cluster_fits() {
    static const bool fits = [] {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        cluster_config(cfg, at, nullptr);
        int clusters = 0;
        bool ok = cudaFuncSetAttribute(k_greedy<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&clusters, k_greedy<true>, &cfg) == cudaSuccess && clusters > 0;
        if (!ok) cudaGetLastError();
        return ok;
    }();
    return fits;
}
}  // namespace

hyperim_status greedy(hyperim_graph* g, hyperim_pool* p, int32_t k, int32_t* seeds_host,
                      uint64_t lambda_s[HYPERIM_NSTRATA], uint64_t* prefix_upper, const uint64_t* lim) {
    cudaStream_t s = g->stream;
    const int32_t n = g->n;
    const int64_t N = p->count, T = p->total;
    const int sm = g->sm_count;
    if (N >= (int64_t)0xFFFFFFFFll) return set_error(HYPERIM_EOVERFLOW, "more than 2^32 - 1 RR sets");
    uint64_t view_ns[HYPERIM_NSTRATA];
    const Limits L = make_limits(p, lim, view_ns);
    Weights W;
    for (int i = 0; i < HYPERIM_NSTRATA; ++i)
        W.w[i] = stratum_weight(g, p->root_mode, view_ns[i], i);
    hyperim_status st;
    CallBuffers tmp(g);
    uint32_t *cnt = nullptr, *inv = nullptr, *cidx = nullptr, *memc = nullptr, *pid = nullptr, *cand = nullptr;
    int64_t* inv_off = nullptr;
    unsigned long long *score = nullptr, *pscore = nullptr, *psum = nullptr;
    int32_t *act = nullptr, *seeds_d = nullptr;
    // cleared together: the output record, barrier, counters, histograms, picked and covered flags
    struct Zero {
        GreedyOut out;
        unsigned int bar, nact, ncand, pad;
        unsigned int hist[3 * kTopBins];
    };
    uint8_t* zero = nullptr;
    const size_t bytes_zero = sizeof(Zero) + (size_t)n + (size_t)N;
    const size_t bytes_cnt = sizeof(uint32_t) * ((size_t)n + 1);
    const size_t members = (size_t)std::max<int64_t>(T, 1);
    if ((st = tmp.alloc(&cnt, bytes_cnt))) return st;
    if ((st = tmp.alloc(&inv_off, sizeof(int64_t) * ((size_t)n + 1)))) return st;
    if ((st = tmp.alloc(&inv, sizeof(uint32_t) * members))) return st;
    if ((st = tmp.alloc(&score, sizeof(unsigned long long) * (size_t)n))) return st;
    if ((st = tmp.alloc(&zero, bytes_zero))) return st;
    const int most_blocks = std::max(sm, kGCluster);
    if ((st = tmp.alloc(&pscore, sizeof(unsigned long long) * 3 * (size_t)most_blocks))) return st;
    if ((st = tmp.alloc(&pid, sizeof(uint32_t) * (size_t)most_blocks))) return st;
    if ((st = tmp.alloc(&cand, sizeof(uint32_t) * kCandCap))) return st;
    if ((st = tmp.alloc(&seeds_d, sizeof(int32_t) * (size_t)k))) return st;
    psum = pscore + most_blocks;
    Zero* z = reinterpret_cast<Zero*>(zero);
    HYP_CUDA(cudaMemsetAsync(cnt, 0, bytes_cnt, s));
    HYP_CUDA(cudaMemsetAsync(zero, 0, bytes_zero, s));
    if (T > 0 && !L.on) { k_count_occ<<<grid_cap(T, 256, sm, 32), 256, 0, s>>>(p->rr_mem, T, cnt); count_launch(); }
    if (T > 0 && L.on)
        { k_count_occ_view<<<grid_cap(N * 32, 256, sm, 32), 256, 0, s>>>(p->rr_off, p->rr_mem, p->rr_stratum,
                                                                        p->rr_j, N, L, cnt); count_launch(); }
    if ((st = exclusive_scan_u32_to_i64(g, cnt, inv_off, n))) return st;
    // under a budget, and where the memory for numbers and renumbered members is not to be had (all that the
    // call cannot do without is there by now), the vertices keep their ids
    bool numbered = false;
    if (takes_optional(g)) {
        const size_t needed = tmp.count();
        numbered = tmp.try_alloc(&memc, sizeof(uint32_t) * members) &&
                   tmp.try_alloc(&act, sizeof(int32_t) * (size_t)n) &&
                   tmp.try_alloc(&cidx, sizeof(uint32_t) * (size_t)n);
        if (!numbered) {
            tmp.release_after(needed);
            memc = cidx = nullptr;
            act = nullptr;
        }
    }
    if (numbered) {
        k_active<<<(unsigned)(((int64_t)n + kActThreads * kActItems - 1) / (kActThreads * kActItems)), kActThreads, 0, s>>>(
            cnt, n, act, cidx, score, &z->nact);
        count_launch();
    } else {
        HYP_CUDA(cudaMemsetAsync(cnt, 0, bytes_cnt, s));
        HYP_CUDA(cudaMemsetAsync(score, 0, sizeof(unsigned long long) * (size_t)n, s));
    }
    if (N > 0)
        { k_scatter_active<<<grid_cap(N * 32 / kSetsPerWarp, kGThreads, sm, 32), kGThreads, 0, s>>>(p->rr_off, p->rr_mem, p->rr_stratum, p->rr_j,
                                                                       N, L, inv_off, cnt, inv, cidx, memc, score,
                                                                       W); count_launch(); }
    HYP_CUDA(cudaGetLastError());
    // Blocks: by the pool's members, all resident together when more than one; by the vertices too where they
    // are not numbered, since a look at every vertex then reads all n scores. Without numbers a cluster's 16 SMs
    // do that quickly enough up to kGClusterScan vertices, beyond it only with members for a sixteenth of them
    // (else there are no candidates to keep). 100 seeds under a budget, by members alone / now (with two launches a
    // round): 5,389 members of 2M vertices 26.9 / 0.9 ms (1.8), 34,034 29.6 / 1.0 (1.9), 341,753 1.2 / 1.1 (1.9)
    // and 1.4 in the grid, 3,548 of 200k 3.4 / 0.9 (1.6), 26,041 of 600k 1.0 in the grid, 2.0 in a cluster.
    const int64_t work = numbered ? T : std::max<int64_t>(T, n);
    int blocks = (int)std::min<int64_t>(std::max<int64_t>(work / kGMembersPerBlock, 1), sm);
    const bool cluster = blocks > 1 && T <= kGClusterMembers && (numbered || n <= kGClusterScan || T >= n / 16) && cluster_fits();
    if (cluster) {
        blocks = kGCluster;
    } else if (blocks > 1) {
        int per_sm = 0;
        HYP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy<false>, kGThreads, 0));
        blocks = std::max(1, std::min(blocks, per_sm * sm));
    }
    GreedyParams G{act, score, &z->nact, inv_off, inv, p->rr_off,
                   numbered ? memc : reinterpret_cast<const uint32_t*>(p->rr_mem), p->rr_stratum,
                   zero + sizeof(Zero) + (size_t)n, zero + sizeof(Zero), seeds_d, &z->out, W, n, k,
                   prefix_upper ? 1 : 0, cand, &z->ncand, pscore, pid, psum, z->hist, &z->bar, g->d_status, wait_rounds(g)};
    if (cluster) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        cluster_config(cfg, at, s);
        HYP_CUDA(cudaLaunchKernelEx(&cfg, k_greedy<true>, G));
    } else if (blocks > 1) {
        void* args[] = {&G};
        HYP_CUDA(cudaLaunchCooperativeKernel((const void*)k_greedy<false>, dim3((unsigned)blocks), dim3(kGThreads), args,
                                             0, s));
    } else {
        k_greedy<false><<<1, kGThreads, 0, s>>>(G);
    }
    count_launch();
    HYP_CUDA(cudaGetLastError());
    GreedyOut out;
    HYP_CUDA(cudaMemcpyAsync(seeds_host, seeds_d, sizeof(int32_t) * (size_t)k, cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaMemcpyAsync(&out, &z->out, sizeof(out), cudaMemcpyDeviceToHost, s));
    if ((st = check_device_status(g, "greedy"))) return st;  // synchronises
    for (int i = 0; i < HYPERIM_NSTRATA; ++i) lambda_s[i] = out.lam[i];
    if (prefix_upper) {
        prefix_upper[0] = out.best_lo;
        prefix_upper[1] = out.best_hi;
    }
    return HYPERIM_OK;
}

hyperim_status coverage(hyperim_graph* g, hyperim_pool* p, const int32_t* seeds_host, int32_t k,
                        uint64_t lambda_s[HYPERIM_NSTRATA], const uint64_t* lim) {
    cudaStream_t s = g->stream;
    const int64_t N = p->count;
    uint64_t view_ns[HYPERIM_NSTRATA];
    const Limits L = make_limits(p, lim, view_ns);
    hyperim_status st;
    CallBuffers tmp(g);
    uint8_t* in_s = nullptr;
    unsigned long long* lam = nullptr;
    int32_t* sd = nullptr;
    const size_t kk = (size_t)std::max(k, 1);
    const bool on_chip = k <= kCoverSeeds;
    if (!on_chip && (st = tmp.alloc(&in_s, (size_t)g->n))) return st;
    if ((st = tmp.alloc(&lam, sizeof(unsigned long long) * HYPERIM_NSTRATA))) return st;
    if ((st = tmp.alloc(&sd, sizeof(int32_t) * kk))) return st;
    HYP_CUDA(cudaMemsetAsync(lam, 0, sizeof(unsigned long long) * HYPERIM_NSTRATA, s));
    if (k > 0) HYP_CUDA(cudaMemcpyAsync(sd, seeds_host, sizeof(int32_t) * (size_t)k, cudaMemcpyHostToDevice, s));
    if (!on_chip) {
        HYP_CUDA(cudaMemsetAsync(in_s, 0, (size_t)g->n, s));
        { k_mark<<<grid_cap(k, 256, g->sm_count, 4), 256, 0, s>>>(sd, k, in_s); count_launch(); }
    }
    if (N > 0 && on_chip) {
        const int per = cover_per(N, g->sm_count);
        { k_cover_sets<<<cover_blocks(N, per, k, g->sm_count), kCoverThreads,
                       cover_smem(k), s>>>(p->rr_off, p->rr_mem, p->rr_stratum, p->rr_j, N, L, g->n, sd, k, per,
                                           lam); count_launch(); }
    } else if (N > 0)
        { k_coverage<<<grid_cap(N * 32, 256, g->sm_count, 32), 256, 0, s>>>(p->rr_off, p->rr_mem,
                                                                          p->rr_stratum, p->rr_j, N, L, in_s,
                                                                          lam); count_launch(); }
    HYP_CUDA(cudaGetLastError());
    unsigned long long hl[HYPERIM_NSTRATA];
    HYP_CUDA(cudaMemcpyAsync(hl, lam, sizeof(hl), cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < HYPERIM_NSTRATA; ++i) lambda_s[i] = hl[i];
    return check_device_status(g, "coverage");
}

}  // namespace hyperim

// ---- greedy one round at a time (sharded pools) ---------------------------------------------
// The state of Algorithm 1 on one pool (a prefix view of it): the inverted index and the
// weighted marginal scores of its RR sets, which sets are covered, which vertices are picked and
// Lambda per stratum. greedy_pick takes the argmax over a score vector the caller supplies --
// the sum, over every shard of a pool, of their scores (integer sums: the order of the shards'
// additions does not matter) -- then retires the pick's uncovered sets of this shard.
namespace hyperim {

struct GreedyState {
    hyperim_graph* g = nullptr;
    hyperim_pool* p = nullptr;
    std::shared_lock<std::shared_mutex> lock;  // the pool may not grow while the state lives
    Weights W{};
    int ablocks = 0;
    uint32_t *cnt = nullptr, *inv = nullptr, *covered = nullptr, *bid = nullptr, *ticket = nullptr;
    int64_t* inv_off = nullptr;
    unsigned long long *score = nullptr, *lam = nullptr, *bscore = nullptr;
    uint8_t* picked = nullptr;
    int32_t* best = nullptr;
    size_t bytes_cnt = 0, bytes_inv = 0, bytes_cov = 0;
};

namespace {
void free_state(GreedyState* s) {
    hyperim_graph* g = s->g;
    const size_t n = (size_t)g->n;
    dev_free(g, s->cnt, s->bytes_cnt);
    dev_free(g, s->inv_off, sizeof(int64_t) * (n + 1));
    dev_free(g, s->inv, s->bytes_inv);
    dev_free(g, s->score, sizeof(unsigned long long) * n);
    dev_free(g, s->picked, n);
    dev_free(g, s->covered, s->bytes_cov);
    dev_free(g, s->lam, sizeof(unsigned long long) * HYPERIM_NSTRATA);
    dev_free(g, s->bscore, sizeof(unsigned long long) * s->ablocks);
    dev_free(g, s->bid, sizeof(uint32_t) * s->ablocks);
    dev_free(g, s->ticket, sizeof(uint32_t) * 2);
    dev_free(g, s->best, sizeof(int32_t) * 2);
    cudaStreamSynchronize(g->stream);
    delete s;
}
}  // namespace

hyperim_status greedy_begin(hyperim_graph* g, hyperim_pool* p, const uint64_t* lim, GreedyState** out) {
    *out = nullptr;
    GreedyState* s = new (std::nothrow) GreedyState();
    if (!s) return set_error(HYPERIM_ENOMEM, "host allocation failed");
    s->g = g;
    s->p = p;
    s->lock = std::shared_lock<std::shared_mutex>(p->mu);
    cudaStream_t st_ = g->stream;
    const int32_t n = g->n;
    const int64_t N = p->count, T = p->total;
    const int sm = g->sm_count;
    if (N >= (int64_t)0xFFFFFFFFll) {
        delete s;
        return set_error(HYPERIM_EOVERFLOW, "more than 2^32 - 1 RR sets");
    }
    uint64_t view_ns[HYPERIM_NSTRATA];
    const Limits L = make_limits(p, lim, view_ns);
    for (int i = 0; i < HYPERIM_NSTRATA; ++i) s->W.w[i] = stratum_weight(g, p->root_mode, view_ns[i], i);
    s->ablocks = grid_cap(n, kArgThreads, sm, 2);
    s->bytes_cnt = sizeof(uint32_t) * ((size_t)n + 1);
    s->bytes_inv = sizeof(uint32_t) * (size_t)std::max<int64_t>(T, 1);
    s->bytes_cov = sizeof(uint32_t) * (size_t)std::max<int64_t>(N, 1);
    hyperim_status st;
    auto fail = [&](hyperim_status e) {
        free_state(s);
        return e;
    };
    if ((st = dev_alloc(g, (void**)&s->cnt, s->bytes_cnt)) || (st = dev_alloc(g, (void**)&s->inv_off, sizeof(int64_t) * ((size_t)n + 1))) ||
        (st = dev_alloc(g, (void**)&s->inv, s->bytes_inv)) || (st = dev_alloc(g, (void**)&s->score, sizeof(unsigned long long) * (size_t)n)) ||
        (st = dev_alloc(g, (void**)&s->picked, (size_t)n)) || (st = dev_alloc(g, (void**)&s->covered, s->bytes_cov)) ||
        (st = dev_alloc(g, (void**)&s->lam, sizeof(unsigned long long) * HYPERIM_NSTRATA)) ||
        (st = dev_alloc(g, (void**)&s->bscore, sizeof(unsigned long long) * s->ablocks)) ||
        (st = dev_alloc(g, (void**)&s->bid, sizeof(uint32_t) * s->ablocks)) || (st = dev_alloc(g, (void**)&s->ticket, sizeof(uint32_t) * 2)) ||
        (st = dev_alloc(g, (void**)&s->best, sizeof(int32_t) * 2)))
        return fail(st);
    cudaError_t e = cudaMemsetAsync(s->cnt, 0, s->bytes_cnt, st_);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->score, 0, sizeof(unsigned long long) * (size_t)n, st_);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->picked, 0, (size_t)n, st_);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->covered, 0, s->bytes_cov, st_);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->lam, 0, sizeof(unsigned long long) * HYPERIM_NSTRATA, st_);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->ticket, 0, sizeof(uint32_t) * 2, st_);
    if (e != cudaSuccess) return fail(cuda_fail(e, "greedy state"));
    if (T > 0 && !L.on) { k_count_occ<<<grid_cap(T, 256, sm, 32), 256, 0, st_>>>(p->rr_mem, T, s->cnt); count_launch(); }
    if (T > 0 && L.on)
        { k_count_occ_view<<<grid_cap(N * 32, 256, sm, 32), 256, 0, st_>>>(p->rr_off, p->rr_mem, p->rr_stratum, p->rr_j, N, L,
                                                                          s->cnt); count_launch(); }
    if ((st = exclusive_scan_u32_to_i64(g, s->cnt, s->inv_off, n))) return fail(st);
    e = cudaMemsetAsync(s->cnt, 0, s->bytes_cnt, st_);
    if (e != cudaSuccess) return fail(cuda_fail(e, "greedy state"));
    if (N > 0)
        { k_scatter_inv<<<grid_cap(N * 32, 256, sm, 32), 256, 0, st_>>>(p->rr_off, p->rr_mem, p->rr_stratum, p->rr_j, N, L,
                                                                      s->inv_off, s->cnt, s->inv, s->score, s->W); count_launch(); }
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(cuda_fail(e, "greedy index"));
    *out = s;
    return HYPERIM_OK;
}

hyperim_status greedy_scores(GreedyState* s, unsigned long long* dev_out) {
    HYP_CUDA(cudaMemcpyAsync(dev_out, s->score, sizeof(unsigned long long) * (size_t)s->g->n, cudaMemcpyDeviceToDevice,
                             s->g->stream));
    return HYPERIM_OK;
}

hyperim_status greedy_pick(GreedyState* s, const unsigned long long* dev_total, int32_t* picked) {
    hyperim_graph* g = s->g;
    hyperim_pool* p = s->p;
    cudaStream_t st_ = g->stream;
    { k_argmax<<<s->ablocks, kArgThreads, 0, st_>>>(dev_total ? dev_total : s->score, s->picked, g->n, s->bscore, s->bid,
                                                    s->ticket, s->best); count_launch(); }
    { k_retire<<<g->sm_count * 8, 256, 0, st_>>>(s->best, s->inv_off, s->inv, p->rr_off, p->rr_mem, p->rr_stratum,
                                                 s->covered, s->score, s->lam, s->W); count_launch(); }
    HYP_CUDA(cudaGetLastError());
    HYP_CUDA(cudaMemcpyAsync(picked, s->best, sizeof(int32_t), cudaMemcpyDeviceToHost, st_));
    HYP_CUDA(cudaStreamSynchronize(st_));
    return check_device_status(g, "greedy pick");
}

hyperim_status greedy_end(GreedyState* s, uint64_t lambda_s[HYPERIM_NSTRATA]) {
    unsigned long long hl[HYPERIM_NSTRATA];
    cudaError_t e = cudaMemcpyAsync(hl, s->lam, sizeof(hl), cudaMemcpyDeviceToHost, s->g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->g->stream);
    if (e == cudaSuccess && lambda_s)
        for (int i = 0; i < HYPERIM_NSTRATA; ++i) lambda_s[i] = hl[i];
    free_state(s);
    if (e != cudaSuccess) return cuda_fail(e, "greedy end");
    return HYPERIM_OK;
}

hyperim_status greedy_batch(hyperim_graph* g0, const GreedyBatchItem* items, int nitems) {
    if (nitems < 1) return HYPERIM_OK;
    cudaStream_t s = g0->stream;
    hyperim_status st;
    std::vector<GreedyBatchQuery> hq((size_t)nitems);
    int64_t n_cap = 1, inv_cap = 1, cov_cap = 1, kmax = 1;
    for (int i = 0; i < nitems; ++i) {
        const GreedyBatchItem& it = items[i];
        const hyperim_pool *p1 = it.r1, *p2 = it.r2;
        if (p1->count >= (int64_t)0xFFFFFFFFll || p1->total >= (int64_t)0xFFFFFFFFll)
            return set_error(HYPERIM_EOVERFLOW, "more than 2^32 - 1 RR sets or members in a pool");
        uint64_t v1[HYPERIM_NSTRATA], v2[HYPERIM_NSTRATA];
        GreedyBatchQuery& Q = hq[i];
        Q.off1 = p1->rr_off;
        Q.mem1 = p1->rr_mem;
        Q.str1 = p1->rr_stratum;
        Q.j1 = p1->rr_j;
        Q.count1 = p1->count;
        Q.L1 = make_limits(p1, it.lim1, v1);
        Q.off2 = p2->rr_off;
        Q.mem2 = p2->rr_mem;
        Q.str2 = p2->rr_stratum;
        Q.j2 = p2->rr_j;
        Q.count2 = p2->count;
        Q.L2 = make_limits(p2, it.lim2, v2);
        for (int x = 0; x < HYPERIM_NSTRATA; ++x) Q.W.w[x] = stratum_weight(it.g, p1->root_mode, v1[x], x);
        Q.n = it.g->n;
        Q.k = it.k;
        n_cap = std::max<int64_t>(n_cap, it.g->n);
        inv_cap = std::max<int64_t>(inv_cap, p1->total);
        cov_cap = std::max<int64_t>(cov_cap, p1->count);
        kmax = std::max<int64_t>(kmax, it.k);
    }
    n_cap = (n_cap + 3) & ~(int64_t)3;  // per-block score / flag arrays stay 16- and 4-byte aligned
    // one block per SM at most, and no more blocks than the scratch budget allows
    const size_t per_block = 8 * (size_t)n_cap + 4 * ((size_t)n_cap + 1) + (size_t)n_cap + 4 * (size_t)inv_cap +
                             4 * (size_t)cov_cap;
    const size_t budget = (size_t)2 << 30;
    int blocks = (int)std::min<int64_t>(nitems, std::max(1, g0->sm_count));
    blocks = (int)std::max<size_t>(1, std::min<size_t>((size_t)blocks, budget / std::max<size_t>(per_block, 1)));
    CallBuffers tmp(g0);
    GreedyBatchQuery* d_q = nullptr;
    int32_t* d_seeds = nullptr;
    unsigned long long* d_lam = nullptr;
    unsigned int* d_next = nullptr;
    unsigned long long* score = nullptr;
    uint32_t *off = nullptr, *inv = nullptr, *covered = nullptr;
    uint8_t* picked = nullptr;
    if ((st = tmp.alloc(&d_q, sizeof(GreedyBatchQuery) * (size_t)nitems))) return st;
    if ((st = tmp.alloc(&d_seeds, sizeof(int32_t) * (size_t)nitems * (size_t)kmax))) return st;
    if ((st = tmp.alloc(&d_lam, sizeof(unsigned long long) * 2 * HYPERIM_NSTRATA * (size_t)nitems))) return st;
    if ((st = tmp.alloc(&d_next, sizeof(unsigned int)))) return st;
    if ((st = tmp.alloc(&score, sizeof(unsigned long long) * (size_t)n_cap * blocks))) return st;
    if ((st = tmp.alloc(&off, sizeof(uint32_t) * ((size_t)n_cap + 1) * blocks))) return st;
    if ((st = tmp.alloc(&picked, (size_t)n_cap * blocks))) return st;
    if ((st = tmp.alloc(&inv, sizeof(uint32_t) * (size_t)inv_cap * blocks))) return st;
    if ((st = tmp.alloc(&covered, sizeof(uint32_t) * (size_t)cov_cap * blocks))) return st;
    for (int i = 0; i < nitems; ++i) {
        hq[i].seeds = d_seeds + (size_t)i * (size_t)kmax;
        hq[i].lam = d_lam + (size_t)i * 2 * HYPERIM_NSTRATA;
    }
    HYP_CUDA(cudaMemcpyAsync(d_q, hq.data(), sizeof(GreedyBatchQuery) * hq.size(), cudaMemcpyHostToDevice, s));
    HYP_CUDA(cudaMemsetAsync(d_next, 0, sizeof(unsigned int), s));
    GreedyBatchParams B;
    B.q = d_q;
    B.nq = nitems;
    B.next = d_next;
    B.score = score;
    B.off = off;
    B.picked = picked;
    B.inv = inv;
    B.covered = covered;
    B.n_cap = n_cap;
    B.inv_cap = inv_cap;
    B.cov_cap = cov_cap;
    { k_greedy_batch<<<blocks, kGBThreads, 0, s>>>(B); count_launch(); }
    HYP_CUDA(cudaGetLastError());
    std::vector<int32_t> seeds((size_t)nitems * (size_t)kmax);
    std::vector<unsigned long long> lam((size_t)nitems * 2 * HYPERIM_NSTRATA);
    HYP_CUDA(cudaMemcpyAsync(seeds.data(), d_seeds, sizeof(int32_t) * seeds.size(), cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaMemcpyAsync(lam.data(), d_lam, sizeof(unsigned long long) * lam.size(), cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < nitems; ++i) {
        const GreedyBatchItem& it = items[i];
        for (int x = 0; x < it.k; ++x) it.seeds_host[x] = seeds[(size_t)i * (size_t)kmax + x];
        for (int x = 0; x < HYPERIM_NSTRATA; ++x) {
            it.lambda_r1[x] = lam[(size_t)i * 2 * HYPERIM_NSTRATA + x];
            it.lambda_r2[x] = lam[(size_t)i * 2 * HYPERIM_NSTRATA + HYPERIM_NSTRATA + x];
        }
    }
    return check_device_status(g0, "greedy (batch)");
}

}  // namespace hyperim
