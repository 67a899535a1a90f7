// Chunk index of large neighbourhoods (a lookup structure over the layers of Sec. 3.1.1).
//
// A pick of Algorithm 3 is "the a-th member of layer L_i of A(mu) in id order". For a vertex
// whose hyperedges hold thousands of members, materialising all of A(mu) to find a handful of
// picks is most of the RR kernel's work. The index splits the id space into C = 2^c chunks (top
// c id bits) and stores, per layer and chunk, how many members of the layer lie in the earlier
// chunks. A pick's position then names its chunk, and the RR kernel reads only that id range of
// mu's hyperedges (each hyperedge's members are sorted, so the range is found by binary search).
// The index holds counts only (l x C words per indexed vertex), never neighbour lists.
//
// Build (after the layer profile):
//   k_idx_candidates  vertices with d_H >= 2, more than kIdxMinT members besides mu, l <= kIdxMaxL
//   k_idx_plan        per candidate: the expected picks per pop decide the chunk target (or
//                     no index); c = the fewest bits for which no chunk holds more than the target
//                     (0 bits: not indexed), found by the layer profile on its sorted members (a pass
//                     over the members of its own took 8.7 ms of a 2M-vertex load); entries = l 2^c
//   scan              table offsets
//   k_idx_fill        per indexed vertex: members sorted by id on chip (bucketed through a global
//                     scratch area when large), runs (multiplicity w -> layer) counted per
//                     (layer, chunk); each layer row becomes an exclusive prefix
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "mat.cuh"

namespace hyperim {
namespace {

constexpr int kBins = 1 << kIdxMaxBits;

__device__ __forceinline__ void dev_fail(DevStatus* st, int32_t code, int32_t detail) {
    if (atomicCAS(&st->code, 0, code) == 0) st->detail = detail;
}

__global__ void k_idx_candidates(int32_t n, const int4* __restrict__ vinfo, const int32_t* __restrict__ tsum,
                                 uint32_t* __restrict__ flag) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int4 vi = vinfo[v];
        const int T = tsum[v] - vi.w;
        flag[v] = (vi.w >= 2 && T > kIdxMinT && vi.y >= 1 && vi.y <= kIdxMaxL) ? 1u : 0u;
    }
}

__global__ void k_idx_list(int32_t n, const uint32_t* __restrict__ flag, const int64_t* __restrict__ pos,
                           int32_t* __restrict__ list) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        if (flag[v]) list[pos[v]] = (int32_t)v;
}

// exclusive scan of a[0, count) in place by warp 0 (count <= kBins); returns nothing, callers sync
__device__ void warp0_exclusive_scan(int* a, int count) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    int carry = 0;
    for (int base = 0; base < count; base += 32) {
        const int i = base + lane;
        const int v = i < count ? a[i] : 0;
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += t;
        }
        if (i < count) a[i] = carry + inc - v;
        carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
}

__global__ void k_idx_plan(const int32_t* __restrict__ list, int32_t nlist, const int4* __restrict__ vinfo,
                           const int32_t* __restrict__ tsum, const uint4* __restrict__ prof,
                           const uint8_t* __restrict__ chunk_bits, uint8_t* __restrict__ bits_out,
                           uint32_t* __restrict__ entries) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlist; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t mu = list[i];
        const int4 vi = vinfo[mu];
        // expected picks per pop, sum_i n_i p_i, against kIdxFewPicks on the integers
        // n_i floor(p_i 2^32) (p = 1 counts 2^32), stopping once the bound is reached
        const unsigned long long cap = kIdxFewPicks << 32;
        unsigned long long acc = 0;
        for (int q = 0; q < vi.y && acc < cap; ++q) {
            const uint4 e = prof[2 * ((int64_t)vi.x + q)];
            const unsigned long long t = (e.x & kPOneFlag) ? (1ull << 32) : (unsigned long long)e.z;
            acc += (unsigned long long)e.y * t;
        }
        const int both = chunk_bits[mu];
        // many picks on a neighbourhood one warp sorts whole: no index
        const int best = acc < cap ? both & 15 : tsum[mu] - vi.w > kIdxMinTMany ? both >> 4 : 0;
        bits_out[i] = (uint8_t)best;
        entries[i] = best ? (uint32_t)vi.y << best : 0u;
    }
}

__global__ void k_idx_word(const int32_t* __restrict__ list, int32_t nlist, const uint8_t* __restrict__ bits,
                           const uint32_t* __restrict__ entries, const int64_t* __restrict__ off,
                           uint64_t* __restrict__ idx) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlist;
         i += (int64_t)gridDim.x * blockDim.x)
        if (entries[i]) idx[list[i]] = ((uint64_t)bits[i] << kIdxBitsShift) | (uint64_t)off[i];
}

// Per indexed vertex (one block, vertices taken from a shared counter): the members of mu's
// hyperedges in ascending id order -- sorted whole on chip when at most kFillBuf of them, else
// bucketed by their top id bits (a bucket is 2^3 whole index chunks, so at most 8 x 1,024
// members) through a global scratch area and sorted bucket by bucket -- are walked run by run:
// each distinct neighbour (multiplicity w -> layer by search in the descending w list) adds one
// to its count of (layer, chunk, eighth of the chunk). The counts are 16-bit halves of on-chip
// words, as many chunks at a time as fit kFillCells of them (all of a small vertex's chunks, one
// bucket's eight of a large one's): no count ever goes to global memory. They then become the
// entries of those chunks, lanes side by side along the chunks of a layer, with one running total per
// layer carried on.
constexpr int kFillThreads = 512;  // two blocks (32 warps) per SM: the sorts are latency-bound
constexpr int kFillBuf = 8192;  // members sorted on chip at once (power of two)
constexpr int kFillCnt = 4096;  // words of two counts each
constexpr int kFillCells = 2 * kFillCnt;
static_assert(kFillCells >= kIdxMaxL << kIdxSubBits, "one chunk of the most layers must fit");
static_assert(2 * kFillThreads + 1 >= kIdxMaxL, "the prefix area holds the layers' running totals");
constexpr int kFillBkt = kBins;
constexpr int kFillTop = 1 << (kIdxMaxBits - 3);  // top-bit buckets: eight whole chunks each
// the shared memory above fits three 512-thread blocks per SM
constexpr int kFillCtrl = 64;
constexpr size_t kFillSmem = sizeof(uint32_t) * (kFillBuf + kFillCnt + kIdxMaxL) +
                             sizeof(int) * (kFillBkt + kFillTop + 2 * kFillThreads + 1 + kFillCtrl);

__global__ void __launch_bounds__(kFillThreads)
k_idx_fill(const int32_t* __restrict__ list, int32_t nlist, const uint8_t* __restrict__ bits_in,
           const uint32_t* __restrict__ entries, const int64_t* __restrict__ off,
           const int4* __restrict__ vinfo, const int2* __restrict__ v_span,
           const int32_t* __restrict__ he_mem, const int32_t* __restrict__ tsum,
           const uint4* __restrict__ prof, int id_bits, uint32_t* __restrict__ tab, uint4* __restrict__ sub,
           uint32_t* __restrict__ scratch, int64_t scratch_cap, const int32_t* __restrict__ order,
           int* __restrict__ next, DevStatus* st) {
    extern __shared__ __align__(16) unsigned char fill_smem[];
    uint32_t* buf = reinterpret_cast<uint32_t*>(fill_smem);             // kFillBuf
    uint32_t* cnt_s = buf + kFillBuf;                                   // kFillCnt
    uint32_t* lw = cnt_s + kFillCnt;                                    // kIdxMaxL
    int* bkt = reinterpret_cast<int*>(lw + kIdxMaxL);                   // kFillBkt (on-chip sorts)
    int* bucket_end = bkt + kFillBkt;                                   // kFillBkt (top-bit buckets)
    int* pre = bucket_end + kFillTop;                                   // 2 kFillThreads + 1
    int* ctrl = pre + 2 * kFillThreads + 1;  // kFillCtrl: [0] ticket, [8, 8 + warps) maxima, [32, 48) sort scratch
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kFillThreads / 32;
    uint32_t* big = scratch + (int64_t)blockIdx.x * scratch_cap;
    for (;;) {
        if (threadIdx.x == 0) ctrl[0] = atomicAdd(next, 1);
        __syncthreads();
        const int ticket = ctrl[0];
        __syncthreads();
        if (ticket >= nlist) break;
        const int i = order[ticket];  // largest first
        if (entries[i] == 0) continue;
        const int32_t mu = list[i];
        const int4 vi = vinfo[mu];
        const int l = vi.y, c = bits_in[i];
        const int C = 1 << c, shift = id_bits - c;
        const int T = tsum[mu] - vi.w;
        uint32_t* t = tab + off[i];
        uint4* ts = sub ? sub + off[i] : nullptr;
        uint32_t* carry = reinterpret_cast<uint32_t*>(pre);  // per layer (pre is free between gathers)
        const int fb = idx_sub_bits(shift), fshift = shift - fb;
        int gch = C;  // chunks counted at once
        while (gch > 1 && ((int64_t)l * gch << kIdxSubBits) > kFillCells) gch >>= 1;
        for (int q = threadIdx.x; q < l; q += kFillThreads) lw[q] = prof[2 * ((int64_t)vi.x + q)].x & ~kPOneFlag;
        __syncthreads();
        // Entries of the chunks [k0, k0 + nk) from the sorted keys[0, got), their members. A group of gch chunks
        // walks its own keys, and groups without any get their entries at once: members crowded into few ids
        // make few of very many chunks busy. (678 vertices of up to 120 layers, 2^11 chunks, 76M entries: load
        // 13.9 ms when every group walked all keys, 3.1 so, 2.7 before there were eighths to write.)
        auto count_and_emit = [&](const uint32_t* keys, int got, int k0, int nk) {
            int from = 0;  // keys of the groups so far
            for (int kb = k0; kb < k0 + nk; kb += gch) {
                // groups without a key: every layer's running total, no member in any eighth
                const int kn = from < got ? (int)(keys[from] >> shift) & -gch : k0 + nk;
                if (kb < kn) {
                    for (int q = wid; q < l; q += kWarps)
                        for (int k = kb + lane; k < kn; k += 32) {
                            t[(int64_t)q * C + k] = carry[q];
                            if (ts) ts[(int64_t)q * C + k] = make_uint4(0, 0, 0, 0);
                        }
                    kb = kn;
                    if (kb >= k0 + nk) break;
                }
                const int g = min(gch, k0 + nk - kb);  // a power of two
                int to = got;
                if (kb + g < k0 + nk) {  // the first key of the next group
                    const uint32_t next_id = (uint32_t)(kb + g) << shift;
                    for (int lo = from; lo < to;) {
                        const int mid = (lo + to) >> 1;
                        if (keys[mid] < next_id) lo = mid + 1; else to = mid;
                    }
                }
                const int words = (l * g) << (kIdxSubBits - 1);
                for (int x = threadIdx.x; x < words; x += kFillThreads) cnt_s[x] = 0;
                __syncthreads();
                walk_runs<kFillThreads>(keys + from, to - from, [&](bool start, uint32_t x, int mult) -> bool {
                    if (start) {
                        const int k = (int)(x >> shift) - kb;
                        int lo = 0, hi = l;  // lw descends: first q with lw[q] <= mult
                        while (lo < hi) {
                            const int mid = (lo + hi) >> 1;
                            if (lw[mid] > (uint32_t)mult) lo = mid + 1; else hi = mid;
                        }
                        if (lo < l && lw[lo] == (uint32_t)mult) {
                            const int cell = ((lo * g + k) << kIdxSubBits) + (int)((x >> fshift) & ((1u << fb) - 1));
                            atomicAdd(&cnt_s[cell >> 1], 1u << (16 * (cell & 1)));
                        } else {
                            dev_fail(st, kErrProfile, mu);
                        }
                    }
                    return false;
                });
                from = to;
                __syncthreads();
                const int gw = min(g, 32), rows = 32 / gw;  // layers side by side in a warp
                for (int q0 = wid * rows; q0 < l; q0 += kWarps * rows) {
                    const int q = q0 + lane / gw;
                    uint32_t run = q < l ? carry[q] : 0u;
                    for (int kk = lane % gw; kk < g; kk += 32) {  // gw < 32: one step
                        uint4 w = make_uint4(0, 0, 0, 0);
                        if (q < l) w = reinterpret_cast<const uint4*>(cnt_s)[q * g + kk];
                        const uint32_t v[8] = {w.x & 0xFFFFu, w.x >> 16, w.y & 0xFFFFu, w.y >> 16,
                                               w.z & 0xFFFFu, w.z >> 16, w.w & 0xFFFFu, w.w >> 16};
                        uint32_t e[8], sum = 0;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            e[u] = sum;
                            sum += v[u];
                        }
                        uint32_t inc = sum;  // along the chunks of this layer
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                            if (o < gw && lane % gw >= o) inc += x;
                        }
                        if (q < l) {
                            const int64_t at = (int64_t)q * C + kb + kk;
                            t[at] = run + inc - sum;
                            if (ts)
                                ts[at] = make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16,
                                                    e[6] | e[7] << 16);
                        }
                        run += __shfl_sync(0xFFFFFFFFu, inc, lane | (gw - 1));
                    }
                    if (q < l && lane % gw == 0) carry[q] = run;
                }
                __syncthreads();
            }
        };
        if (T <= kFillBuf) {
            const int got = sorted_nbhd<kFillThreads>(v_span, he_mem, mu, vi.z, vi.w, T, id_bits, buf, bkt, 12,
                                                      pre, ctrl + 32);
            for (int q = threadIdx.x; q < l; q += kFillThreads) carry[q] = 0;
            __syncthreads();
            count_and_emit(buf, got, 0, C);
        } else {
            if ((int64_t)T > scratch_cap) {
                if (threadIdx.x == 0) dev_fail(st, kErrCapacity, mu);
                __syncthreads();
                continue;
            }
            const int b = c > 3 ? c - 3 : 0;
            const int nb = 1 << b, bshift = id_bits - b;
            for (int q = threadIdx.x; q < nb; q += kFillThreads) bucket_end[q] = 0;
            __syncthreads();
            for_each_member<kFillThreads>(v_span, he_mem, mu, vi.z, vi.w, pre,
                                          [&](uint32_t x) { atomicAdd(&bucket_end[x >> bshift], 1); });
            __syncthreads();
            int mx = 0;
            for (int q = threadIdx.x; q < nb; q += kFillThreads) mx = max(mx, bucket_end[q]);
            mx = __reduce_max_sync(0xFFFFFFFFu, mx);
            if (lane == 0) ctrl[8 + wid] = mx;
            __syncthreads();
            int all = 0;
            for (int w = 0; w < kWarps; ++w) all = max(all, ctrl[8 + w]);
            if (all > kFillBuf) {  // uniform; the plan's chunk bound rules this out
                if (threadIdx.x == 0) dev_fail(st, kErrBucket, mu);
                __syncthreads();
                continue;
            }
            warp0_exclusive_scan(bucket_end, nb);
            __syncthreads();
            for_each_member<kFillThreads>(v_span, he_mem, mu, vi.z, vi.w, pre,
                                          [&](uint32_t x) { big[atomicAdd(&bucket_end[x >> bshift], 1)] = x; });
            __threadfence_block();
            __syncthreads();
            // bucket_end[q] is now the end of bucket q
            for (int q = threadIdx.x; q < l; q += kFillThreads) carry[q] = 0;
            __syncthreads();
            int begin = 0;
            for (int q = 0; q < nb; ++q) {
                const int end = bucket_end[q];
                if (end > begin) {
                    sort_chunk<kFillThreads>(big + begin, end - begin, bshift, buf, bkt, 12, ctrl + 32);
                }
                count_and_emit(buf, end - begin, q << (c - b), 1 << (c - b));
                begin = end;
            }
        }
        __syncthreads();
    }
}

int grid_for(int64_t items, int threads, int sm) {
    int64_t b = (items + threads - 1) / threads;
    int64_t cap = (int64_t)sm * 32;
    if (b < 1) b = 1;
    return (int)(b < cap ? b : cap);
}

}  // namespace

hyperim_status build_chunk_index(hyperim_graph* g, const uint8_t* chunk_bits) {
    cudaStream_t s = g->stream;
    const int32_t n = g->n;
    const int sm = g->sm_count;
    hyperim_status st;
    CallBuffers tmp(g);
    if ((st = dev_alloc(g, (void**)&g->idx, sizeof(uint64_t) * (size_t)(n > 0 ? n : 1)))) return st;
    HYP_CUDA(cudaMemsetAsync(g->idx, 0, sizeof(uint64_t) * (size_t)(n > 0 ? n : 1), s));
    g->idx_entries = 0;
    g->idx_vertices = 0;
    if (n == 0 || g->max_tsum <= kIdxMinT) return HYPERIM_OK;

    uint32_t* d_flag = nullptr;
    int64_t* d_pos = nullptr;
    if ((st = tmp.alloc(&d_flag, sizeof(uint32_t) * (size_t)n))) return st;
    if ((st = tmp.alloc(&d_pos, sizeof(int64_t) * ((size_t)n + 1)))) return st;
    { k_idx_candidates<<<grid_for(n, 256, sm), 256, 0, s>>>(n, g->vinfo, g->tsum, d_flag); count_launch(); }
    if ((st = exclusive_scan_u32_to_i64(g, d_flag, d_pos, n))) return st;
    int64_t ncand = 0;
    HYP_CUDA(cudaMemcpyAsync(&ncand, d_pos + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaStreamSynchronize(s));
    if (ncand == 0) return HYPERIM_OK;
    int32_t* d_list = nullptr;
    uint8_t* d_bits = nullptr;
    uint32_t* d_entries = nullptr;
    int64_t* d_off = nullptr;
    if ((st = tmp.alloc(&d_list, sizeof(int32_t) * (size_t)ncand))) return st;
    if ((st = tmp.alloc(&d_bits, (size_t)ncand))) return st;
    if ((st = tmp.alloc(&d_entries, sizeof(uint32_t) * (size_t)ncand))) return st;
    if ((st = tmp.alloc(&d_off, sizeof(int64_t) * ((size_t)ncand + 1)))) return st;
    { k_idx_list<<<grid_for(n, 256, sm), 256, 0, s>>>(n, d_flag, d_pos, d_list); count_launch(); }
    const int nl = (int)ncand;
    // the candidates' indices, largest neighbourhood first (the fill takes them in this order)
    int32_t* d_order = nullptr;
    int* d_next = nullptr;
    if ((st = tmp.alloc(&d_order, sizeof(int32_t) * (size_t)ncand))) return st;
    if ((st = tmp.alloc(&d_next, sizeof(int)))) return st;
    if ((st = size_order(g, d_list, ncand, true, d_order))) return st;
    { k_idx_plan<<<grid_for(ncand, 256, sm), 256, 0, s>>>(d_list, nl, g->vinfo, g->tsum, g->prof, chunk_bits, d_bits,
                                                        d_entries); count_launch(); }
    if ((st = exclusive_scan_u32_to_i64(g, d_entries, d_off, ncand))) return st;
    int64_t total = 0;
    HYP_CUDA(cudaMemcpyAsync(&total, d_off + ncand, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    HYP_CUDA(cudaStreamSynchronize(s));
    if (total >= ((int64_t)1 << kIdxBitsShift)) return set_error(HYPERIM_EOVERFLOW, "chunk index too large");
    g->idx_entries = total;
    if (total > 0) {
        if ((st = dev_alloc(g, (void**)&g->idx_tab, sizeof(uint32_t) * (size_t)total))) return st;
        { k_idx_word<<<grid_for(ncand, 256, sm), 256, 0, s>>>(d_list, nl, d_bits, d_entries, d_off, g->idx); count_launch(); }
        // per resident block, room for the largest neighbourhood
        HYP_CUDA(cudaFuncSetAttribute(k_idx_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFillSmem));
        int per_sm = 0;
        HYP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_idx_fill, kFillThreads, kFillSmem));
        if (per_sm < 1) per_sm = 1;
        const int64_t cap = g->max_tsum;
        int fblocks = (int)std::min<int64_t>(ncand, (int64_t)sm * per_sm);
        // keep the scratch area within 2 GiB
        while (fblocks > sm && (int64_t)fblocks * cap * 4 > ((int64_t)2 << 30)) fblocks -= sm;
        uint32_t* d_scratch = nullptr;
        if ((st = tmp.alloc(&d_scratch, sizeof(uint32_t) * (size_t)cap * fblocks))) return st;
        // the eighths, if there is room
        if (takes_optional(g) && dev_try_alloc(g, (void**)&g->idx_sub, sizeof(uint4) * (size_t)total) == HYPERIM_OK)
            g->optional_bytes += sizeof(uint4) * (size_t)total;
        HYP_CUDA(cudaMemsetAsync(d_next, 0, sizeof(int), s));
        { k_idx_fill<<<fblocks, kFillThreads, kFillSmem, s>>>(d_list, nl, d_bits, d_entries, d_off, g->vinfo, g->v_span,
                                                  g->he_mem, g->tsum, g->prof, g->id_bits, g->idx_tab, g->idx_sub, d_scratch,
                                                  cap, d_order, d_next, g->d_status); count_launch(); }
        if ((st = check_device_status(g, "chunk index"))) return st;
        // indexed vertices
        std::vector<uint32_t> e((size_t)ncand);
        HYP_CUDA(cudaMemcpyAsync(e.data(), d_entries, sizeof(uint32_t) * (size_t)ncand, cudaMemcpyDeviceToHost, s));
        HYP_CUDA(cudaStreamSynchronize(s));
        int32_t cnt = 0;
        for (uint32_t x : e) cnt += x ? 1 : 0;
        g->idx_vertices = cnt;
    }
    HYP_CUDA(cudaGetLastError());
    return HYPERIM_OK;
}

}  // namespace hyperim
