// Kernels on finished canonical labels (the label of a site is the smallest
// site of its cluster, end of Section 3):
//  * sequential relabelling: clusters numbered 0..C-1 in the order of their
//    smallest sites (the renumbering the end of Section 3 mentions), plus
//    the size of every cluster;
//  * the spanning test of Section 4: the smallest label found both among the
//    labels of a set of "top" sites and among those of "bottom" sites;
//  * the largest cluster (its size and label).
#pragma once
#include <stdint.h>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "ccl_types.cuh"

namespace ccl {

constexpr int kRelThreads = 256;
constexpr int kRelPerThread = 32;
constexpr int kRelBlock = kRelThreads * kRelPerThread;   // sites per relabel block

// number of roots (label[i] == i) in each block of kRelBlock sites, and a bit
// per site, set for roots. A warp takes 1024 consecutive sites and keeps the 32
// ballots one per lane. The block's words wait in the first places of its own
// part of `out`, which k_root_ids and k_site_ids write afterwards (word t belongs
// to sites from 32 t on, so a short block's words fit too): no scratch for them.
__global__ void __launch_bounds__(kRelThreads) k_root_counts(int32_t n, const int32_t *__restrict__ lab,
                                                             int32_t *__restrict__ block_cnt,
                                                             int32_t *__restrict__ out) {
    __shared__ int s_w[kRelThreads / 32];
    static_assert(kRelPerThread == 32, "one ballot per lane");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kRelBlock + warp * (32 * kRelPerThread) + lane;
    unsigned mine = 0;                  // lane u: the roots among the warp's u-th 32 sites
#pragma unroll 8
    for (int u = 0; u < kRelPerThread; ++u) {
        const int64_t i = base + 32 * u;
        const unsigned b = __ballot_sync(kFull, i < n && __ldg(lab + i) == (int32_t)i);
        if (lane == u) mine = b;
    }
    const int64_t first = (int64_t)blockIdx.x * kRelBlock;
    if (first + 32 * (int)threadIdx.x < n) out[first + threadIdx.x] = (int32_t)mine;
    const int c = __reduce_add_sync(kFull, __popc(mine));
    if (lane == 0) s_w[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kRelThreads / 32; ++w) t += s_w[w];
        block_cnt[blockIdx.x] = t;
    }
}

// exclusive scan of the block counts in place (one CTA); *total = sum
__global__ void __launch_bounds__(1024) k_scan_counts(int32_t nb, int32_t *__restrict__ cnt,
                                                      int32_t *__restrict__ total) {
    __shared__ int32_t s_part[1024];
    const int per = (nb + 1023) / 1024;
    const int b0 = min((int)threadIdx.x * per, nb), b1 = min(b0 + per, nb);
    int32_t part = 0;
    for (int b = b0; b < b1; ++b) part += cnt[b];
    s_part[threadIdx.x] = part;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {         // Hillis-Steele inclusive scan
        const int32_t v = threadIdx.x >= (unsigned)o ? s_part[threadIdx.x - o] : 0;
        __syncthreads();
        s_part[threadIdx.x] += v;
        __syncthreads();
    }
    int32_t acc = s_part[threadIdx.x] - part;
    for (int b = b0; b < b1; ++b) {
        const int32_t c = cnt[b];
        cnt[b] = acc;
        acc += c;
    }
    if (threadIdx.x == 1023) *total = s_part[1023];
}

// sequential id of every root: its block's offset plus the roots before it in
// the block, in site order; zeroes the size counter of each id. The roots come
// from the bits of k_root_counts, not from the labels again, and a warp needs
// the other warps' totals once, so the block meets at one barrier (stepping the
// whole block through 256 sites at a time took 96 barriers).
__global__ void __launch_bounds__(kRelThreads) k_root_ids(int32_t n, const int32_t *__restrict__ block_off,
                                                          int32_t *__restrict__ out, int32_t *__restrict__ sizes) {
    __shared__ int32_t s_w[kRelThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kRelBlock + warp * (32 * kRelPerThread) + lane;
    // (every thread has its word before the barrier below, none writes before it)
    const int64_t first = (int64_t)blockIdx.x * kRelBlock;
    const unsigned mine = first + 32 * (int)threadIdx.x < n ? (unsigned)out[first + threadIdx.x] : 0u;
    int incl = __popc(mine);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    int32_t off = block_off[blockIdx.x];
    for (int w = 0; w < warp; ++w) off += s_w[w];
    const int32_t before = off + incl - __popc(mine);
    for (int u = 0; u < kRelPerThread; ++u) {
        const unsigned b = __shfl_sync(kFull, mine, u);
        const int32_t id = __shfl_sync(kFull, before, u) + __popc(b & ((1u << lane) - 1u));
        if ((b >> lane) & 1u) {
            out[base + 32 * u] = id;
            if (sizes) sizes[id] = 0;
        }
    }
}

// Counts of a warp's values (cluster ids or labels), added to cnt[value] with
// as few atomics as the values allow: lanes with the same value add once, and
// the value that fills the warp (the giant cluster above the threshold) is
// counted in a register until another takes its place. Without the register
// every warp of the GPU adds to the giant cluster's counter, one address:
// a realisation of honeycomb 2896^2 at 1.25 p_c (labelling, spanning, largest
// cluster) took 845 us that way and 448 this way; relabelling triangle 4096^2
// at 0.9 p_c, whose ids and sizes are one pass now, 205 and 110.
// Tracks the largest (count, smallest value) key seen after an add; the keys of a
// lane's own adds are folded in by the caller, several at a time, so that a warp
// does not wait for its atomics one by one (largest cluster of triangle 4096^2 at
// 0.9 p_c 95 -> 87 us, at 1.25 p_c 104 -> 91).
struct Added {                  // the counter before an add, what was added, to which value
    int32_t was, by, at;
};
struct WarpCounter {
    int32_t *cnt;
    int32_t hot = -1;           // warp-uniform
    int held = 0;
    unsigned long long key = 0;

    __device__ __forceinline__ explicit WarpCounter(int32_t *c) : cnt(c) {}
    __device__ __forceinline__ void fold(const Added &a) {
        const unsigned long long k = ((unsigned long long)(unsigned)(a.was + a.by) << 32) | (0xffffffffu - (uint32_t)a.at);
        key = k > key ? k : key;
    }
    // adds one of value v for every lane (v < 0: none); the whole warp calls. Returns
    // the lane's own add.
    __device__ __forceinline__ Added add(int32_t v, int lane) {
        Added mine{0, 0, -1};
        const bool is_hot = v >= 0 && v == hot;
        const int hits = __popc(__ballot_sync(kFull, is_hot));
        held += hits;
        if (is_hot) v = -1;
        if (!__any_sync(kFull, v >= 0)) return mine;
        const unsigned peers = __match_any_sync(kFull, v);
        const bool lead = v >= 0 && __ffs(peers) - 1 == lane;
        const int c = __popc(peers);
        // a value on more lanes than the held one's, and on at least a quarter
        // of the warp, is held instead of it
        const unsigned big = __reduce_max_sync(kFull, lead ? (unsigned)c * 32u + (unsigned)lane : 0u);
        const bool swap = (int)(big >> 5) >= 8 && (int)(big >> 5) > hits;
        const int by = (int)(big & 31u);
        const int32_t next = __shfl_sync(kFull, v, by);
        if (lead && !(swap && lane == by)) mine = Added{atomicAdd(cnt + v, c), c, v};
        if (swap) {
            flush(lane);
            hot = next;
            held = (int)(big >> 5);
        }
        return mine;
    }
    __device__ __forceinline__ void flush(int lane) {
        if (lane == 0 && held > 0) fold(Added{atomicAdd(cnt + hot, held), held, hot});
        held = 0;
    }
};

// Sites [lo, hi) of this warp when n sites are cut into runs of whole 128-site
// groups, one run per warp of the grid (consecutive sites share clusters, so a
// run keeps its held value).
__device__ __forceinline__ void warp_run(int64_t n, int64_t &lo, int64_t &hi) {
    const int64_t groups = (n + 127) / 128, warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t per = (groups + warps - 1) / warps;
    const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    lo = min(w * per * 128, n);
    hi = min((w + 1) * per * 128, n);
}

// every other site takes its root's id; with sizes, every site is counted
// under its id in the same pass
__global__ void __launch_bounds__(256) k_site_ids(int32_t n, const int32_t *__restrict__ lab, int32_t *out,
                                                  int32_t *__restrict__ sizes) {
    const int lane = threadIdx.x & 31;
    int64_t lo, hi;
    warp_run(n, lo, hi);
    WarpCounter wc(sizes);
    for (int64_t g = lo; g < hi; g += 128) {
        int32_t l[4], id[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = g + 32 * u + lane;
            l[u] = i < hi ? __ldg(lab + i) : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) id[u] = l[u] >= 0 ? out[l[u]] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = g + 32 * u + lane;
            if (l[u] >= 0 && l[u] != (int32_t)i) out[i] = id[u];
        }
        if (sizes)
#pragma unroll
            for (int u = 0; u < 4; ++u) wc.add((uint32_t)id[u] < (uint32_t)n ? id[u] : -1, lane);
    }
    if (sizes) wc.flush(lane);
}

// spanning: mark the labels of the top sites, then look for them at the bottom
__global__ void k_span_mark(int32_t n, const int32_t *__restrict__ lab, const int32_t *__restrict__ top,
                            int32_t n_top, uint32_t *__restrict__ flags, int32_t *__restrict__ best,
                            unsigned *err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_top; t += stride) {
        const int32_t s = top[t];
        if ((uint32_t)s >= (uint32_t)n) { atomicOr(err, kErrIndex); continue; }
        const int32_t l = lab[s];
        if ((uint32_t)l >= (uint32_t)n) { atomicOr(err, kErrIndex); continue; }
        atomicOr(flags + (l >> 5), 1u << (l & 31));
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *best = -1;     // none (the largest as unsigned)
}

__global__ void k_span_check(int32_t n, const int32_t *__restrict__ lab, const int32_t *__restrict__ bottom,
                             int32_t n_bottom, const uint32_t *__restrict__ flags, int32_t *__restrict__ best,
                             unsigned *err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_bottom; t += stride) {
        const int32_t s = bottom[t];
        if ((uint32_t)s >= (uint32_t)n) { atomicOr(err, kErrIndex); continue; }
        const int32_t l = lab[s];
        if ((uint32_t)l >= (uint32_t)n) { atomicOr(err, kErrIndex); continue; }
        if ((__ldg(flags + (l >> 5)) >> (l & 31)) & 1u) atomicMin((unsigned *)best, (unsigned)l);
    }
}

// The spanning test of few sites in one launch of one cluster: every CTA keeps all
// top labels in a hash set in its shared memory (open addressing, at most a
// quarter full: the slowest lane of a warp decides) and looks its share of the
// bottom labels up. Clearing a bit per site, marking, checking and finishing took
// four launches. An SM loads scattered labels at 1 ns a site, so the loads are split
// over the CTAs, and the top labels are then read from each other's shared memory.
// Four launches / this, 4096 + 4096 and 8192 + 12,288 scattered sites of 16.8M: 17 / 13
// and 17 / 17 us, 2 x 5792 in rows 17 / 11 (one CTA: 17, 35 and 11). The line lies
// at 16,384 bottom sites: 8192 + 65,536 scattered ones 17 / 21.
constexpr int kSpanTop = 8192;              // most top sites of this path
constexpr int kSpanBottom = 16384;          // most bottom sites
constexpr int kSpanSpread = 4;              // slots per top site, at least
constexpr int kSpanThreads = 1024;
constexpr int kSpanCtas = kSpanTop / kSpanThreads;      // (a top site per thread)
__global__ void __cluster_dims__(kSpanCtas, 1, 1) __launch_bounds__(kSpanThreads)
    k_span_few(int32_t n, const int32_t *__restrict__ lab, const int32_t *__restrict__ top, int32_t n_top,
               const int32_t *__restrict__ bottom, int32_t n_bottom, int32_t slots, int32_t *__restrict__ best,
               unsigned *err) {
    extern __shared__ __align__(16) int32_t s_set[];    // `slots`, a power of two, -1 where empty
    __shared__ int32_t s_top[kSpanThreads]; // the labels of the CTA's top sites
    __shared__ unsigned s_best;             // (the first CTA's is used)
    const auto cluster = cooperative_groups::this_cluster();
    const int first = (int)cluster.block_rank() * kSpanThreads + (int)threadIdx.x;
    const auto label = [&](const int32_t *__restrict__ sites, int t) {
        const int32_t s = sites[t];
        const int32_t l = (uint32_t)s < (uint32_t)n ? lab[s] : -1;
        if ((uint32_t)l < (uint32_t)n) return l;
        atomicOr(err, kErrIndex);
        return -1;
    };
    s_top[threadIdx.x] = first < n_top ? label(top, first) : -1;
    for (int t = threadIdx.x; t < slots / 4; t += kSpanThreads)
        reinterpret_cast<int4 *>(s_set)[t] = make_int4(-1, -1, -1, -1);
    if (threadIdx.x == 0) s_best = 0xffffffffu;         // -1: no cluster spans
    cluster.sync();
    const unsigned mask = (unsigned)slots - 1u;
    int32_t l[kSpanCtas];
#pragma unroll
    for (int c = 0; c < kSpanCtas; ++c)
        l[c] = c * kSpanThreads < n_top ? cluster.map_shared_rank(s_top, c)[threadIdx.x] : -1;
#pragma unroll
    for (int c = 0; c < kSpanCtas; ++c) {
        if (l[c] < 0) continue;
        unsigned h = ((unsigned)l[c] * 2654435761u >> 16) & mask;
        for (int probe = 0; probe < slots; ++probe, h = (h + 1u) & mask) {
            const int32_t was = atomicCAS(&s_set[h], -1, l[c]);
            if (was == -1 || was == l[c]) break;
        }
    }
    __syncthreads();
    unsigned mine = 0xffffffffu;
    for (int t = first; t < n_bottom; t += kSpanCtas * kSpanThreads) {
        const int32_t b = label(bottom, t);
        if (b < 0 || (unsigned)b >= mine) continue;
        unsigned h = ((unsigned)b * 2654435761u >> 16) & mask;
        for (int probe = 0; probe < slots && s_set[h] != -1; ++probe, h = (h + 1u) & mask)
            if (s_set[h] == b) { mine = (unsigned)b; break; }
    }
    mine = __reduce_min_sync(kFull, mine);
    if ((threadIdx.x & 31) == 0 && mine != 0xffffffffu) atomicMin(cluster.map_shared_rank(&s_best, 0), mine);
    cluster.sync();                         // (also: no CTA leaves while another reads its labels)
    if (first == 0) *best = (int32_t)s_best;
}

// Largest cluster (Section 4's largest-cluster statistic): cnt[l] = sites
// whose canonical label is l. Every add returns the count so far, and the last
// add of a label its size, so the largest (size, smallest label) key over all
// adds is the answer: no pass over the counters. The last CTA to finish
// writes the result. (scratch: the best key, the finished CTAs.)
struct LargestScratch {
    unsigned long long best;
    unsigned done, pad_;
};
constexpr int kLargestCtas = 6;     // per SM
__global__ void __launch_bounds__(256, kLargestCtas) k_largest(int32_t n, const int32_t *__restrict__ lab, int32_t *__restrict__ cnt,
                                                 LargestScratch *scratch, int32_t *__restrict__ result, unsigned *err) {
    const int lane = threadIdx.x & 31;
    int64_t lo, hi;
    warp_run(n, lo, hi);
    WarpCounter wc(cnt);
    bool bad = false;
    for (int64_t g = lo; g < hi; g += 128) {
        int32_t l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = g + 32 * u + lane;
            l[u] = i < hi ? __ldg(lab + i) : -1;
            bad |= i < hi && (uint32_t)l[u] >= (uint32_t)n;
        }
        Added mine[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) mine[u] = wc.add((uint32_t)l[u] < (uint32_t)n ? l[u] : -1, lane);
#pragma unroll
        for (int u = 0; u < 4; ++u) wc.fold(mine[u]);
    }
    wc.flush(lane);
    if (bad) atomicOr(err, kErrIndex);
    unsigned long long key = wc.key;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(kFull, key, o);
        key = t > key ? t : key;
    }
    if (lane == 0 && key > *(volatile unsigned long long *)&scratch->best) atomicMax(&scratch->best, key);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&scratch->done, 1u) == gridDim.x - 1) {
        __threadfence();
        const unsigned long long k = atomicMax(&scratch->best, 0ull);
        result[0] = (int32_t)(k >> 32);
        result[1] = k ? (int32_t)(0xffffffffu - (uint32_t)(k & 0xffffffffu)) : -1;
    }
}

}  // namespace ccl
