// Step (i) on the dense strided nearest-neighbour list of Section 3: the list
// has W = (largest number of neighbours of any site) slots per site, and
// neighbour slot k of site i is nn[i + k*N]. A slot holding -1 is empty (the
// site has fewer than W neighbours); every other slot must hold a site in
// [0, N). Slot e = i + k*N has its open bit at bit e of the bit words (word
// e >> 5, bit e & 31), or draws it on the device like the CSR path.
//
// As in the CSR kernel, only the slots of row i with j < i are read (the bond
// {i, j} is decided in the row of its larger site), label[i] becomes the
// smallest open lower neighbour (or i), and the others are appended to the
// residual queue as pairs (i, j). The queue has the CSR path's band layout:
// CTA b owns the slots [N_b * W, N_b' * W) of its sites [N_b, N_b'), packs its
// pairs from the start of that range and records their count in band[b], so
// steps (ii)-(iv) run unchanged.
//
// Two kernels: lists of at most kRowRegs slots go through shared memory
// (k_init_dense_tma below), wider ones are read in place (k_init_dense): for one k
// the 32 lanes of a warp (32 consecutive sites) read 32 consecutive ints of nn and
// at most two bit words, so every load is a coalesced 128-byte line.
#pragma once
#include <stdint.h>
#include <cuda_runtime.h>

#include "ccl_device.cuh"

namespace ccl {

#ifndef CCL_DENSE_THREADS
#define CCL_DENSE_THREADS 256
#endif
#ifndef CCL_DENSE_CHUNKS
#define CCL_DENSE_CHUNKS 2
#endif
constexpr int kDenseThreads = CCL_DENSE_THREADS;
constexpr int kDenseChunks = CCL_DENSE_CHUNKS;               // chunks a warp scans at once
constexpr int kDenseSpan = kDenseThreads * kDenseChunks;     // sites per CTA step

template <bool kGen>
__device__ __forceinline__ bool dense_open(const Params &P, int64_t e, int32_t i, int32_t j) {
    if (kGen) return gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j, (uint32_t)i);
    return (__ldg(P.one.bits + (e >> 5)) >> (e & 31)) & 1u;
}

// Label of site i with smallest open lower neighbour m (cnt of them): the
// sites of this CTA's band before the current step [vis_lo, vis_hi) hold
// their step-(i) labels and are visible after the step barrier, so a site
// whose m lies there takes label[m] (an ancestor of m) instead of m.
__device__ __forceinline__ int32_t dense_label(const Params &P, int32_t i, int32_t m, int32_t cnt,
                                               int64_t vis_lo, int64_t vis_hi) {
    if (!cnt) return i;
    if (m >= vis_lo && m < vis_hi) return __ldcg(P.one.labels + m);
    return m;
}

// Appends the warp's residual pairs (r of them at this lane) to the band's
// part of the queue: returns this lane's first slot.
__device__ __forceinline__ int64_t dense_emit_slot(int64_t qband, unsigned long long *band_cnt, int lane,
                                                   int r) {
    const int incl = warp_incl_scan(r, lane);
    const int total = __shfl_sync(kFull, incl, 31);
    unsigned long long base = 0;
    if (total) {
        if (lane == 0) base = atomicAdd(band_cnt, (unsigned long long)total);
        base = __shfl_sync(kFull, base, 0);
    }
    return qband + (int64_t)base + (incl - r);
}

template <bool kGen>
__global__ void __launch_bounds__(kDenseThreads) k_init_dense(Params P) {
    __shared__ unsigned long long band_cnt;
    int64_t band_lo, band_hi;
    cta_band(P, band_lo, band_hi);
    const int64_t n = P.one.n;
    const int W = (int)P.nn_width;
    const int64_t s_lo = min(band_lo * kTileSites, n), s_hi = min(band_hi * kTileSites, n);
    const int64_t qband = s_lo * W;
    if (threadIdx.x == 0) {
        band_cnt = 0;
        P.band[P.band_off + blockIdx.x].qbase = qband;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    bool bad = false;
    for (int64_t t0 = s_lo; t0 < s_hi; t0 += kDenseSpan) {
        for (int c = 0; c < kDenseChunks; ++c) {
            const int64_t c0 = t0 + (int64_t)(warp * kDenseChunks + c) * kChunk;
            if (c0 >= s_hi) break;
            const int64_t i64 = c0 + lane;
            const bool live = i64 < s_hi;
            const int32_t i = (int32_t)i64;
            int32_t m = INT32_MAX, mk = -1, cnt = 0;
            if (live) {
                for (int k = 0; k < W; ++k) {
                    const int64_t e = i64 + (int64_t)k * n;
                    const int32_t j = __ldg(P.nn + e);
                    bad |= j < -1 || (int64_t)j >= n;
                    if (j >= 0 && j < i && dense_open<kGen>(P, e, i, j)) {
                        ++cnt;
                        if (j < m) { m = j; mk = k; }
                    }
                }
                P.one.labels[i] = dense_label(P, i, m, cnt, s_lo, t0);
            }
            const int r = cnt > 1 ? cnt - 1 : 0;
            int64_t slot = dense_emit_slot(qband, &band_cnt, lane, r);
            if (r > 0) {
                for (int k = 0; k < W; ++k) {
                    const int64_t e = i64 + (int64_t)k * n;
                    const int32_t j = __ldg(P.nn + e);
                    if (k != mk && j >= 0 && j < i && dense_open<kGen>(P, e, i, j)) P.q[slot++] = make_int2(i, j);
                }
            }
        }
        __syncthreads();        // this step's labels become visible to the CTA's next steps
    }
    if (bad) raise_err(P.err, kErrIndex);
    if (threadIdx.x == 0) P.band[P.band_off + blockIdx.x].cnt = band_cnt;      // (after the last step's barrier)
}

// ---------------------------------------------------------------------------
// Dense list through the step-(i) pipeline of k_init: for lists of at most
// kRowRegs slots, a producer lane streams each 1024-site tile's W slot slabs
// (slot k: the tile's sites' entries nn[s0 + k*N ...], contiguous) and their
// bit words into a 3-stage shared-memory ring with bulk asynchronous copies;
// eight consumer warps scan four 32-site chunks each (k_init's scan on slots),
// store the labels after all are scanned and append the residual pairs of all
// through one prefix sum. As in k_init the scan's instructions bound it:
// against sixteen warps of two chunks, step (i) of the cubic lattice 200^3 (8M
// sites, six slots) went from 105 to 89 us, and to 66 with the producer's work
// spread over its lanes (below).

constexpr int kDenseSlab = kTileSites + 8;        // a slot's slab, + 16-byte rounding
constexpr int kDenseWords = kTileSites / 32 + 8;  // its bit words, + rounding

struct __align__(16) DenseStageHdr {
    int2 off[kRowRegs];        // staged tiles: slab[k] index and bw[k] bit index of site s0
    int64_t nn_lo[kRowRegs];   // element of nn held at slab[k][0]
    int64_t w_lo[kRowRegs];    // word of the bit array held at bw[k][0]
    int32_t nn_cnt[kRowRegs];  // elements held
    int32_t w_cnt[kRowRegs];   // words held
    int64_t qband;             // first queue slot of the CTA's band
    int32_t s0, ts;            // first site and sites of the tile
    int32_t staged;            // 1: every slab and its bits are held whole
    int32_t pad_;
};

struct __align__(16) DenseStage {
    DenseStageHdr h;
    int32_t nn[kRowRegs][kDenseSlab];
    uint32_t bw[kRowRegs][kDenseWords];
};

constexpr size_t kDenseSmem = 64 + sizeof(DenseStage) * kStages;

// The producer warp: lane k computes and issues slot k's two copies. (One lane
// working through the slots took longer than the consumers: 3.4 us a tile of
// six slots, now 2.6.)
template <bool kGen>
__device__ __forceinline__ void dense_produce(const Params &P, DenseStage *st, uint64_t *full, uint64_t *empty,
                                              int lane) {
    int64_t band_lo, band_hi;
    cta_band(P, band_lo, band_hi);
    const int64_t n = P.one.n;
    const int W = (int)P.nn_width;
    const int64_t n_words = ((int64_t)W * n + 31) >> 5;
    const int32_t *nn_end = P.nn + (int64_t)W * n;
    const uint32_t *bits_end = kGen ? nullptr : P.one.bits + n_words;
    const int64_t qband = min(band_lo * kTileSites, n) * W;
    if (lane == 0 && band_lo < band_hi) P.band[P.band_off + blockIdx.x].qbase = qband;
    int64_t t_local = 0;
    for (int64_t tile = band_lo; tile < band_hi; ++tile, ++t_local) {
        const int s = (int)(t_local % kStages);
        const int64_t use = t_local / kStages;
        if (use > 0 && !__all_sync(kFull, mbar_wait_bounded(&empty[s], (uint32_t)((use - 1) & 1)))) {
            if (lane == 0) raise_err(P.err, kErrNonconv);
            break;
        }
        DenseStage &T = st[s];
        DenseStageHdr &h = T.h;
        const int64_t s0 = tile * kTileSites;
        const int64_t ts = min((int64_t)kTileSites, n - s0);
        int64_t nn_lo = 0, nn_hi = 0, w_lo = 0, w_hi = 0;
        bool staged = true;
        if (lane < W) {
            const int64_t e0 = s0 + (int64_t)lane * n, e1 = e0 + ts;
            copy_window(P.nn, e0, e1, P.nn, nn_end, kDenseSlab, nn_lo, nn_hi);
            staged = nn_lo <= e0 && nn_hi >= e1;
            if (!kGen) {
                const int64_t w0 = e0 >> 5, w1 = ((e1 - 1) >> 5) + 1;
                copy_window(P.one.bits, w0, w1, P.one.bits, bits_end, kDenseWords, w_lo, w_hi);
                staged = staged && w_lo <= w0 && w_hi >= w1;
            }
            h.nn_lo[lane] = nn_lo;
            h.nn_cnt[lane] = (int32_t)(nn_hi - nn_lo);
            h.w_lo[lane] = w_lo;
            h.w_cnt[lane] = (int32_t)(w_hi - w_lo);
            if (staged) h.off[lane] = make_int2((int32_t)(e0 - nn_lo), kGen ? 0 : (int32_t)(e0 - 32 * w_lo));
        }
        const uint32_t b_nn = 4u * (uint32_t)(nn_hi - nn_lo), b_w = 4u * (uint32_t)(w_hi - w_lo);
        const uint32_t bytes = __reduce_add_sync(kFull, b_nn + b_w);
        staged = __all_sync(kFull, staged);
        __syncwarp();                   // the lanes' header fields come before the barrier's release
        if (lane == 0) {
            h.s0 = (int32_t)s0;
            h.ts = (int32_t)ts;
            h.qband = qband;
            h.staged = staged ? 1 : 0;
            mbar_arrive_expect_tx(&full[s], bytes);
        }
        __syncwarp();
        if (b_nn) bulk_g2s(T.nn[lane], P.nn + nn_lo, b_nn, &full[s]);
        if (b_w) bulk_g2s(T.bw[lane], P.one.bits + w_lo, b_w, &full[s]);
    }
    if (lane == 0) drain_armed(full, t_local, P.err);
    __syncwarp();
}

// one lane's site of a staged chunk: slot k's neighbour and its open bit
template <bool kGen>
__device__ __forceinline__ void dense_slot(const Params &P, const DenseStage &S, int k, int64_t e, int32_t i,
                                           int32_t &j, bool &open) {
    const DenseStageHdr &h = S.h;
    const int64_t r = e - h.nn_lo[k];
    j = (r >= 0 && r < h.nn_cnt[k]) ? S.nn[k][r] : __ldg(P.nn + e);
    if (kGen) {
        open = j >= 0 && j < i && gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j, (uint32_t)i);
    } else {
        const int64_t w = (e >> 5) - h.w_lo[k];
        const uint32_t word = (w >= 0 && w < h.w_cnt[k]) ? S.bw[k][w] : __ldg(P.one.bits + (e >> 5));
        open = (word >> (e & 31)) & 1u;
    }
}

struct DenseChunk {
    int32_t i, lab;
    uint32_t lowmask;       // open lower slots
    int32_t r;
};

template <bool kGen>
__device__ __forceinline__ void dense_scan_chunk(const Params &P, const DenseStage &S, int cc, int lane,
                                                 const TileCtx &tc, DenseChunk &c) {
    const DenseStageHdr &h = S.h;
    const int64_t n = P.one.n;
    const int W = (int)P.nn_width;
    const int32_t loc = cc * kChunk + lane;
    const int32_t i = h.s0 + loc;
    const bool live = loc < h.ts;
    int32_t m = INT32_MAX, mk = 0;
    uint32_t lowmask = 0;
    bool bad = false;
    if (tc.staged) {
#pragma unroll
        for (int k = 0; k < kRowRegs; ++k) {
            if (k >= W) break;
            const int2 off = h.off[k];
            const int32_t j = live ? S.nn[k][off.x + loc] : -1;
            bool open;
            if (kGen) {
                open = (uint32_t)j < (uint32_t)i &&
                       gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j, (uint32_t)i);
            } else {
                const int32_t b = off.y + loc;
                open = (S.bw[k][b >> 5] >> (b & 31)) & 1u;
            }
            bad |= (uint32_t)(j + 1) > (uint32_t)n;        // j < -1 or j >= n
            if (open && (uint32_t)j < (uint32_t)i) {         // 0 <= j < i
                lowmask |= 1u << k;
                if (j < m) { m = j; mk = k; }
            }
        }
    } else {
        for (int k = 0; k < W; ++k) {
            int32_t j = -1;
            bool open = false;
            if (live) dense_slot<kGen>(P, S, k, (int64_t)i + (int64_t)k * n, i, j, open);
            bad |= j < -1 || (int64_t)j >= n;
            if (j >= 0 && j < i && open) {
                lowmask |= 1u << k;
                if (j < m) { m = j; mk = k; }
            }
        }
    }
    if (bad) raise_err(P.err, kErrIndex);
    const int cnt = __popc(lowmask);
    int32_t lab = cnt ? m : i;
    if (cnt) {
        const int32_t mt = (int32_t)((uint32_t)m / kTileSites);
        if (mt >= tc.vis_lo && mt <= tc.vis_hi) lab = __ldcg(P.one.labels + m);
    }
    c.i = i;
    c.lab = lab;
    c.lowmask = cnt ? (lowmask & ~(1u << mk)) : 0u;
    c.r = cnt > 1 ? cnt - 1 : 0;
}

// The four chunks of a consumer warp at once, on a staged tile that has them
// whole: slot k of the lane's sites i0 + 32 c. Keys, place bits and kWide as in
// scan_rows (bit W - 1 - k of `low` is slot k).
struct DenseRows {
    int32_t lab[kRows];
    uint32_t res;           // residual slots: slot k of row c at bit 8 c + W - 1 - k
};

template <bool kGen, bool kWide>
__device__ __forceinline__ void dense_scan_rows(const Params &P, const DenseStage &S, int loc0, const TileCtx &tc,
                                                DenseRows &q) {
    const DenseStageHdr &h = S.h;
    const uint32_t n = (uint32_t)P.one.n;
    const int W = (int)P.nn_width;
    const int32_t i0 = h.s0 + loc0;
    uint32_t low[kRows], at[kRows], jmax = 0;
    int32_t m[kRows];
#pragma unroll
    for (int c = 0; c < kRows; ++c) {
        low[c] = at[c] = 0;
        m[c] = INT32_MAX;
    }
#pragma unroll
    for (int k = 0; k < kRowRegs; ++k) {
        if (k >= W) break;
        const int2 off = h.off[k];
        const int32_t *nn = S.nn[k] + off.x + loc0;
        const int32_t b = off.y + loc0;
        const uint32_t *bw = S.bw[k] + (b >> 5);        // the lane's bit of chunk c: bit b & 31 of bw[c]
#pragma unroll
        for (int c = 0; c < kRows; ++c) {
            const int32_t i = i0 + kChunk * c;
            const int32_t j = nn[kChunk * c];           // -1: an empty slot, whatever its bit
            jmax = max(jmax, (uint32_t)j + 1u);
            const bool open = kGen ? (uint32_t)j < (uint32_t)i &&
                                         gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j, (uint32_t)i)
                                   : ((bw[c] >> (b & 31)) & 1u) && j >= 0;
            if (kWide) {
                const bool lower = open && (uint32_t)j < (uint32_t)i;
                low[c] = 2u * low[c] + (lower ? 1u : 0u);
                if (lower && j < m[c]) { m[c] = j; at[c] = (uint32_t)k; }
            } else {
                const int32_t key = open ? (int32_t)(8u * (uint32_t)j + (uint32_t)k) : INT32_MAX;
                m[c] = min(m[c], key);
                low[c] = __funnelshift_l((uint32_t)key - 8u * (uint32_t)i, low[c], 1);
            }
        }
    }
    const bool bad = jmax > n;          // j < -1 or j >= n
    if (bad) raise_err(P.err, kErrIndex);
    q.res = 0;
#pragma unroll
    for (int c = 0; c < kRows; ++c) {
        const bool any = low[c] != 0 && !bad;
        const int place = kWide ? (int)at[c] : m[c] & 7;
        q.lab[c] = any ? (kWide ? m[c] : m[c] >> 3) : i0 + kChunk * c;
        if (any) q.res |= (low[c] & ~(1u << (W - 1 - place))) << (8 * c);
    }
    jump_and_shortcut(P.one.labels, h.s0 + (loc0 & ~31), tc, q.lab);
}

template <bool kGen>
__device__ __forceinline__ void dense_emit_rows(const Params &P, const DenseStage &S, const DenseRows &q, int loc0,
                                                int64_t slot, int rr) {
    const int iters = (int)__reduce_max_sync(kFull, (uint32_t)rr);
    const int last = (int)P.nn_width - 1;
    uint32_t mm = q.res;
    int2 *qp = P.q + slot;
    for (int it = 0; it < iters; ++it) {
        const bool put = mm != 0;
        const int t = put ? __ffs(mm) - 1 : 0;
        mm &= mm - 1;
        const int k = last - (t & 7);
        const int32_t up = t & 8 ? q.lab[1] : q.lab[0], up2 = t & 8 ? q.lab[3] : q.lab[2];
        const int2 pr = make_int2(t & 16 ? up2 : up, S.nn[k][S.h.off[k].x + loc0 + kChunk * (t >> 3)]);
        if (put) *qp = pr;
        ++qp;
    }
}

template <bool kGen>
__device__ __forceinline__ void dense_emit_chunk(const Params &P, const DenseStage &S, const DenseChunk &c,
                                                 bool staged, int64_t slot) {
    const int64_t n = P.one.n;
    const int32_t loc = c.i - S.h.s0;
    uint32_t rm = c.lowmask;
    while (rm) {
        const int k = __ffs(rm) - 1;
        rm &= rm - 1;
        int32_t j;
        if (staged) {
            j = S.nn[k][S.h.off[k].x + loc];
        } else {
            bool open;
            dense_slot<kGen>(P, S, k, (int64_t)c.i + (int64_t)k * n, c.i, j, open);
        }
        P.q[slot++] = make_int2(c.lab, j);      // (parent of i, j): see init_emit_chunk
    }
}

template <bool kGen>
__global__ void __launch_bounds__(kInitThreads, kInitCtas) k_init_dense_tma(Params P) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw);
    uint64_t *empty = full + kStages;
    DenseStage *st = reinterpret_cast<DenseStage *>(smem_raw + 64);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kInitConsumers);
        }
        mbar_fence_init();
    }
    __shared__ unsigned long long band_cnt;
    if (threadIdx.x == 0) band_cnt = 0;
    chain_next();
    __syncthreads();
    if (warp == kInitConsumers) {
        dense_produce<kGen>(P, st, full, empty, lane);
        return;
    }
    int64_t band_lo, band_hi;
    cta_band(P, band_lo, band_hi);
    int64_t t_local = 0;
    for (int64_t tile = band_lo; tile < band_hi; ++tile, ++t_local) {
        const int s = (int)(t_local % kStages);
        if (!mbar_wait_bounded(&full[s], (uint32_t)((t_local / kStages) & 1))) {
            raise_err(P.err, kErrNonconv);
            break;
        }
        const DenseStage &S = st[s];
        TileCtx tc;
        tc.rb0 = 0;
        tc.nbits = 0;
        tc.staged = S.h.staged != 0;
        {
            const int64_t hi = tile - kStages;
            tc.vis_lo = (int32_t)band_lo;
            tc.vis_hi = hi < band_lo ? -1 : (int32_t)hi;
        }
        const int loc = warp * kRows * kChunk, loc0 = loc + lane;       // the warp's first site, the lane's
        if (loc < S.h.ts) {
            DenseRows q;
            DenseChunk c[kRows];
            const bool fast = tc.staged && loc + kRows * kChunk <= S.h.ts;
            int rr = 0;
            if (fast) {
                if (P.one.n > (1 << 28)) dense_scan_rows<kGen, true>(P, S, loc0, tc, q);
                else dense_scan_rows<kGen, false>(P, S, loc0, tc, q);
                rr = __popc(q.res);
            } else {
#pragma unroll
                for (int k = 0; k < kRows; ++k) {
                    c[k].r = 0;
                    if (loc + k * kChunk < S.h.ts) dense_scan_chunk<kGen>(P, S, warp * kRows + k, lane, tc, c[k]);
                    rr += c[k].r;
                }
            }
            const int incl = warp_incl_scan(rr, lane);
            const int total = __shfl_sync(kFull, incl, 31);
            unsigned long long base = 0;
            if (total > 0) {
                if (lane == 0) base = atomicAdd(&band_cnt, (unsigned long long)total);
                base = __shfl_sync(kFull, base, 0);
            }
            if (fast) {
                int32_t *out = P.one.labels + S.h.s0 + loc0;
#pragma unroll
                for (int k = 0; k < kRows; ++k) out[kChunk * k] = q.lab[k];
            } else {
#pragma unroll
                for (int k = 0; k < kRows; ++k)
                    if (loc + k * kChunk < S.h.ts && c[k].i < P.one.n) P.one.labels[c[k].i] = c[k].lab;
            }
            if (total > 0) {
                int64_t slot = S.h.qband + (int64_t)base + (incl - rr);
                if (fast) {
                    dense_emit_rows<kGen>(P, S, q, loc0, slot, rr);
                } else {
#pragma unroll
                    for (int k = 0; k < kRows; ++k) {
                        if (c[k].r > 0) dense_emit_chunk<kGen>(P, S, c[k], tc.staged, slot);
                        slot += c[k].r;
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
    }
    consumers_sync<32 * kInitConsumers>();
    if (threadIdx.x == 0) P.band[P.band_off + blockIdx.x].cnt = band_cnt;
}

}  // namespace ccl
