// Device side of the labelling library: the four steps of Section 3 of
// Komura, "A generalized GPU-based connected component labeling algorithm",
// as sm_103a kernels over one or many instances.
//
// Sites are grouped in chunks of 32 consecutive sites of one instance and
// chunks in tiles of kTileSites sites.
//  * Step (i) streams the CSR input: per CTA one producer warp moves each
//    tile's row pointers, column indices and bit words into shared memory with
//    bulk asynchronous copies (cp.async.bulk, completion on mbarriers, a ring
//    of kStages stages); kInitConsumers consumer warps scan the rows (four
//    chunks per warp and tile, one row of each per lane, interleaved), write
//    the labels and append the residual pairs to their band's part of the
//    queue through one prefix sum per warp and tile. A CTA works through
//    contiguous bands of tiles, one or, in large batches, up to kRounds; a
//    site whose smallest lower neighbour lies in a tile of the band finished
//    kStages tiles earlier takes that neighbour's label (most of step (ii) on
//    lattices).
//  * Step (iii) runs Algorithm 1 over the queue: each warp drains a window of
//    pairs, by short walks of two pairs a lane (labels of at most 3/8 of L2) or
//    with six or eight pairs per lane in lockstep rounds (one load or atomicMin
//    per live pair per round, next state from a small table).
//  * Steps (ii)/(iv) chase every site's chain to its root, three chains per
//    lane at once, each warp over contiguous runs of sites (or interleaved,
//    for inputs without locality).
#pragma once
#include <stdint.h>
#include <cuda_runtime.h>

#include "ccl_types.cuh"

namespace ccl {

// ---------------------------------------------------------------------------
// small helpers

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

__device__ __forceinline__ void raise_err(unsigned *err, unsigned bit) {
    if ((*(volatile unsigned *)err & bit) == 0) atomicOr(err, bit);
}

// Bond state drawn on the device. SplitMix64 (Steele, Lea & Flood 2014) in
// counter form: output number `key` of the generator started from state `seed`
// is mix(seed + (key + 1) * 0x9E3779B97F4A7C15); the bond {lo, hi} (lo < hi)
// has key lo * 2^32 + hi and is open iff (output >> 11) < thr, i.e. iff
// (output >> 11) * 2^-53 < p for thr = ceil(p * 2^53).
__device__ __forceinline__ bool gen_bond_open(uint64_t seed, uint64_t thr, uint32_t lo, uint32_t hi) {
    const uint64_t key = ((uint64_t)lo << 32) | hi;
    uint64_t z = seed + (key + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (z >> 11) < thr;
}

// largest k with insts[k].chunk_begin <= c (instances ordered)
__device__ __forceinline__ int find_inst(const Params &P, int64_t c) {
    int lo = 0, hi = P.K - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&P.insts[mid].chunk_begin) <= c) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int find_inst_tile(const Params &P, int64_t t) {
    int lo = 0, hi = P.K - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&P.insts[mid].tile_begin) <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <bool kBatched>
__device__ __forceinline__ Inst inst_of(const Params &P, int k) {
    if (!kBatched) return P.one;
    return P.insts[k];
}

// The instance of a staged tile as the step (i) consumers use it: from the
// kernel parameters for one instance, else from the stage header (shared
// memory) that the producer filled from the instance table.
template <bool kBatched>
__device__ __forceinline__ Inst stage_inst(const Params &P, const StageHdr &h) {
    if (!kBatched) return P.one;
    Inst I;
    I.row_ptr = h.i_rp;
    I.col_idx = h.i_ci;
    I.bits = h.i_bits;
    I.labels = h.i_lab;
    I.bit_off = h.i_bit_off;
    I.tile_begin = h.i_tile_begin;
    I.n = h.i_n;
    I.nnz = h.i_nnz;
    I.rp_lo = I.rp_hi = I.ci_lo = I.ci_hi = I.bits_lo = I.bits_hi = nullptr;   // not used by consumers
    I.q_off = I.chunk_begin = 0;
    return I;
}

// ---------------------------------------------------------------------------
// mbarrier / bulk-copy primitives (inline PTX)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}"
                 ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}"
                 ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Small calls run their kernels as a programmatic chain: each lets the next
// one start while it still runs (chain_next), and the next one waits, before it
// touches memory, until the one before has finished and its writes are visible
// (chain_wait; both do nothing in a kernel launched without the attribute).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// barrier of the first kThreads threads of the CTA
template <int kThreads>
__device__ __forceinline__ void consumers_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
}

// Waits for the phase of `parity` to complete; gives up after a bounded
// number of polls (each poll itself suspends for a hardware-bounded time).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
    for (uint32_t it = 0; it < (1u << 22); ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Called by the producer lane before it returns: waits (bounded) until the
// copies of the last kStages tiles it armed (tiles 0 .. n_armed-1 of its
// band, stage t % kStages) have landed. Copies of earlier tiles have landed
// already: their stages were released by consumers that waited for them. So
// the CTA never exits with bulk copies still writing into its shared memory,
// also when a bounded wait expired and a loop was left early.
__device__ __forceinline__ void drain_armed(uint64_t *full, int64_t n_armed, unsigned *err) {
    for (int64_t t = n_armed > kStages ? n_armed - kStages : 0; t < n_armed; ++t)
        if (!mbar_wait_bounded(&full[t % kStages], (uint32_t)((t / kStages) & 1))) raise_err(err, kErrNonconv);
}

// 1-D bulk copy global -> shared, completing `bytes` on the mbarrier.
// dst, src and bytes are multiples of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// The 16-byte aligned span covering elements [lo, hi) of the 4-byte array
// `arr`, clipped to the readable memory [mlo, mhi). Returns the element range
// [c_lo, c_hi) it covers (relative to arr; may extend past [lo, hi)), or an
// empty range if nothing can be copied or it exceeds `cap` elements.
__device__ __forceinline__ void copy_window(const void *arr, int64_t lo, int64_t hi, const void *mlo,
                                            const void *mhi, int cap, int64_t &c_lo, int64_t &c_hi) {
    const uintptr_t base = (uintptr_t)arr;
    uintptr_t a = (base + 4 * (uintptr_t)lo) & ~(uintptr_t)15;
    uintptr_t b = (base + 4 * (uintptr_t)hi + 15) & ~(uintptr_t)15;
    const uintptr_t l = ((uintptr_t)mlo + 15) & ~(uintptr_t)15;
    const uintptr_t h = (uintptr_t)mhi & ~(uintptr_t)15;
    if (a < l) a = l;
    if (b > h) b = h;
    if (hi <= lo || b <= a || (b - a) / 4 > (uintptr_t)cap) { c_lo = c_hi = lo; return; }
    c_lo = ((intptr_t)a - (intptr_t)base) / 4;
    c_hi = ((intptr_t)b - (intptr_t)base) / 4;
}

// ---------------------------------------------------------------------------
// Step (i): initialisation. For site i: lower = open entries j < i of row i;
// label[i] = min(lower) or i; every other entry of `lower` (one occurrence of
// the minimum removed) is a residual pair (i, j).

// tiles of CTA b: the contiguous band [band_lo, band_hi) of the launch's
// P.n_tiles tiles, which start at tile P.tile_off (0 unless step (i) runs in
// parts); its band record is P.band[P.band_off + b]
__device__ __forceinline__ void cta_band(const Params &P, int64_t &band_lo, int64_t &band_hi) {
    const int64_t per = (P.n_tiles + gridDim.x - 1) / gridDim.x;
    const int64_t lo = min((int64_t)blockIdx.x * per, P.n_tiles);
    band_lo = P.tile_off + lo;
    band_hi = P.tile_off + min(lo + per, P.n_tiles);
}

// Tiles of band `band` of a launch of P.init_bands bands. Bands come in rounds
// of one per CTA, those of round r of P.round_per[r] tiles. A CTA takes band
// blockIdx.x and then, while there are bands left, the next one from a ticket
// counter.
__device__ __forceinline__ void band_tiles(const Params &P, int32_t band, int64_t &lo, int64_t &hi) {
    int32_t r = 0, in = band;
    int64_t first = 0;
    for (; in >= (int32_t)gridDim.x; ++r, in -= (int32_t)gridDim.x) first += (int64_t)gridDim.x * P.round_per[r];
    lo = P.tile_off + min(first + (int64_t)in * P.round_per[r], P.n_tiles);
    hi = P.tile_off + min(first + (int64_t)(in + 1) * P.round_per[r], P.n_tiles);
}

// The bands a CTA has under way (shared memory): at most kStages tiles are, so
// band number `seq` of the CTA can use the place of band seq - kBandSlots.
constexpr int kBandSlots = kStages + 1;
struct BandSlots {
    unsigned long long cnt[kBandSlots];     // pairs found so far
    int32_t band[kBandSlots];
    int32_t taken;                          // bands the CTA has taken
};

// Stores the pair count of a finished band.
__device__ __forceinline__ void store_band(const Params &P, const BandSlots &B, int slot) {
    BandRec &rec = P.band[P.band_off + B.band[slot]];
    const long long room = max((long long)(P.q_cap - rec.qbase), 0ll);      // (less only for corrupt rows)
    rec.cnt = min(B.cnt[slot], (unsigned long long)room);
}

template <bool kBatched, bool kGen = false>
__device__ __forceinline__ void init_produce(const Params &P, Stage *st, uint64_t *full,
                                             uint64_t *empty, BandSlots &B) {
    int64_t t_local = 0;
    int64_t qband = 0;
    int kc = 0;                              // cached instance and its tile range
    int64_t kc_lo = 0, kc_hi = kBatched ? 0 : P.n_tiles;
    int32_t band = blockIdx.x, next = 0;
    bool ok = true;
    for (int32_t seq = 0; ok && band < P.init_bands; ++seq, band = next) {
    int64_t band_lo, band_hi;
    band_tiles(P, band, band_lo, band_hi);
    // the next band is known before this one's last tile is published
    next = gridDim.x < (unsigned)P.init_bands ? (int32_t)(gridDim.x + atomicAdd(P.ticket, 1u)) : P.init_bands;
    // every tile but the last kStages has been consumed, hence all of the
    // band that had this place
    const int slot = seq % kBandSlots;
    if (seq >= kBandSlots) store_band(P, B, slot);
    B.cnt[slot] = 0;
    B.band[slot] = band;
    B.taken = seq + 1;
    for (int64_t tile = band_lo; tile < band_hi; ++tile, ++t_local) {
        const int s = (int)(t_local % kStages);
        const int64_t use = t_local / kStages;
        if (use > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)((use - 1) & 1))) {
            raise_err(P.err, kErrNonconv);
            ok = false;
            break;
        }
        if (kBatched && (tile < kc_lo || tile >= kc_hi)) {
            kc = find_inst_tile(P, tile);
            kc_lo = P.insts[kc].tile_begin;
            kc_hi = kc + 1 < P.K ? P.insts[kc + 1].tile_begin : P.n_tiles;
        }
        const int k = kc;
        const Inst I = inst_of<kBatched>(P, k);
        StageHdr h;
        h.k = k;
        h.s0 = (int32_t)((tile - I.tile_begin) * kTileSites);
        h.ts = min(kTileSites, I.n - h.s0);
        h.e0 = __ldcs(I.row_ptr + h.s0);
        h.e1 = __ldcs(I.row_ptr + h.s0 + h.ts);
        h.status = (h.e0 < 0 || h.e1 < h.e0 || h.e1 > I.nnz) ? 1 : 0;
        // row_ptr[0] == 0 and row_ptr[n] == nnz, once per instance
        if (h.s0 == 0 && h.e0 != 0) raise_err(P.err, kErrShape);
        if (h.s0 + h.ts == I.n && h.e1 != I.nnz) raise_err(P.err, kErrShape);
        h.i_rp = I.row_ptr;
        h.i_ci = I.col_idx;
        h.i_bits = I.bits;
        h.i_lab = I.labels;
        h.i_bit_off = I.bit_off;
        h.i_tile_begin = I.tile_begin;
        h.i_n = I.n;
        h.i_nnz = I.nnz;
        if (tile == band_lo) {
            qband = I.q_off + (h.status ? 0 : h.e0);
            P.band[P.band_off + band].qbase = qband;
        }
        h.qband = qband;
        h.slot = slot;
        h.last = tile + 1 == band_hi && next >= P.init_bands;
        int64_t lo, hi;
        copy_window(I.row_ptr, h.s0, (int64_t)h.s0 + h.ts + 1, I.rp_lo, I.rp_hi, kRpBuf, lo, hi);
        h.rp_lo = (int32_t)lo;
        h.rp_hi = (int32_t)hi;
        if (h.status == 0) {
            copy_window(I.col_idx, h.e0, h.e1, I.ci_lo, I.ci_hi, kColBuf, lo, hi);
            h.ci_lo = (int32_t)lo;
            h.ci_hi = (int32_t)hi;
            const int64_t w0 = (I.bit_off + h.e0) >> 5;
            const int64_t w1 = (h.e1 > h.e0 && !kGen) ? ((I.bit_off + h.e1 - 1) >> 5) + 1 : w0;
            copy_window(I.bits, w0, w1, I.bits_lo, I.bits_hi, kBitBuf, h.w_lo, h.w_hi);
        } else {
            h.ci_lo = h.ci_hi = 0;
            h.w_lo = h.w_hi = 0;
        }
        h.t_rb0 = (int32_t)(I.bit_off - (h.w_lo << 5));
        h.t_nbits = (int32_t)(32 * (h.w_hi - h.w_lo));
        h.t_staged = h.status == 0 && h.e0 >= h.ci_lo && h.e1 <= h.ci_hi &&
                     (kGen || (h.t_rb0 + h.e0 >= 0 && h.t_rb0 + h.e1 <= h.t_nbits));
        {
            // tiles of this band finished at least kStages tiles ago
            const int64_t lo = max(band_lo, I.tile_begin) - I.tile_begin;
            const int64_t hi = tile - kStages - I.tile_begin;
            h.t_vis_lo = (int32_t)lo;
            h.t_vis_hi = hi < lo ? -1 : (int32_t)hi;
        }
        st[s].h = h;
        const uint32_t b_rp = 4u * (uint32_t)(h.rp_hi - h.rp_lo);
        const uint32_t b_ci = 4u * (uint32_t)(h.ci_hi - h.ci_lo);
        const uint32_t b_bw = 4u * (uint32_t)(h.w_hi - h.w_lo);
        mbar_arrive_expect_tx(&full[s], b_rp + b_ci + b_bw);
        if (b_rp) bulk_g2s(st[s].rp, I.row_ptr + h.rp_lo, b_rp, &full[s]);
        if (b_ci) bulk_g2s(st[s].ci, I.col_idx + h.ci_lo, b_ci, &full[s]);
        if (b_bw) bulk_g2s(st[s].bw, I.bits + h.w_lo, b_bw, &full[s]);
    }
    }
    drain_armed(full, t_local, P.err);
}

// Per-tile values a consumer warp computes once: the stage-relative bit
// offset of entry 0 and the number of copied bits (32-bit), and the range of
// the instance's tiles whose labels are final and visible here.
struct TileCtx {
    int32_t rb0;        // stage-relative bit index of local entry 0
    int32_t nbits;      // bits present in the stage
    int32_t vis_lo;     // instance-local tiles [vis_lo, vis_hi] are visible
    int32_t vis_hi;
    bool staged;        // the stage holds the columns and bits of the tile's whole entry range
};

// The stage header words the register path reads, copied to registers once
// per tile with 16-byte shared-memory loads.
struct TileHdr {
    int32_t k, s0, ts, e0, e1, rp_lo, rp_hi, ci_lo;
};

__device__ __forceinline__ void load_tile_hdr(const StageHdr &h, TileHdr &th, TileCtx &tc) {
    const int4 a = *reinterpret_cast<const int4 *>(&h.k);
    const int4 b = *reinterpret_cast<const int4 *>(&h.e1);
    const int4 c = *reinterpret_cast<const int4 *>(&h.t_rb0);
    th.k = a.x; th.s0 = a.y; th.ts = a.z; th.e0 = a.w;
    th.e1 = b.x; th.rp_lo = b.y; th.rp_hi = b.z; th.ci_lo = b.w;
    tc.rb0 = c.x; tc.nbits = c.y; tc.staged = c.z != 0; tc.vis_lo = c.w;
    tc.vis_hi = h.t_vis_hi;
}

// The open lower entries among the `cnt` (at most kRowRegs) entries from e on of
// row i, as a mask, and their columns. A tile's entries are in the stage or, when
// it has more than the stage holds, all read from global memory; either way a
// lane's loads of a block do not depend on one another.
template <bool kGen>
__device__ __forceinline__ uint32_t lower_block(const Params &P, const Stage &S, const Inst &I, const TileCtx &tc,
                                                int32_t e, int32_t cnt, int32_t i, int32_t (&j)[kRowRegs], bool &bad) {
    uint32_t win = 0;
    if (tc.staged) {
        const int32_t *col = S.ci + (e - S.h.ci_lo);
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) j[u] = u < cnt ? col[u] : -1;
        if (!kGen && cnt > 0) {
            const int32_t rel = tc.rb0 + e;
            win = __funnelshift_r(S.bw[rel >> 5], S.bw[(rel + cnt - 1) >> 5], (uint32_t)rel & 31u);
        }
    } else {
        const int32_t *col = I.col_idx + e;
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) j[u] = u < cnt ? __ldg(col + u) : -1;
        if (!kGen && cnt > 0) {
            const int64_t ge = I.bit_off + e;
            win = __funnelshift_r(__ldg(I.bits + (ge >> 5)), __ldg(I.bits + ((ge + cnt - 1) >> 5)), (uint32_t)ge & 31u);
        }
    }
    uint32_t low = 0;
#pragma unroll
    for (int u = 0; u < kRowRegs; ++u) {
        const bool lower = (uint32_t)j[u] < (uint32_t)i;            // (none past cnt)
        const bool open = kGen ? lower && gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j[u], (uint32_t)i)
                               : lower && ((win >> u) & 1u);
        bad |= u < cnt && (uint32_t)j[u] >= (uint32_t)I.n;
        low |= open ? 1u << u : 0u;
    }
    return low;
}

// One chunk of 32 sites, whatever its rows: in blocks of kRowRegs entries. The tiles
// of this CTA's band that were finished at least kStages tiles ago are visible
// (their labels were released through the stage barriers): a site whose smallest
// open lower neighbour m lies in such a tile takes label[m] (the root of m's tree
// after steps (i)/(ii)) instead of m, which shortcuts the chain step (ii) would walk.
// What bounds it is the latency of the columns when the stage does not hold them:
// the blocks' loads overlap. Step (i) of 4M sites with 12 random near entries each
// took 550 us entry by entry with four rows a lane (349 with two, twice the warps),
// 150 so; of a tree of 23,437 sites, whose last tile the stage holds short of its last
// entries, 18 (13) and 14.
struct ChunkRes {           // what the emission needs (per lane)
    int32_t i, a, deg, mk;
    int32_t lab;            // label[i] to store (may be a load still in flight)
    uint32_t resmask;       // residual entries among the row's first 32
    int32_t r;              // residual pairs of the lane's site
};

template <bool kGen>
__device__ __forceinline__ void init_scan_chunk(const Params &P, const Stage &S, const Inst &I,
                                                int cc, int lane, const TileCtx &tc, ChunkRes &cr) {
    const StageHdr &h = S.h;
    const int32_t n = I.n;
    const int32_t s0 = h.s0 + cc * kChunk;
    const int32_t i = s0 + lane;
    const int32_t slast = min(s0 + kChunk, n);
    int32_t a, a_next;
    if (s0 >= h.rp_lo && slast < h.rp_hi) {
        a = S.rp[min(i, slast) - h.rp_lo];
        a_next = S.rp[min(i + 1, slast) - h.rp_lo];
    } else {
        a = __ldcs(I.row_ptr + min(i, slast));
        a_next = __ldcs(I.row_ptr + min(i + 1, slast));
    }
    // A row outside the tile's entry range, or running backwards, is read as
    // empty and flagged; the rows of a valid input always pass.
    if (!(a >= h.e0 && a <= a_next && a_next <= h.e1 && h.status == 0)) {
        raise_err(P.err, kErrIndex);
        a = a_next = h.e0 > 0 ? h.e0 : 0;
    }
    // rows now lie inside [e0, e1]; tc.staged says whether the stage holds
    // all of that range (columns and bits)
    const int32_t deg = a_next - a;
    const int32_t dmax = __reduce_max_sync(kFull, (uint32_t)deg);
    int32_t m = INT32_MAX, cnt = 0, mk = -1;
    uint32_t resmask = 0;
    bool bad = false;
    for (int32_t t = 0; t < dmax; t += kRowRegs) {
        int32_t j[kRowRegs];
        const uint32_t low = lower_block<kGen>(P, S, I, tc, a + t, min(max(deg - t, 0), kRowRegs), i, j, bad);
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u)
            if (((low >> u) & 1u) && j[u] < m) { m = j[u]; mk = t + u; }
        cnt += __popc(low);
        if (t < 32) resmask |= low << t;
    }
    if (cnt && mk < 32) resmask &= ~(1u << mk);
    if (bad) raise_err(P.err, kErrIndex);
    // the label; the caller stores it after the prefix sum over the pairs, so the
    // shortcut's load below has that time to arrive
    int32_t lab = cnt ? m : i;
    if (cnt) {
        const int32_t mt = (int32_t)((uint32_t)m / kTileSites);
        if (mt >= tc.vis_lo && mt <= tc.vis_hi) lab = __ldcg(I.labels + m);
    }
    cr.lab = lab;
    cr.i = i;
    cr.a = a;
    cr.deg = deg;
    cr.mk = mk;
    cr.resmask = resmask;
    cr.r = cnt > 1 ? cnt - 1 : 0;
}

// The four rows of a lane on the register path.
struct RowsRes {
    int32_t lab[kRows];     // labels to store (may be loads still in flight)
    int32_t off[kRows];     // stage index of each row's first column
    uint32_t res;           // residual entries: entry t of row k at bit 8 k + last - t
    int32_t last;
};

// Scans four rows per lane, rows s00 + 32 k + lane. kD > 0: every row has kD
// entries; kD = 0: row k has d[k] <= kRowRegs entries, dmax the longest of the
// warp. The rows are interleaved, so their loads and dependent arithmetic
// overlap.
//
// Step (i) is bound by the instructions of this scan (the integer pipe), not
// by memory, until rows are cheap. With four rows a lane the tile's header, the
// prefix sum and the queue bookkeeping are paid once for 128 sites; rows of one
// degree need no row ends, no per-entry tests of the row's length and half the
// loads (the rows of a lane lie 32 apart, so 8-byte loads of degree 4 and 6 and
// 4-byte loads of degree 3 spread over the banks); keys find the smallest
// neighbour and its place with one minimum; mixed rows read past their ends and
// mask instead of branching. Against two rows a lane entry by entry, step (i) of
// triangle 4096^2 160 -> 116 us (5.0 TB/s; streaming alone takes 88), of the Bethe
// lattice of 24 shells 390 -> 318; a call of few tiles pays 1 us for the longer
// lanes (honeycomb 64^2).
template <bool kGen, int kD, bool kWide = false>
__device__ __forceinline__ void scan_rows(const Params &P, const Stage &S, const TileCtx &tc, const TileHdr &h,
                                          int32_t n, int32_t s00, int lane, const int32_t (&a)[kRows],
                                          const int32_t (&d)[kRows], int32_t dmax, RowsRes &q, bool &bad) {
    const int32_t *col[kRows];
    uint32_t w[kRows], low[kRows];
    int32_t m[kRows];
    uint32_t jmax = 0;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        q.off[k] = a[k] - h.ci_lo;
        col[k] = S.ci + q.off[k];
        low[k] = 0;
        m[k] = INT32_MAX;
        w[k] = 0;
        if (!kGen) {
            const int32_t rel = tc.rb0 + a[k];
            const uint32_t *bw = S.bw + (rel >> 5);
            // (an empty row's may lie past the copied words)
            if (kD > 0 || d[k] > 0) w[k] = __funnelshift_r(bw[0], bw[1], (uint32_t)rel & 31u);
            w[k] &= kD > 0 ? 0xffu : 0xffu >> (kRowRegs - d[k]);        // the row's own bits
        } else {
            w[k] = kD > 0 ? 0xffu : 0xffu >> (kRowRegs - d[k]);
        }
    }
    // Open entries as keys 8 j + t (closed ones above every site's): the
    // smallest key is the smallest open neighbour and its place, and entry t
    // is an open lower one iff its key is below 8 i. The signs of the keys'
    // differences to 8 i collect in `low`, entry t of T at bit T - 1 - t.
    // Keys need sites below 2^28; kWide keeps the neighbour and its place apart.
    // (entries past a row's end, closed by w, are read all the same: the scan of
    // mixed rows does not branch)
    auto entry = [&](int k, int t, int32_t j, bool in_row) {
        const int32_t i = s00 + kChunk * k + lane;
        jmax = max(jmax, in_row ? (uint32_t)j : 0u);
        bool open = (w[k] >> t) & 1u;
        if (kGen) open = open && (uint32_t)j < (uint32_t)i && gen_bond_open(P.gen_seed, P.gen_thr, (uint32_t)j, (uint32_t)i);
        if (kWide) {
            const bool lower = open && (uint32_t)j < (uint32_t)i;
            low[k] = 2u * low[k] + (lower ? 1u : 0u);
            if (lower && j < m[k]) { m[k] = j; w[k] = (w[k] & 0xffu) | ((uint32_t)t << 8); }
        } else {
            const int32_t key = open ? (int32_t)(8u * (uint32_t)j + (uint32_t)t) : INT32_MAX;
            m[k] = min(m[k], key);
            low[k] = __funnelshift_l((uint32_t)key - 8u * (uint32_t)i, low[k], 1);
        }
    };
    if (kD > 0 && kD % 2 == 0) {
        // the rows start at even stage indices: two columns per load
#pragma unroll
        for (int t = 0; t < kD; t += 2)
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const int2 jj = *reinterpret_cast<const int2 *>(col[k] + t);
                entry(k, t, jj.x, true);
                entry(k, t + 1, jj.y, true);
            }
    } else if (kD > 0) {
#pragma unroll
        for (int t = 0; t < kD; ++t)
#pragma unroll
            for (int k = 0; k < kRows; ++k) entry(k, t, col[k][t], true);
    } else {
#pragma unroll
        for (int t = 0; t < kRowRegs; ++t) {
            if (t >= dmax) break;
#pragma unroll
            for (int k = 0; k < kRows; ++k) entry(k, t, col[k][t], t < d[k]);
        }
    }
    bad = jmax >= (uint32_t)n;
    q.res = 0;
    q.last = (kD > 0 ? kD : dmax) - 1;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        // (no label comes from a row of a lane that saw a column out of range)
        const bool any = low[k] != 0 && !bad;
        const int at = kWide ? (int)(w[k] >> 8) : m[k] & 7;      // place of the smallest
        q.lab[k] = any ? (kWide ? m[k] : m[k] >> 3) : s00 + kChunk * k + lane;
        if (any) q.res |= (low[k] & ~(1u << (q.last - at))) << (8 * k);
    }
}

// The labels of a warp's four chunks from site s00 on before they are stored.
__device__ __forceinline__ void jump_and_shortcut(const int32_t *labels, int32_t s00, const TileCtx &tc,
                                                  int32_t (&lab)[kRows]) {
    // One pointer jump inside each chunk: a label that points to a site of the
    // chunk takes that site's label. The value taken is an ancestor of the
    // site, so it stays a valid label, and a chain along a lattice row shortens
    // by half before step (iii) and the analysis follow it.
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        const uint32_t in = (uint32_t)(lab[k] - (s00 + kChunk * k));
        const int32_t up = __shfl_sync(kFull, lab[k], (int)(in & 31u));
        if (in < 32u) lab[k] = up;
    }
    // a label in a tile of this band finished kStages tiles ago: take that
    // site's label (the band shortcut)
    const uint32_t vis_lo = (uint32_t)tc.vis_lo * kTileSites;
    const uint32_t vis_n = tc.vis_hi < tc.vis_lo ? 0u : (uint32_t)(tc.vis_hi + 1 - tc.vis_lo) * kTileSites;
#pragma unroll
    for (int k = 0; k < kRows; ++k)
        if ((uint32_t)lab[k] - vis_lo < vis_n) lab[k] = __ldcg(labels + lab[k]);
}

// Whether rows lie in the tile's entries [e0, e1], given the first row's start
// and the last one's end and that every row is between 0 and kRowRegs long modulo
// 2^32: row pointers that pass 2^31 on the way come out below where they began.
__host__ __device__ constexpr bool rows_inside(int32_t first, int32_t last, int32_t e0, int32_t e1) {
    return first >= e0 && last >= first && last <= e1;
}
static_assert(rows_inside(0, 384, 0, 3072) && rows_inside(2688, 3072, 0, 3072) && rows_inside(5, 5, 5, 5), "valid rows");
static_assert(!rows_inside(INT32_MAX - 60, INT32_MIN + 323, 0, 3072), "wrapped row pointers");
static_assert(!rows_inside(-1, 383, 0, 3072) && !rows_inside(2689, 3073, 0, 3072), "outside the tile");

// The four chunks of a consumer warp at once, when all their rows exist, are
// short and staged (the common case). Returns false (having done nothing)
// otherwise.
template <bool kGen>
__device__ __forceinline__ bool init_scan_rows(const Params &P, const Stage &S, const Inst &I, int32_t s00, int lane,
                                               const TileCtx &tc, const TileHdr &h, RowsRes &q) {
    const int32_t n = I.n;
    if (!tc.staged || s00 + kRows * kChunk > n || s00 < h.rp_lo || s00 + kRows * kChunk >= h.rp_hi) return false;
    const int32_t *rp = S.rp + (s00 - h.rp_lo);
    int32_t a[kRows], d[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) a[k] = rp[lane + kChunk * k];
    // rows of one degree D throughout (a lattice): a[k] = first + D * (lane + 32 k)
    const int32_t first = __shfl_sync(kFull, a[0], 0);
    const uint32_t D = (uint32_t)__shfl_sync(kFull, a[0], 1) - (uint32_t)first;
    const int32_t last = rp[kRows * kChunk];
    uint32_t x = (uint32_t)a[0] - (uint32_t)first - D * (uint32_t)lane;
#pragma unroll
    for (int k = 1; k < kRows; ++k) x |= (uint32_t)a[k] - (uint32_t)a[k - 1] - kChunk * D;
    x |= (uint32_t)last - (uint32_t)first - kRows * kChunk * D;
    const bool inside = rows_inside(first, last, h.e0, h.e1);
    const bool one_degree = __all_sync(kFull, x == 0) && inside;
    const bool wide = n > (1 << 28);
    bool bad = false;
    if (one_degree && !wide && D == 3) {
        scan_rows<kGen, 3>(P, S, tc, h, n, s00, lane, a, d, 3, q, bad);
    } else if (one_degree && !wide && D == 6 && ((first - h.ci_lo) & 1) == 0) {
        scan_rows<kGen, 6>(P, S, tc, h, n, s00, lane, a, d, 6, q, bad);
    } else if (one_degree && !wide && D == 4 && ((first - h.ci_lo) & 1) == 0) {
        scan_rows<kGen, 4>(P, S, tc, h, n, s00, lane, a, d, 4, q, bad);
    } else {
        uint32_t dm = 0;
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            d[k] = rp[lane + kChunk * k + 1] - a[k];
            dm = max(dm, (uint32_t)d[k]);       // (a row running backwards counts as long)
        }
        const int32_t dmax = (int32_t)__reduce_max_sync(kFull, dm);
        if ((uint32_t)dmax > (uint32_t)kRowRegs || !inside) return false;
        if (wide) scan_rows<kGen, 0, true>(P, S, tc, h, n, s00, lane, a, d, dmax, q, bad);
        else scan_rows<kGen, 0>(P, S, tc, h, n, s00, lane, a, d, dmax, q, bad);
    }
    if (bad) raise_err(P.err, kErrIndex);
    jump_and_shortcut(I.labels, s00, tc, q.lab);
    return true;
}

// Writes the residual pairs of one scanned chunk from queue slot `slot` on (the
// warp's slots have been checked against the queue's end).
// A pair {i, j} is stored as (label[i], j): label[i] is i's parent in the
// label forest and, i not being a root, step (iii) never rewrites it, so the
// pair joins the same two trees and its root search starts one hop higher.
template <bool kBatched, bool kGen = false>
__device__ __forceinline__ void init_emit_chunk(const Params &P, const Stage &S, const Inst &I, const TileCtx &tc,
                                                const ChunkRes &cr, int64_t slot) {
    const auto put = [&](int32_t j) {
        P.q[slot] = make_int2(cr.lab, j);
        if (kBatched) P.qk[slot] = S.h.k;
        ++slot;
    };
    const int32_t *col = tc.staged ? S.ci + (cr.a - S.h.ci_lo) : I.col_idx + cr.a;
    for (uint32_t res = cr.resmask; res; res &= res - 1) put(col[__ffs(res) - 1]);
    for (int32_t t = 32; t < cr.deg; t += kRowRegs) {           // past the mask: scanned again
        int32_t j[kRowRegs];
        bool bad = false;
        const uint32_t low = lower_block<kGen>(P, S, I, tc, cr.a + t, min(cr.deg - t, kRowRegs), cr.i, j, bad);
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u)
            if (((low >> u) & 1u) && t + u != cr.mk) put(j[u]);
    }
}

// The residual pairs of a lane's four rows on the register path, in one loop
// with a warp-uniform trip count and without branches, so the warp neither
// diverges nor loops four times (with a branch around lanes that have no pair
// left: step (i) of 1024 mixed instances 3.15 ms instead of 3.08, of the Bethe
// lattice 325 us instead of 318). The warp's queue slots have been checked
// against the queue's end.
template <bool kBatched>
__device__ __forceinline__ void init_emit_rows(const Params &P, const Stage &S, const TileHdr &h, const RowsRes &q,
                                               int64_t slot, int rr) {
    const int iters = (int)__reduce_max_sync(kFull, (uint32_t)rr);
    uint32_t mm = q.res;
    int2 *qp = P.q + slot;
    int32_t *kp = kBatched ? P.qk + slot : nullptr;
    for (int it = 0; it < iters; ++it) {
        // (a lane without a pair left reads some column and stores nothing)
        const bool put = mm != 0;
        const int t = put ? __ffs(mm) - 1 : 0;
        mm &= mm - 1;
        int32_t off = t & 8 ? q.off[1] : q.off[0], up = t & 8 ? q.lab[1] : q.lab[0];
        const int32_t off2 = t & 8 ? q.off[3] : q.off[2], up2 = t & 8 ? q.lab[3] : q.lab[2];
        if (t & 16) { off = off2; up = up2; }
        const int2 pr = make_int2(up, S.ci[off + q.last - (t & 7)]);
        if (put) {
            *qp = pr;
            if (kBatched) *kp = h.k;
        }
        ++qp;
        if (kBatched) ++kp;
    }
}

// Queue slots for the residual pairs of a warp's sites, r of the lane's: sets the
// first slot and the warp's total, returns the pairs of the lanes before.
__device__ __forceinline__ int take_slots(const Stage &S, BandSlots &bands, int lane, int r, int64_t &slot, int &total) {
    const int incl = warp_incl_scan(r, lane);
    total = __shfl_sync(kFull, incl, 31);
    unsigned long long base = 0;
    if (total > 0) {
        if (lane == 0) base = atomicAdd(&bands.cnt[S.h.slot], (unsigned long long)total);
        base = __shfl_sync(kFull, base, 0);
    }
    slot = S.h.qband + (int64_t)base;
    return incl - r;
}

// Whether the slots end inside the queue (always, but for corrupt rows: then what is
// left of it becomes pairs (0, 0), as step (iii) reads every slot up to the end).
template <bool kBatched>
__device__ __forceinline__ bool slots_fit(const Params &P, int32_t k, int64_t slot, int total, int lane) {
    if (slot + total <= P.q_cap) return true;
    if (lane == 0) raise_err(P.err, kErrIndex);
    for (int64_t e = slot + lane; e < P.q_cap; e += 32) {
        P.q[e] = make_int2(0, 0);
        if (kBatched) P.qk[e] = k;
    }
    return false;
}

template <bool kBatched, bool kGen = false>
__global__ void __launch_bounds__(kInitThreads, kInitCtas) k_init(Params P) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw);
    uint64_t *empty = full + kStages;
    Stage *st = reinterpret_cast<Stage *>(smem_raw + 64);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kInitConsumers);
        }
        mbar_fence_init();
    }
    __shared__ BandSlots bands;
    if (threadIdx.x == 0) bands.taken = 0;
    chain_next();
    __syncthreads();
    if (warp == kInitConsumers) {               // producer warp
        if (lane == 0) init_produce<kBatched, kGen>(P, st, full, empty, bands);
        return;
    }
    // stage and phase parity of the CTA's tile number t are t % kStages and
    // (t / kStages) & 1, kept incrementally in 32-bit (no 64-bit division)
    int s = 0;
    uint32_t ph = 0;
    for (bool last = false; !last; s = (s + 1 == kStages) ? 0 : s + 1, ph ^= (s == 0) ? 1u : 0u) {
        if (!mbar_wait_bounded(&full[s], ph)) {
            raise_err(P.err, kErrNonconv);
            break;
        }
        last = st[s].h.last != 0;
        const Stage &S = st[s];
        const Inst I = stage_inst<kBatched>(P, S.h);
        TileCtx tc;
        TileHdr th;
        load_tile_hdr(S.h, th, tc);
        // The warp's rows are scanned first; their pairs then take one range of
        // queue slots (one prefix sum and one band counter update per tile),
        // taken before the labels are stored: the shortcut's label loads land
        // meanwhile.
        const int32_t loc = warp * kRows * kChunk;      // the warp's first site in the tile
        if (loc < th.ts) {
            const int32_t s00 = th.s0 + loc;
            RowsRes q;
            // (both ways meet here before the slots are taken: with a prefix sum of its
            // own behind the scan the labels' loads were waited for earlier, 3 % of step
            // (i) beyond L2, triangle 16384^2 1845 us)
            const bool fast = init_scan_rows<kGen>(P, S, I, s00, lane, tc, th, q);
            const int rr = fast ? __popc(q.res) : 0;
            int64_t slot;
            int total;
            const int before = take_slots(S, bands, lane, rr, slot, total);
            if (fast) {
                int32_t *out = I.labels + s00 + lane;
#pragma unroll
                for (int k = 0; k < kRows; ++k) out[kChunk * k] = q.lab[k];
                if (total > 0 && slots_fit<kBatched>(P, th.k, slot, total, lane))
                    init_emit_rows<kBatched>(P, S, th, q, slot + before, rr);
            } else {
                // chunk by chunk, in one copy of the code: a call of few tiles runs it
                // from a cold instruction cache (a whole call of honeycomb 256^2 at
                // 1.2 p_c with four copies 41 us, 38 so; registers 90, 70 so)
#pragma unroll 1
                for (int k = 0; k < kRows && loc + k * kChunk < th.ts; ++k) {
                    ChunkRes c;
                    init_scan_chunk<kGen>(P, S, I, warp * kRows + k, lane, tc, c);
                    const int before = take_slots(S, bands, lane, c.r, slot, total);
                    if (c.i < I.n) I.labels[c.i] = c.lab;
                    if (total > 0 && slots_fit<kBatched>(P, th.k, slot, total, lane) && c.r > 0)
                        init_emit_chunk<kBatched, kGen>(P, S, I, tc, c, slot + before);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
    }
    // the last bands' pair counts, once every consumer warp has added its own
    // (the producer warp may have returned)
    consumers_sync<32 * kInitConsumers>();
    if (threadIdx.x == 0)
        for (int32_t q = max(bands.taken - kBandSlots, 0); q < bands.taken; ++q) store_band(P, bands, q % kBandSlots);
}

// ---------------------------------------------------------------------------
// Steps (ii) and (iv): analysis. Every site follows its label chain to the
// root and stores the root. No atomics run concurrently with this kernel and
// every value written is an ancestor of the site, so plain stores are safe.
//
// A warp visits groups of kAnaChunks chunks, one chain per lane and chunk, all
// chains of a round in flight together; a finished chain is predicated off (its
// repeated loads would take the L1's gather bandwidth). Runs of P.ana_group = G
// groups go to the warps in turn, so all warps work inside one super-chunk of
// nwarps * G groups at a time and the labels in use (and the roots the chains
// reach, in the same instances) stay in L2 when the whole array does not fit;
// G = 0: one run per warp (everything fits). Sites come in increasing order
// inside a run, so its later chains run into roots it has already stored.
//
// The gathers hit L1 and L2 for the most part; what bounds the kernel is their
// latency and the instructions around them, so a run is cut into stretches of
// one instance with 32-bit site numbers, and a round is a load, a compare and
// a move per chain. Against the same walk with the instance, 64-bit chunk
// numbers and caps looked at for every chunk: 1024 mixed instances 2.54 -> 1.23 ms,
// triangle 4096^2 66 -> 47 us (2.8 TB/s of its 8 bytes per site); a Bethe lattice's
// random gathers over 201 MB hardly gain. Three chunks a group beat two and four
// (0.67 ms on triangle 16384^2, 0.87, 0.79), two rounds between votes beat one;
// 256 threads of 32 registers fill the SM.
constexpr int kAnaRounds = 4;                        // rounds before a chain is set aside (kPark)
constexpr int kParkCap = 32 * kAnaChunks + 32;       // < 32 left + one group's chains

// kPark = true (an option): a chain unfinished after kAnaRounds rounds goes to
// a per-warp list in shared memory, finished 32 at a time, one per lane, so a
// few long chains do not hold up the lanes of a whole group. (Slower than
// waiting on every input measured: triangle 4096^2 55 us, 1024 mixed instances
// 1.53 ms.)
//
// kSample = true (step (ii) when the library chooses): an instance is left alone
// unless fewer than one in kSampleRoots of kSampleChunks chunks spread over it
// are roots (which sites are roots does not change here, so every warp decides
// alike). A chain ends at each hop with about that probability: where roots
// are common chains are a few hops long and step (iii) does better alone, where
// they are rare each of its pairs would walk a long chain. Calls without / with
// the pass, and by sample: honeycomb 2896^2 at 1.5 p_c 581 / 308 / 302 us, triangle
// 2048^2 155 / 122 / 124; at p_c, left alone, it costs its launch and one read:
// triangle 4096^2 250 / 279 / 254. The line lies at 0.125: triangles at 1.5 p_c
// (0.11) and honeycomb lattices at 1.2 p_c (0.13) are about even. Deciding per
// stretch of 96 sites instead costs more than either (triangle 2048^2 173).
constexpr int kSampleRoots = 8, kSampleChunks = 12;
// Calls of at most this many sites are walked without a sample. They are launches
// and latency: the walk costs them what the sample does, and mends the inputs the
// sample leaves alone although step (iii) has long chains to follow (square 256^2 at
// 1.3 p_c 41 us sampled, 36 walked; triangle 256^2 at 1.5 p_c 46 and 38; at p_c
// honeycomb 64^2 27 and 26, triangle 512^2 38 and 39). From a million sites on the
// walk costs more at p_c than it gives (triangle 1024^2 52 and 55).
constexpr int64_t kWalkSites = 1 << 18;
// Instances of more than kDeepSites sites of whose sample fewer than one in
// kDeepRoots is a root: see drain_deep.
constexpr int64_t kDeepSites = 1 << 21;
constexpr int kDeepRoots = 18;
template <bool kBatched, bool kPark, bool kSample = false>
__global__ void __launch_bounds__(512, 4) k_analysis(Params P) {
    extern __shared__ int s_park[];                  // kPark: site and label of kParkCap chains per warp
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31;
    int *s_site = s_park + (threadIdx.x >> 5) * (2 * kParkCap), *s_x = s_site + kParkCap;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t ngroups = (P.n_chunks + kAnaChunks - 1) / kAnaChunks;
    const int64_t per = (ngroups + nwarps - 1) / nwarps;
    const int64_t G = P.ana_group > 0 && P.ana_group < per ? (int64_t)P.ana_group : per;
    // the instance of the current stretch: its chunks, labels and sites
    int64_t kc_lo = 0, kc_hi = kBatched ? 0 : P.n_chunks;
    int32_t *lab = P.one.labels;
    int32_t n = P.one.n;
    int cnt = 0;                                     // chains set aside
    // no chain of valid labels is longer than n
    const auto cap = [&]() { return P.iter_cap > 0 ? P.iter_cap : n; };
    const auto drain = [&](int take) {
        const int base = cnt - take;
        const bool mine = lane < take;
        int site = 0, x = 0;
        if (mine) {
            site = s_site[base + lane];
            x = s_x[base + lane];
        }
        bool act = mine;
        for (int32_t it = 0;; ++it) {
            int32_t y = x;
            if (act) y = lab[x];
            act = y != x;
            x = y;
            if (!__any_sync(kFull, act)) break;
            if (it >= cap()) { raise_err(P.err, kErrNonconv); break; }
        }
        if (mine) lab[site] = x;
        cnt = base;
        __syncwarp();
    };
    const auto sample = [&]() {
        const int32_t step = n / kSampleChunks;
        int roots = 0, sites = 0;
#pragma unroll
        for (int u = 0; u < kSampleChunks; ++u) {
            const int32_t i = u * step + step / 2 + lane;
            roots += __popc(__ballot_sync(kFull, i < n && lab[min(i, n - 1)] == i));
            sites += __popc(__ballot_sync(kFull, i < n));
        }
        if (!kBatched && P.deep && wid == 0 && lane == 0) *P.deep = roots * kDeepRoots < sites;
        return roots * kSampleRoots < sites;
    };
    bool walk = kSample && !kBatched && sample();
    if (kSample && !kBatched && !walk) return;
    for (int64_t run = wid * G; run < ngroups; run += nwarps * G) {
        int64_t c = run * kAnaChunks;
        const int64_t c_end = min((run + G) * kAnaChunks, P.n_chunks);
        while (c < c_end) {
            if (kBatched && (c < kc_lo || c >= kc_hi)) {
                const int kc = find_inst(P, c);
                kc_lo = P.insts[kc].chunk_begin;
                kc_hi = kc + 1 < P.K ? P.insts[kc + 1].chunk_begin : P.n_chunks;
                lab = P.insts[kc].labels;
                n = P.insts[kc].n;
                if (kSample) walk = sample();
            }
            // the stretch of this run inside the instance: the lane's sites s
            // + 32 u below s_end
            const int64_t ce = min(c_end, kc_hi);
            int32_t s = (int32_t)((c - kc_lo) * kChunk) + lane;
            const int32_t s_end = (int32_t)min((ce - kc_lo) * kChunk, (int64_t)n);
            c = ce;
            if (kSample && !walk) continue;
            for (; s - lane < s_end; s += kChunk * kAnaChunks) {
                int32_t x[kAnaChunks], first[kAnaChunks];
                bool act[kAnaChunks];
                int32_t *p = lab + s;
#pragma unroll
                for (int u = 0; u < kAnaChunks; ++u) {
                    x[u] = s + kChunk * u;
                    if (s + kChunk * u < s_end) x[u] = p[kChunk * u];
                }
#pragma unroll
                for (int u = 0; u < kAnaChunks; ++u) {
                    first[u] = x[u];
                    act[u] = x[u] != s + kChunk * u;
                }
                const auto round = [&]() {
                    int32_t y[kAnaChunks];
#pragma unroll
                    for (int u = 0; u < kAnaChunks; ++u) {
                        y[u] = x[u];
                        if (act[u]) y[u] = lab[x[u]];
                    }
#pragma unroll
                    for (int u = 0; u < kAnaChunks; ++u) {
                        act[u] = y[u] != x[u];
                        x[u] = y[u];
                    }
                };
                if (kPark) {
#pragma unroll
                    for (int r = 0; r < kAnaRounds; ++r) round();
#pragma unroll
                    for (int u = 0; u < kAnaChunks; ++u) {
                        if (!act[u] && x[u] != first[u]) p[kChunk * u] = x[u];
                        const unsigned pk = __ballot_sync(kFull, act[u]);
                        if (pk) {
                            const int pos = cnt + __popc(pk & lt);
                            if (act[u]) {
                                s_site[pos] = s + kChunk * u;
                                s_x[pos] = x[u];
                            }
                            cnt += __popc(pk);
                            __syncwarp();
                            if (cnt >= 32) drain(32);
                        }
                    }
                } else {
                    for (int32_t it = 2;; it += 2) {
                        round();
                        round();
                        bool any = false;
#pragma unroll
                        for (int u = 0; u < kAnaChunks; ++u) any |= act[u];
                        if (!__any_sync(kFull, any)) break;
                        if (it >= cap()) { raise_err(P.err, kErrNonconv); break; }
                    }
#pragma unroll
                    for (int u = 0; u < kAnaChunks; ++u)
                        if (x[u] != first[u]) p[kChunk * u] = x[u];
                }
            }
            if (kPark && kBatched) while (cnt > 0) drain(min(cnt, 32));     // (they belong to this instance)
        }
    }
    if (kPark) while (cnt > 0) drain(min(cnt, 32));
}

// ---------------------------------------------------------------------------
// Step (iii): label reduction, Algorithm 1 for every residual pair (i, j).
// The pairs of all bands form one flat index space (prefix sums of the band
// counts, in shared memory). A warp drains a window of pairs (at most
// kRedWindowMax, fewer when the queue is short so every warp has one); each
// lane carries six or eight pairs and takes the next pair of the window as soon
// as one finishes, so a long walk holds up one slot, not the warp. Every
// round issues one load or one atomicMin per live slot before any result is
// used, so a lane's slots are in flight together.
//
// Root finding walks the larger of the two current nodes (labels decrease
// towards a root, so the larger one cannot be an ancestor of the other):
// meeting means one tree (Algorithm 1's label_1 == label_2, nothing to do);
// reaching a root at the larger node means two trees, and that root is
// linked by Algorithm 1's atomicMin loop under the other tree's root (link
// mode 0) or under the other chain's current node (link mode 1).

enum : int32_t { kTaskDone = 0, kTaskChase = 1, kTaskRoot = 2, kTaskMerge = 3 };

// Next state of a slot, 2 bits at index 4 * state + 2 * (y == a) + (y == b):
//   Done  -> Done;
//   Chase -> y == a: Root (link mode 0) or Merge (link mode 1);
//            else y == b: Done (one tree); else Chase;
//   Root  -> y == b: Merge; else Root;
//   Merge -> y == a or y == b: Done; else Merge.
constexpr uint32_t red_next_table(int link_mode) {
    uint32_t t = 0;
    for (uint32_t idx = 0; idx < 16; ++idx) {
        const uint32_t s = idx >> 2;
        const bool eq_a = (idx & 2u) != 0, eq_b = (idx & 1u) != 0;
        uint32_t nx = kTaskDone;
        if (s == kTaskChase) nx = eq_a ? (link_mode ? kTaskMerge : kTaskRoot) : (eq_b ? kTaskDone : kTaskChase);
        else if (s == kTaskRoot) nx = eq_b ? kTaskMerge : kTaskRoot;
        else if (s == kTaskMerge) nx = (eq_a || eq_b) ? kTaskDone : kTaskMerge;
        t |= nx << (2u * idx);
    }
    return t;
}
constexpr uint32_t kRedNextLink0 = red_next_table(0), kRedNextLink1 = red_next_table(1);


// Chase loads may be served from L1: a stale label is an older ancestor,
// which only lengthens a walk (labels only decrease), and every merge goes
// through an atomicMin whose returned value is current.
__device__ __forceinline__ int32_t red_load(const int32_t *p) { return __ldca(p); }

// Two ways of handing a window's pairs to the slots:
//  kStatic = false: every round, the warp's empty slots take the window's
//    next pairs in order (ballot + popc), which balances lanes whose chains
//    differ in length (randomly numbered trees);
//  kStatic = true: lane l serves pairs wbeg + l, wbeg + l + 32, ... and loads
//    its next pair a round before a slot needs it: fewer instructions per
//    round and no exposed queue load (lattices).
//
// The pairs are cut into windows inside each band, so a window's pairs are
// consecutive queue slots. Every CTA finds the windows of all bands by itself:
// s_win[b] = windows before band b, in dynamic shared memory, only as much as
// there are bands (the rest of the SM's memory is cache for the labels).
// Against one index space over all bands (8 KB of 64-bit prefix sums, a band
// look-up per pair): triangle 16384^2 1.46 -> 1.37 ms.
constexpr int kRedThreads = 256;

// Exclusive prefix sum of one value per thread over the CTA; *sum = the total.
__device__ __forceinline__ long long block_excl_scan(long long v, long long *s_warp, long long *sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    long long before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kRedThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        all += s_warp[w];
    }
    __syncthreads();
    *sum = all;
    return before + incl - v;
}

// Cuts the call's pairs into windows: fills s_win[0 .. n_bands], stores the
// statistics and returns the number of windows; total = all pairs. The whole
// CTA calls.
__device__ __forceinline__ uint32_t red_windows(const Params &P, uint32_t *s_win, long long *s_warp, int lane,
                                                long long nwarps, long long &total) {
    // Every warp takes as many windows as every other, the fewest that keeps
    // them below the limit: a last round of a few windows leaves the chip idle
    // (Bethe lattice of 24 shells, 5.5M pairs: 254 us with windows of 1024 pairs,
    // 1.1 rounds; 233 with two rounds). Bands round their window counts up, at
    // most one more each. At least 64 pairs.
    const auto window = [&](long long total) {
        const long long wmax = P.red_window > 0 ? P.red_window : kRedWindowMax;
        const long long room = max(nwarps - P.n_bands, nwarps / 2);
        const long long waves = max((total + room * wmax - 1) / (room * wmax), 1ll);
        return min(max((total + room * waves - 1) / (room * waves), 64ll), wmax);
    };
    if (P.n_bands <= 32) {
        // a small call: every warp by itself, without barriers (all write the
        // same values)
        const long long cnt = lane < P.n_bands ? (long long)P.band[lane].cnt : 0;
        total = cnt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
        const long long win = window(total);
        const int nw = (int)((cnt + win - 1) / win), upto = warp_incl_scan(nw, lane);
        if (lane < P.n_bands) s_win[lane + 1] = (uint32_t)upto;
        if (lane == 0) s_win[0] = 0;
        __syncwarp();
    } else {
        const int per = (P.n_bands + kRedThreads - 1) / kRedThreads;
        const int b0 = min((int)threadIdx.x * per, P.n_bands), b1 = min(b0 + per, P.n_bands);
        long long part = 0, sum;
        for (int b = b0; b < b1; ++b) part += (long long)P.band[b].cnt;
        block_excl_scan(part, s_warp, &total);
        const long long win = window(total);
        long long nw = 0;
        for (int b = b0; b < b1; ++b) nw += ((long long)P.band[b].cnt + win - 1) / win;
        long long acc = block_excl_scan(nw, s_warp, &sum);
        for (int b = b0; b < b1; ++b) {
            s_win[b] = (uint32_t)acc;
            acc += ((long long)P.band[b].cnt + win - 1) / win;
        }
        if (threadIdx.x == 0) s_win[P.n_bands] = (uint32_t)sum;
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // the call's statistics (a call in parts adds its later parts' pairs)
        if (P.more_pairs) P.counters[0] += (unsigned long long)total;
        else P.counters[0] = (unsigned long long)total;
    }
    return s_win[P.n_bands];
}

// Window w: its pairs and, batched, their instances.
struct RedWindow {
    const int2 *q;
    const int32_t *qk;
    int len;
};
template <bool kBatched>
__device__ __forceinline__ RedWindow red_window(const Params &P, const uint32_t *s_win, uint32_t w) {
    // its band: the last one with at most w windows before it (all lanes
    // search; smem broadcast)
    int band = 0;
    for (int hi = P.n_bands - 1; band < hi;) {
        const int mid = (band + hi + 1) >> 1;
        if (s_win[mid] <= w) band = mid; else hi = mid - 1;
    }
    // the band's pairs are spread evenly over its windows
    const long long cnt = (long long)P.band[band].cnt;
    const uint32_t before = s_win[band];
    const int wins = (int)(s_win[band + 1] - before);
    const long long most = (cnt + wins - 1) / wins;
    const long long beg = (long long)(w - before) * most;
    RedWindow r;
    r.len = (int)max(min(beg + most, cnt) - beg, 0ll);
    r.q = P.q + P.band[band].qbase + beg;
    r.qk = kBatched ? P.qk + P.band[band].qbase + beg : nullptr;
    return r;
}

// A batch with corrupt row pointers may emit more pairs than its rows have
// entries, and then a band's pairs and their instances are overwritten by
// another's, each by two stores. When an error is latched, every pair of a window
// is compared with its instance's size before it is followed, and one that does
// not fit becomes the pair (0, 0) of the first instance with sites. (A pair of
// one instance always fits.)
__device__ __forceinline__ void check_window(const Params &P, const RedWindow &w, int lane) {
    const int32_t first = find_inst_tile(P, 0);
    for (int e = lane; e < w.len; e += 32) {
        const int2 q = w.q[e];
        const int32_t k = w.qk[e];
        const uint32_t n = (uint32_t)k < (uint32_t)P.K ? (uint32_t)P.insts[k].n : 0u;
        if ((uint32_t)q.x < n && (uint32_t)q.y < n) continue;
        const_cast<int2 *>(w.q)[e] = make_int2(0, 0);
        const_cast<int32_t *>(w.qk)[e] = first;
    }
    __syncwarp();
}

// A pair needs at most 4n + 8 rounds (its chains and Algorithm 1's loop are
// bounded by the instance's n <= 32 n_chunks); a lane serves at most len pairs.
// Past this many rounds a window is abandoned with an error.
__device__ __forceinline__ long long red_round_cap(const Params &P, int len) {
    return P.iter_cap > 0 ? (long long)P.iter_cap : (128ll * P.n_chunks + 8) * (long long)len;
}

//
// kFar: the labels of a batch's instances lie anywhere, and a slot carries
// their address; else they lie within 2^32 labels from P.lab_base on, and a slot
// carries a 32-bit offset. That leaves registers for eight slots instead of
// six, and fewer warps with more slots keep the labels in use in the caches:
// 1024 mixed instances 2.53 ms (six slots with addresses, four CTAs per SM,
// windows of 512 pairs) -> 2.24 (eight with offsets, three CTAs, 1024; six with
// offsets: 2.37).
template <bool kBatched, bool kStatic, bool kFar>
__global__ void __launch_bounds__(kRedThreads, !kBatched ? 5 : kFar ? 4 : 3) k_reduce(Params P) {
    constexpr bool kOff = kBatched && !kFar;
    constexpr int kRedSlots = kOff ? 8 : 6;
    extern __shared__ uint32_t s_win[];             // [n_bands + 1]
    __shared__ long long s_warp[kRedThreads / 32];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long nwarps = (long long)gridDim.x * (kRedThreads / 32);
    long long total;
    const long long nwin = red_windows(P, s_win, s_warp, lane, nwarps, total);
    const unsigned latched = kBatched ? __ldcg(P.err) : 0u;
    // Few pairs: the clusters are small or tree-like (see `far` below).
    const bool few = !kBatched && kStatic && P.link_mode < 0 && total <= P.one.n / 4;
#ifdef CCL_DEVICE_STATS
    unsigned long long st_hops = 0, st_atom = 0, st_iter = 0;
#endif
    for (long long w = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < nwin; w += nwarps) {
        const RedWindow win = red_window<kBatched>(P, s_win, (uint32_t)w);
        if (kBatched && latched) check_window(P, win, lane);
        const int wlen = win.len;
        const int2 *wq = win.q;
        const int32_t *wqk = win.qk;
        const long long round_cap = red_round_cap(P, wlen);
        long long rounds = 0;
        int nxt = 0;        // pairs of the window handed to slots so far
        // kStatic: the lane's next pair, loaded ahead
        int pnext = lane;
        int2 pf = make_int2(0, 0);
        int pfk = 0;
        bool pf_ok = false;
        // batched: the labels of the lane's last instance (consecutive pairs
        // of a lane mostly come from one instance)
        int lk = 0;
        int32_t *llab = kFar ? P.insts[0].labels : nullptr;
        uint32_t loff = kOff ? (uint32_t)(P.insts[0].labels - P.lab_base) : 0u;
        // node x of slot u: its own address, or an offset from one base
        int32_t *const base = kBatched ? P.lab_base : P.one.labels;
        auto fetch = [&]() {
            pf = wq[pnext];
            if (kBatched) pfk = wqk[pnext];
            pf_ok = true;
            pnext += 32;
        };
        if (kStatic && pnext < wlen) fetch();
        // Link mode 1 (a root goes under the other chain's node, whose own root
        // need not be found) where it cannot build deep trees: an instance of
        // few pairs whose ends lie far apart in the numbering, a sixteenth of
        // the sites or more in half of the window's first 32 pairs. On randomly
        // numbered trees it saves a quarter of the loads (Bethe lattice of 24
        // shells at 0.5 / 1 / 1.5 p_c 71 / 235 / 498 -> 49 / 173 / 391 us); on
        // lattices it builds chains along the rows (triangle 4096^2 94 -> 613),
        // and on a random graph of 1.07 pairs per site 956 -> 1655.
        const bool far = few && __popc(__ballot_sync(kFull, pf_ok && abs(pf.x - pf.y) > P.one.n / 16)) >= 16;
        // (one copy of the loop per link choice: with the choice in a register
        // the common copy was 6 % slower)
        const auto drain = [&](const uint32_t table) {
            int32_t *L[kRedSlots];
            uint32_t off[kRedSlots];
            int32_t a[kRedSlots], b[kRedSlots], st[kRedSlots];
#pragma unroll
            for (int u = 0; u < kRedSlots; ++u) {
                st[u] = kTaskDone;
                L[u] = nullptr;
                off[u] = 0;
                a[u] = b[u] = 0;
            }
            for (;;) {
                if (kStatic) {
                    // at most one empty slot per lane and round takes the prefetched pair
                    int take = -1;
#pragma unroll
                    for (int u = kRedSlots - 1; u >= 0; --u)
                        if (st[u] == kTaskDone) take = u;
                    if (take >= 0 && pf_ok) {
                        const int32_t na = max(pf.x, pf.y), nb = min(pf.x, pf.y);
                        if (kBatched && pfk != lk) {
                            lk = pfk;
                            int32_t *l = P.insts[pfk].labels;
                            if (kFar) llab = l; else loff = (uint32_t)(l - base);
                        }
#pragma unroll
                        for (int u = 0; u < kRedSlots; ++u)
                            if (u == take) {
                                a[u] = na;
                                b[u] = nb;
                                st[u] = kTaskChase;
                                if (kFar) L[u] = llab;
                                if (kOff) off[u] = loff;
                            }
                        pf_ok = false;
                        if (pnext < wlen) fetch();
                    }
                } else {
                    // refill empty slots with the window's next pairs, in order (the
                    // tests are warp-uniform: nothing runs once the window is handed out)
                    if (nxt < wlen) {
#pragma unroll
                        for (int u = 0; u < kRedSlots; ++u) {
                            const unsigned need = __ballot_sync(kFull, st[u] == kTaskDone);
                            if (need == 0) continue;
                            const int pos = nxt + __popc(need & lt);
                            if (st[u] == kTaskDone && pos < wlen) {
                                const int2 pr = wq[pos];
                                if (kBatched) {
                                    const int k = wqk[pos];
                                    if (k != lk) {
                                        lk = k;
                                        int32_t *l = P.insts[k].labels;
                                        if (kFar) llab = l; else loff = (uint32_t)(l - base);
                                    }
                                    if (kFar) L[u] = llab;
                                    if (kOff) off[u] = loff;
                                }
                                a[u] = max(pr.x, pr.y);
                                b[u] = min(pr.x, pr.y);
                                st[u] = kTaskChase;
                            }
                            nxt = min(nxt + __popc(need), wlen);
                            if (nxt >= wlen) break;
                        }
                    }
                }
#ifdef CCL_DEVICE_STATS
                st_iter++;
#endif
                // issue: one load or one atomicMin per live slot
                int32_t v[kRedSlots];
#pragma unroll
                for (int u = 0; u < kRedSlots; ++u) {
                    const int32_t x = st[u] == kTaskRoot ? b[u] : a[u];
                    int32_t *ptr = kFar ? L[u] + x : base + (uint32_t)((kOff ? off[u] : 0u) + (uint32_t)x);
                    v[u] = 0;
                    if (st[u] == kTaskMerge) v[u] = atomicMin(ptr, b[u]);
                    else if (st[u] != kTaskDone) v[u] = red_load(ptr);
                }
                // use: the next state of every slot (no divergent paths). With
                // mx = max(y, b) and mn = min(y, b) every transition sets b = mn
                // and a = mx, except Root, which keeps a:
                //   Chase (y = label[a]): y == a means a root, so mx = a, mn = b;
                //     otherwise the walk goes on from the larger node;
                //   Root (y = label[b] <= b): b = y;
                //   Merge (y = old label[a]): Algorithm 1 continues with (old, b)
                //     when old > b and with (b, old) when old < b.
                // The next state is looked up by (state, y == a, y == b).
                bool any = false;
#pragma unroll
                for (int u = 0; u < kRedSlots; ++u) {
                    const int32_t y = v[u], A = a[u], Bv = b[u];
                    const int s = st[u];
#ifdef CCL_DEVICE_STATS
                    st_hops += (s == kTaskChase || s == kTaskRoot);
                    st_atom += (s == kTaskMerge);
#endif
                    const uint32_t idx = ((uint32_t)s << 2) | ((y == A) ? 2u : 0u) | ((y == Bv) ? 1u : 0u);
                    a[u] = s == kTaskRoot ? A : max(y, Bv);
                    b[u] = min(y, Bv);
                    st[u] = (int32_t)((table >> (2u * idx)) & 3u);
                    any |= st[u] != kTaskDone;
                }
                if (!__any_sync(kFull, any || pf_ok) && (kStatic || nxt >= wlen)) break;
                if (++rounds > round_cap) {
                    raise_err(P.err, kErrNonconv);
                    break;
                }
            }
        };
        if (far) drain(kRedNextLink1);
        else drain(P.link_mode > 0 ? kRedNextLink1 : kRedNextLink0);
    }
#ifdef CCL_DEVICE_STATS
    if (st_hops) atomicAdd(P.counters + 1, st_hops);
    if (st_atom) atomicAdd(P.counters + 2, st_atom);
    if (lane == 0 && st_iter) atomicAdd(P.counters + 3, st_iter);
#endif
}

// A window of k_reduce_park where the sample found chains so long that most pairs
// would be set aside: k_reduce's slots, three a lane, which walk only the larger
// node of a pair and so load half as much. Two walks at once / three slots (slots in
// k_reduce, as before there were short walks): honeycomb 1448^2 at 1.42 and 1.5 p_c
// 133 / 116 (124) and 140 / 111 (122) us a call, 2048^2 at 1.5 p_c 231 / 192 (205).
// The line: honeycomb 2400^2 at 1.36 p_c, one root in 16, takes 228 / 244, at 1.42,
// one in 26, 243 / 250 and 1750^2 there 157 / 148. Below 2M sites (1024^2 at 1.5 p_c
// 96) the caches hide the loads.
struct DeepCount {
    unsigned long long hops, atom, iter;        // (CCL_DEVICE_STATS)
};
__device__ __forceinline__ void drain_deep(const Params &P, const RedWindow &win, int lane, int32_t *labels,
                                           DeepCount &n) {
    constexpr int kSlots = 3;
    const uint32_t table = P.link_mode > 0 ? kRedNextLink1 : kRedNextLink0;
    const long long cap = red_round_cap(P, win.len);
    long long rounds = 0;
    int pnext = lane;
    int2 pf = make_int2(0, 0);
    bool pf_ok = false;
    const auto fetch = [&]() {
        pf = win.q[pnext];
        pf_ok = true;
        pnext += 32;
    };
    if (pnext < win.len) fetch();
    int32_t a[kSlots], b[kSlots], st[kSlots];
#pragma unroll
    for (int u = 0; u < kSlots; ++u) {
        st[u] = kTaskDone;
        a[u] = b[u] = 0;
    }
    for (;;) {
        int take = -1;          // at most one empty slot per lane and round takes the prefetched pair
#pragma unroll
        for (int u = kSlots - 1; u >= 0; --u)
            if (st[u] == kTaskDone) take = u;
        if (take >= 0 && pf_ok) {
            const int32_t na = max(pf.x, pf.y), nb = min(pf.x, pf.y);
#pragma unroll
            for (int u = 0; u < kSlots; ++u)
                if (u == take) {
                    a[u] = na;
                    b[u] = nb;
                    st[u] = kTaskChase;
                }
            pf_ok = false;
            if (pnext < win.len) fetch();
        }
        int32_t v[kSlots];
#pragma unroll
        for (int u = 0; u < kSlots; ++u) {
            int32_t *at = labels + (st[u] == kTaskRoot ? b[u] : a[u]);
            v[u] = 0;
            if (st[u] == kTaskMerge) v[u] = atomicMin(at, b[u]);
            else if (st[u] != kTaskDone) v[u] = red_load(at);
        }
        bool any = false;       // the transitions of k_reduce
#pragma unroll
        for (int u = 0; u < kSlots; ++u) {
            const int32_t y = v[u], A = a[u], B = b[u], s = st[u];
#ifdef CCL_DEVICE_STATS
            n.hops += (s == kTaskChase || s == kTaskRoot);
            n.atom += (s == kTaskMerge);
#endif
            const uint32_t idx = ((uint32_t)s << 2) | ((y == A) ? 2u : 0u) | ((y == B) ? 1u : 0u);
            a[u] = s == kTaskRoot ? A : max(y, B);
            b[u] = min(y, B);
            st[u] = (int32_t)((table >> (2u * idx)) & 3u);
            any |= st[u] != kTaskDone;
        }
#ifdef CCL_DEVICE_STATS
        n.iter++;
#endif
        if (!__any_sync(kFull, any || pf_ok)) break;
        if (++rounds > cap) {
            raise_err(P.err, kErrNonconv);
            break;
        }
    }
}

// Step (iii) for calls whose labels take at most three eighths of L2: two pairs
// a lane start together
// with their warp and run a fixed number of steps, both ends of a pair walking
// at once; the pairs whose ends are roots by then are linked by Algorithm 1's
// atomicMin, and what is not finished goes to a per-warp list in shared memory,
// 32 of which at a time, one per lane, run on. The code of a step is a fraction
// of k_reduce's (no slot to choose, no state table), the first steps of
// consecutive pairs stay coalesced, and few pairs need more: honeycomb 256^2
// 28 -> 21 us, 256 small instances 39 -> 24, honeycomb 2048^2 66 -> 43, cubic
// 200^3 33 -> 30. It loads more labels than k_reduce (which walks only the
// larger node). At half of L2 the two are even (triangle 4096^2 94 -> 85,
// honeycomb 2896^2 at 1.25 p_c 131 -> 147), beyond L2 the loads cost more than
// the code saves (triangle 16384^2 1.37 -> 1.91 ms, 1024 mixed instances
// 2.53 -> 3.07).
constexpr int kParkSteps = 4;                   // steps before a pair is set aside
constexpr int kParkPairs = 2;                   // pairs a lane starts together
constexpr int kParkList = 64;                   // < 32 left + one pair per lane
template <bool kBatched>
__global__ void __launch_bounds__(kRedThreads, kBatched ? 6 : 8) k_reduce_park(Params P) {
    extern __shared__ uint32_t s_win[];             // [n_bands + 1]
    __shared__ long long s_warp[kRedThreads / 32];
    __shared__ int2 s_pair[kRedThreads / 32][kParkList];
    __shared__ int s_k[kBatched ? kRedThreads / 32 : 1][kBatched ? kParkList : 1];
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const long long nwarps = (long long)gridDim.x * (kRedThreads / 32);
    long long total;
    const long long nwin = red_windows(P, s_win, s_warp, lane, nwarps, total);
    const unsigned latched = kBatched ? __ldcg(P.err) : 0u;
    const bool deep = !kBatched && P.deep && __ldcg(P.deep);
    const bool eager = P.link_mode > 0;            // link a root to the other end's node, not its root
    // the labels of the lane's last instance
    int lk = -1;
    int32_t *llab = P.one.labels;
#ifdef CCL_DEVICE_STATS
    unsigned long long st_hops = 0, st_atom = 0, st_iter = 0;
#endif
    struct Pair {
        int32_t a, b;
        bool ra, rb, act;           // a, b are roots; the pair is not done
    };
    const auto step = [&](Pair &p, const int32_t *L) {
        int32_t ya = p.a, yb = p.b;
        if (p.act && !p.ra) ya = red_load(L + p.a);
        if (p.act && !p.rb) yb = red_load(L + p.b);
#ifdef CCL_DEVICE_STATS
        st_hops += (p.act && !p.ra) + (p.act && !p.rb);
#endif
        p.ra = ya == p.a;
        p.rb = yb == p.b;
        p.a = ya;
        p.b = yb;
        p.act = p.act && ya != yb;
    };
    const auto link = [&](Pair &p, int32_t *L) {
        const int32_t hi = max(p.a, p.b), lo = min(p.a, p.b);
        if (p.act && (eager ? (p.a > p.b ? p.ra : p.rb) : (p.ra && p.rb))) {
            // old == hi: linked; old == lo: linked already; else Algorithm 1
            // goes on with the displaced label
            const int32_t old = atomicMin(L + hi, lo);
#ifdef CCL_DEVICE_STATS
            ++st_atom;
#endif
            p.act = old != hi && old != lo;
            p.a = old;
            p.b = lo;
            p.ra = p.rb = false;
        }
    };
    for (long long w = (long long)blockIdx.x * (kRedThreads / 32) + warp; w < nwin; w += nwarps) {
        const RedWindow win = red_window<kBatched>(P, s_win, (uint32_t)w);
        if (kBatched && latched) check_window(P, win, lane);
        if (!kBatched && deep) {
            DeepCount n{0, 0, 0};
            drain_deep(P, win, lane, P.one.labels, n);
#ifdef CCL_DEVICE_STATS
            st_hops += n.hops;
            st_atom += n.atom;
            st_iter += n.iter;
#endif
            continue;
        }
        const int round_cap = (int)min(red_round_cap(P, win.len), (long long)INT32_MAX - 3);
        int rounds = 0;
        int cnt = 0;                // pairs set aside; below 32 whenever pairs are added
        const auto set_aside = [&](const Pair &p, int k) {
            const unsigned m = __ballot_sync(kFull, p.act);
            if (m == 0) return;
            if (p.act) {
                const int pos = cnt + __popc(m & lt);
                s_pair[warp][pos] = make_int2(p.a, p.b);
                if (kBatched) s_k[warp][pos] = k;
            }
            cnt += __popc(m);
            __syncwarp();
        };
        // runs up to 32 of the set-aside pairs on: a few steps, or to the end
        const auto resume = [&](bool to_end) {
            const int take = min(cnt, 32);
            cnt -= take;
            Pair p{0, 0, false, false, lane < take};
            int k = 0;
            if (p.act) {
                const int2 q = s_pair[warp][cnt + lane];
                if (kBatched) k = s_k[warp][cnt + lane];
                p.a = q.x;
                p.b = q.y;
            }
            int32_t *L = kBatched ? P.insts[k].labels : P.one.labels;
            __syncwarp();
            for (int it = 0; to_end || it < 2; ++it) {
#ifdef CCL_DEVICE_STATS
                st_iter += 2;
#endif
                step(p, L);
                step(p, L);
                link(p, L);
                if (!__any_sync(kFull, p.act)) return;
                if ((rounds += 3) > round_cap) {        // the pairs are dropped
                    raise_err(P.err, kErrNonconv);
                    return;
                }
            }
            set_aside(p, k);
        };
        for (int p0 = lane; p0 - lane < win.len; p0 += 32 * kParkPairs) {
            Pair pr[kParkPairs];
            int k[kParkPairs];
            int32_t *L[kParkPairs];
#pragma unroll
            for (int u = 0; u < kParkPairs; ++u) {
                pr[u] = Pair{0, 0, false, false, p0 + 32 * u < win.len};
                k[u] = 0;
                if (pr[u].act) {
                    const int2 q = win.q[p0 + 32 * u];
                    if (kBatched) k[u] = win.qk[p0 + 32 * u];
                    pr[u].a = q.x;
                    pr[u].b = q.y;
                }
            }
#pragma unroll
            for (int u = 0; u < kParkPairs; ++u) {
                if (kBatched && k[u] != lk) { lk = k[u]; llab = P.insts[lk].labels; }
                L[u] = kBatched ? llab : P.one.labels;
            }
#ifdef CCL_DEVICE_STATS
            st_iter += kParkSteps;
#endif
#pragma unroll
            for (int r = 0; r < kParkSteps; ++r)
#pragma unroll
                for (int u = 0; u < kParkPairs; ++u) step(pr[u], L[u]);
#pragma unroll
            for (int u = 0; u < kParkPairs; ++u) link(pr[u], L[u]);
#pragma unroll
            for (int u = 0; u < kParkPairs; ++u) {
                set_aside(pr[u], k[u]);
                while (cnt >= 32) resume(false);        // (every step shortens a walk: this ends)
            }
        }
        while (cnt > 0) resume(true);
    }
#ifdef CCL_DEVICE_STATS
    if (st_hops) atomicAdd(P.counters + 1, st_hops);
    if (st_atom) atomicAdd(P.counters + 2, st_atom);
    if (lane == 0 && st_iter) atomicAdd(P.counters + 3, st_iter);
#endif
}

// ---------------------------------------------------------------------------
// Input check for ccl_validate: one thread per site. (Only the translation
// unit that implements ccl_validate defines it.)

#ifndef CCL_NO_VALIDATE_KERNEL
__global__ void k_validate(int32_t n, int64_t nnz, const int32_t *__restrict__ row_ptr,
                           const int32_t *__restrict__ col_idx, const uint32_t *__restrict__ bits,
                           unsigned *err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t ii = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; ii < n; ii += stride) {
        const int32_t i = (int32_t)ii;
        const int32_t a = row_ptr[i], b = row_ptr[i + 1];
        if (i == 0 && a != 0) raise_err(err, kErrShape);
        if (i == n - 1 && b != nnz) raise_err(err, kErrShape);
        if (a < 0 || b < a || b > nnz) { raise_err(err, kErrIndex); continue; }
        for (int32_t e = a; e < b; ++e) {
            const int32_t j = col_idx[e];
            if ((uint32_t)j >= (uint32_t)n) { raise_err(err, kErrIndex); continue; }
            if (j == i) continue;
            const uint32_t bit = (bits[e >> 5] >> (e & 31)) & 1u;
            const int32_t c0 = row_ptr[j], c1 = row_ptr[j + 1];
            if (c0 < 0 || c1 < c0 || c1 > nnz) { raise_err(err, kErrIndex); continue; }
            bool found = false;
            for (int32_t f = c0; f < c1 && !found; ++f) {
                if (col_idx[f] == i && (((bits[f >> 5] >> (f & 31)) & 1u) == bit)) found = true;
            }
            if (!found) raise_err(err, kErrAsym);
        }
    }
}
#endif  // CCL_NO_VALIDATE_KERNEL

}  // namespace ccl
