// Device building blocks of windowed median / MAD excision (Section II-D, Eq. 1 and Eq. 2).
//
// One data window of n samples lies in shared memory (sample 0 at a 16-byte aligned address).
// A thread group of T threads (the consumer warps of a CTA) processes it in five phases:
//   1. histogram   h[v] = #{i : x_i = v}, exact u32 counts in shared memory
//   2. reduce      fold the privatised histogram copies into one count per bin
//   3. scan        C[v] = sum_{u <= v} h[u] (block-wide prefix sum)
//   4. search      M = smallest v with C[v] >= ceil(n/2)                       (lower median)
//                  D = smallest d with C[M+d] - C[M-d-1] >= ceil(n/2)           (lower MAD)
//                  The second line is the cumulative histogram of |x - M| written through C:
//                  #{|x_i - M| <= d} = C[M+d] - C[M-d-1], so the |x - M| histogram is never
//                  materialised.
//   5. replace     t = ceil(Kq*D / 2^16); x is flagged iff D > 0 and |x - M| >= t, which is
//                  Eq. 2 (x >= tau_U or x <= tau_L) for integer x with Kq = round(k*1.4826*2^16);
//                  flagged samples get the replacement value, the mask bit and the count.
//
// 8-bit samples use a lane-striped histogram: the count of raw byte value u (the int8 sample
// read as unsigned) for lane l is word u*32 + l, so the 32 lanes of a warp always hit 32
// different banks and 32 different words; warps share the table through shared-memory
// atomics, and the reduce phase reads row u into logical bin u ^ 128 = x + 128. 12-bit
// samples use 1, 2 or 4 plain copies of a 4096-bin table selected by lane, of which only the
// totals of 256 rows of 16 bins are scanned (phase_rows12, phase_search12). One warp searches the
// cumulative counts for M and D and broadcasts the threshold and replacement values through
// shared memory.
//
// The int8 replace pass works on four samples per 32-bit word: a native byte absolute
// difference, a three-operation byte compare against t, a byte permute that replicates each
// byte's flag bit into 0x00/0xFF, and a byte dot product that packs the flags into mask bits.
//
// Digital-noise replacement is deferred and shared out over the group, in one of two ways
// chosen by sample width for the flag densities each one serves best. int8 (sparse, bursty
// flags): the replace pass lists the chunks that hold a flagged sample with their flag masks;
// after a group barrier the warps share out the list two chunks at a time, expand each mask
// over a half-warp into a per-warp queue of positions, and evaluate Philox whenever 32 are
// queued, so every lane of a batch has a sample. 12-bit (dense flags): the replace pass writes
// the flagged samples' positions into a per-group list, and after one more group barrier all
// threads evaluate Philox for the list, in slices of 8192 samples where a whole window's flags would
// not fit; what a list has no room for goes through a per-warp path that numbers the samples across
// the warp.
//
// Small int8 windows (2^l = 512..8192 samples) can go several to a table (process_tile_multi8):
// window slot g of a tile is counted by its own group of lanes, so up to eight windows share one
// reduce, one set of barriers and searches on separate warps. The in-place form that writes
// back only what changes skips the stores of chunks without a flagged sample (phase_replace's
// FO parameter).

#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace rfi {
namespace dev {

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void red_add_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

__device__ __forceinline__ void named_bar(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Named barrier that also returns whether any participating thread passed v = true.
__device__ __forceinline__ bool named_bar_or(int id, int nthreads, bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(v)), "r"(id), "r"(nthreads)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t tx) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar),
        "r"(tx)
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// try_wait that lets the hardware suspend the thread for up to ~2 us while the phase is open,
// so a waiting warp does not take issue slots from the warps doing work.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(2000u)
        : "memory");
    return ok != 0;
}

// Wait for the phase of the given parity, giving up after timeout_ns of wall time (and after
// a fixed number of polls in any case). Returns false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint64_t timeout_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1; it < (1u << 24); ++it) {
        if (mbar_try_wait_sleep(bar, parity)) return true;
        if ((it & 7u) == 0 && global_timer_ns() - t0 > timeout_ns) return false;
    }
    return false;
}

// Bulk (non-tensor) asynchronous copy global -> shared, completing on an mbarrier.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// ------------------------------------------------------------------ Philox4x32-10 noise
// Philox4x32-10 as defined by Salmon, Moraes, Dror and Shaw (SC'11): ten rounds; in each the
// words 0 and 2 are multiplied by the two round multipliers, the high product halves are
// xor-ed with words 1 and 3 and with the round key. Round r uses the key advanced by r Weyl
// increments, which a key source gives: precomputed in the kernel parameters (KeysPre), or
// derived from the seed on the fly (KeysSeed, for the per-variant seeds of a digital copy).
struct KeysPre {
    const Params &p;  // the kernel's own parameters: indexed with constants, read in place
    __device__ __forceinline__ uint32_t a(int r) const { return p.rk0[r]; }
    __device__ __forceinline__ uint32_t b(int r) const { return p.rk1[r]; }
};
struct KeysSeed {
    uint32_t s0, s1;
    __device__ __forceinline__ uint32_t a(int r) const { return s0 + static_cast<uint32_t>(r) * 0x9E3779B9u; }
    __device__ __forceinline__ uint32_t b(int r) const { return s1 + static_cast<uint32_t>(r) * 0xBB67AE85u; }
};

// Digital-noise replacement: M + round_half_away(S2 * sigq / (107020 * 2^16)), sigq = 97164*D,
// S2 = 2 * s - 8 * 65535 with s the sum of the eight 16-bit halves of the Philox output at counter
// (idx_lo, idx_hi, stream, 0). It goes in two steps: noise_sum gives s, NoiseScale the value.

// What the first two rounds compute from the stream and the index's high word alone: round 1's
// second product (of the stream) and round 2's first product (of a word that holds no idx_lo).
struct NoiseKey {
    uint32_t a, b, c;  // round 2: z = a ^ (low product of round 1), x = b ^ ...; round 3: z = c ^ ...
    NoiseKey() = default;
    template <class K>
    __device__ __forceinline__ NoiseKey(const K &key, uint32_t sid, uint32_t idx_hi) {
        const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * sid;
        const uint32_t x = static_cast<uint32_t>(p1 >> 32) ^ idx_hi ^ key.a(0);
        const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * x;
        a = static_cast<uint32_t>(p0 >> 32) ^ key.b(1);
        b = static_cast<uint32_t>(p1) ^ key.a(1);
        c = static_cast<uint32_t>(p0) ^ key.b(2);
    }
};

// s of sample index idx_lo: 18 products instead of 20.
template <class K>
__device__ __forceinline__ uint32_t noise_sum(const NoiseKey &nk, const K &key, uint32_t idx_lo) {
    uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * idx_lo;                                          // round 1
    uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * (static_cast<uint32_t>(p0 >> 32) ^ key.b(0));    // round 2
    uint4 c;
    c.x = static_cast<uint32_t>(p1 >> 32) ^ nk.b;
    c.y = static_cast<uint32_t>(p1);
    c.z = nk.a ^ static_cast<uint32_t>(p0);
    p0 = static_cast<uint64_t>(0xD2511F53u) * c.x;  // round 3
    p1 = static_cast<uint64_t>(0xCD9E8D57u) * c.z;
    c = make_uint4(static_cast<uint32_t>(p1 >> 32) ^ c.y ^ key.a(2), static_cast<uint32_t>(p1),
                   static_cast<uint32_t>(p0 >> 32) ^ nk.c, static_cast<uint32_t>(p0));
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        // one 32 x 32 -> 64-bit product per multiplier gives both halves
        p0 = static_cast<uint64_t>(0xD2511F53u) * c.x;
        p1 = static_cast<uint64_t>(0xCD9E8D57u) * c.z;
        c = make_uint4(static_cast<uint32_t>(p1 >> 32) ^ c.y ^ key.a(r), static_cast<uint32_t>(p1),
                       static_cast<uint32_t>(p0 >> 32) ^ c.w ^ key.b(r), static_cast<uint32_t>(p0));
    }
    // each dp2a adds both halves of one word (weights 1, 1)
    return __dp2a_lo(c.x, 0x0101u, __dp2a_lo(c.y, 0x0101u, __dp2a_lo(c.z, 0x0101u, __dp2a_lo(c.w, 0x0101u, 0u))));
}

// The value of a sum s in a window with median M and dispersion D, saturated to the sample range:
// M + floor((S2 * sigq + den / 2) / den), den = 107020 * 2^16, with OFF * den added to keep the
// dividend positive (OFF is above the largest offset, 524280 * 97164 * D / den). The window gives
// sig2 = 2 * sigq and moff = M - OFF. The dividend is below 2^49; dividing by 2^16 (12-bit: 2^17, to
// stay in 32 bits) first and then by the rest of den equals one division, which is the high word of
// the product with ceil(2^48 / 107020), shifted (exact for quotients of these ranges: the product's
// excess over the true one stays below one). Rounding a half up instead of away from zero differs
// only at an exact tie, that is |S2| * D = 2^15 * 26755: an offset of 12145.5, which no sample range
// holds. A 32 x 32 -> 64-bit product runs at 64 lanes a clock and SM here; with a 64-bit addend it
// runs at 25 and the high-word product at 32 (measured), hence the separate additions.
template <int BITS>
struct NoiseScale {
    static constexpr int32_t kOff = BITS == 8 ? 2048 : 30000;
    static constexpr int32_t kSig2 = 2 * 97164;
    __device__ __forceinline__ static int32_t value(uint32_t s, int32_t sig2, int32_t moff) {
        constexpr uint64_t kDen = 107020ull << 16;
        constexpr uint64_t kAdd = kOff * kDen + kDen / 2;
        constexpr int kShift = BITS == 8 ? 16 : 17;
        constexpr int kLo = BITS == 8 ? -128 : -2048, kHi = BITS == 8 ? 127 : 2047;
        uint32_t lo, hi, q;
        asm("{\n\t.reg .b64 t;\n\tmul.wide.s32 t, %2, %3;\n\tmov.b64 {%0, %1}, t;\n\t}"
            : "=r"(lo), "=r"(hi) : "r"(static_cast<int32_t>(s) - 262140), "r"(sig2));
        asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
            : "+r"(lo), "+r"(hi) : "r"(static_cast<uint32_t>(kAdd)), "r"(static_cast<uint32_t>(kAdd >> 32)));
        const uint32_t n = __funnelshift_r(lo, hi, kShift);
        asm("{\n\t.reg .b64 t;\n\t.reg .b32 u;\n\tmul.wide.u32 t, %1, %2;\n\tmov.b64 {u, %0}, t;\n\t}"
            : "=r"(q) : "r"(n), "r"(2630115649u));
        const int32_t v = static_cast<int32_t>(q >> (32 - kShift)) + moff;
        return v < kLo ? kLo : (v > kHi ? kHi : v);
    }
};

// A tile's noise words, computed by the copy warp when it stages the tile: every thread of the
// group computing them per window costs as much as they save on a window with few flags.
struct TileNoise {
    NoiseKey nk;
    uint32_t one_hi;  // every index of the tile has the same high word
};

// Noise over a run of samples of one stream starting at absolute index abs0: value(pos, sig2, moff)
// for sample abs0 + pos. The words that the samples share are computed once where the run's
// indices have one high word (every run but one across a multiple of 2^32).
template <int BITS, class K>
struct NoiseRun {
    const K &key;
    NoiseKey nk;
    uint64_t abs0;
    uint32_t sid;
    bool one_hi;
    __device__ __forceinline__ NoiseRun(const K &k, uint32_t stream, uint64_t a0, uint64_t n)
        : key(k), nk(k, stream, static_cast<uint32_t>(a0 >> 32)), abs0(a0), sid(stream),
          one_hi(((a0 ^ (a0 + n - 1)) >> 32) == 0) {}
    // the words as the tile's copy warp left them (TileNoise)
    __device__ __forceinline__ NoiseRun(const K &k, uint32_t stream, uint64_t a0, const TileNoise &t)
        : key(k), nk(t.nk), abs0(a0), sid(stream), one_hi(t.one_hi != 0u) {}
    // one_hi runs; a branch to the general form here costs 2 % of a call, so the loops below have a
    // general twin instead
    __device__ __forceinline__ uint32_t sum(uint32_t pos) const {
        return noise_sum(nk, key, static_cast<uint32_t>(abs0) + pos);
    }
    __device__ __forceinline__ int32_t value(uint32_t pos, int32_t sig2, int32_t moff) const {
        return NoiseScale<BITS>::value(sum(pos), sig2, moff);
    }
    // two samples at a time: their Philox chains are independent and interleave
    __device__ __forceinline__ int2 value2(uint32_t pa, uint32_t pb, int32_t sig2, int32_t moff) const {
        const uint32_t a = sum(pa), b = sum(pb);
        return make_int2(NoiseScale<BITS>::value(a, sig2, moff), NoiseScale<BITS>::value(b, sig2, moff));
    }
    // any run
    __device__ __forceinline__ int32_t value_any(uint32_t pos, int32_t sig2, int32_t moff) const {
        const uint64_t idx = abs0 + pos;
        return NoiseScale<BITS>::value(
            noise_sum(NoiseKey(key, sid, static_cast<uint32_t>(idx >> 32)), key, static_cast<uint32_t>(idx)), sig2, moff);
    }
};

// ------------------------------------------------------------------ shared-memory layout
template <int BITS>
struct Geo {
    static constexpr int kBins = BITS == 8 ? 256 : 4096;
    static constexpr int kOffset = BITS == 8 ? 128 : 2048;  // logical bin = x + kOffset
    static constexpr int kBps = BITS == 8 ? 1 : 2;          // bytes per sample
    static constexpr int kLo = BITS == 8 ? -128 : -2048;
    static constexpr int kHi = BITS == 8 ? 127 : 2047;
    // 8-bit: 256 cumulative counts (264 words: the distance of two multi-window slots' 16-bit counts);
    // 12-bit: the histogram's second table
    static constexpr int kCumWords = BITS == 8 ? kBins + kBins / 32 : kBins;
    static constexpr int kChunkSamples = 16 / kBps;          // samples per 16-byte chunk
    // 8-bit, one consumer group: a 32 KiB table of 128-byte rows (raw byte u -> row u, lane l
    // -> word l). 8-bit, two groups: one 64 KiB table of 256-byte rows shared by both (group g
    // owns bytes [128g, 128g + 128) of every row). 12-bit: ncopies tables of 4096 words per group
    // (copy 0 of the even windows, then the other copies).
    __host__ __device__ static constexpr int hist_bytes(int ncopies, int groups) {
        return BITS == 8 ? (groups == 2 ? 65536 : 32768) : kBins * 4 * ncopies * groups;
    }
    __host__ __device__ static constexpr int row_bytes(int groups) { return groups == 2 ? 256 : 128; }
};

// Shared-window address of the first byte of dynamic shared memory. The 8-bit histogram sits
// there and its atomics use it as an immediate offset; kernels check it at entry.
constexpr uint32_t kDynSmemShared = 1024;

struct __align__(16) RepShared {
    int32_t M, D, t, hiv, lov;
    uint32_t active;
    int32_t sig2, moff;  // digital noise (NoiseScale)
    // int8 replace constants (see Rep8)
    uint32_t mb4, tlo7, tsmall, c4, hi4, lo4, ulo7, usmall;
    uint32_t unone;
    int32_t cval;  // constant replacement (saturated)
    uint32_t pad2[2];
};

// Digital copy only (its own region, so that other kernels keep their shared-memory size).
struct CopyShared {
    RepShared vrep[kMaxCopies];        // threshold and replacement values per variant
    uint32_t vcount[kMaxCopies][2];    // flagged samples, by variant and window parity
    uint32_t ncount[4 * kMaxCopies];   // digital-noise list entries, by variant, parity and slice
};

// Digital copy, int8: what the variants of one threshold multiple share a pass with (copies_pass8). It lies
// over the cumulative counts, which are idle from the search to the next window's reduce, so that
// copies take no more shared memory for it.
struct CopyPass {
    uint8_t *out[kMaxCopies];          // the window's output and mask, by variant
    uint16_t *mask[kMaxCopies];
    uint32_t group[kMaxCopies];        // bit u: variant u has the same multiple
    uint32_t mode[kMaxCopies];         // rfi_mode
    uint32_t fast;                     // the window goes through copies_pass8
};
static_assert(sizeof(CopyPass) <= 256 * 4, "over the cumulative counts");

// Apply passes over whole tiles: the thresholds and flag counts of the tile's windows.
struct ApplyTile {
    RepShared rep[kApplyTileWindows];
    uint32_t count[kApplyTileWindows];
};

// Multi-window tiles (8-bit, one consumer group): up to K (4 or 8) small windows are
// histogrammed at once, window slot g in lanes (32/K)g .. (32/K)(g+1)-1 of the lane-striped
// table, so that one reduce, one set of barriers and parallel searches serve them all. Their
// cumulative counts (at most 8192, the largest window of this form) are 16-bit: slot g's 256
// entries at (uint16_t *)cum + g * kCumWords.
constexpr int kMultiMax = 8;
struct MultiTile {
    RepShared rep[kMultiMax];
    uint32_t count[kMultiMax];
};

struct Ctl {
    RepShared rep;       // threshold and replacement values of the current window
    uint32_t count[2];   // flagged samples, by window parity
    uint32_t done[2];    // warps finished with the window, by window parity
    uint32_t err[2];     // 12-bit range error seen in the window, by window parity
    uint32_t ncount[4];  // digital-noise list entries, by window parity (and slice of the window, 12-bit)
    unsigned long long pw[2][2];  // power-metered excision: {sum x^2, sum z^2}, by window parity
    uint32_t abort;      // set when any warp gave up on a bounded wait
    int32_t wide;        // 12-bit noise: the window before had few enough flags for one list
    unsigned long long flagged;  // group total
};

// Per-thread running row sums of the 8-bit histogram (the table is never cleared: a window's
// count of a bin is the difference of two consecutive sums, exact modulo 2^32).
struct RowSums {
    uint32_t s[2];
};

// Per-CTA view of the shared-memory regions used by window processing.
struct Shm {
    uint8_t *hist;       // histogram (generic pointer; 8-bit: the 64 KiB table)
    uint32_t hist_s;     // histogram (shared address)
    uint32_t grp;        // 8-bit: byte offset of this group's half row (0 or 128)
    uint32_t *cum;       // cumulative counts; 12-bit: the histogram's second table (table12)
    uint32_t *coarse;    // 12-bit estimation pass: the rows' cumulative counts (or null: phase_rows12)
    Ctl *ctl;
    int ncopies;         // 12-bit only
    int bar_id;          // named barrier of this consumer group
    CopyShared *cp;      // digital copy: per-variant state (or null)
    CopyPass *pass;      // digital copy, int8: the state of shared passes (or null)
    uint16_t *nlist;     // digital noise work area (or null): int8, the entries of the chunks that
                         // hold flagged samples (32-bit); 12-bit, the positions of flagged samples
    uint32_t *nring;     // int8 digital noise: kNoiseRingBytes per consumer warp (or null)
    ApplyTile *at;       // apply passes: the current tile's thresholds and counts (or null)
    struct MultiTile *mt;  // 8-bit, one group: state of a multi-window tile (or null)
};

// Capacity of the 12-bit digital-noise list (16-bit positions in a window of up to 65536 samples).
constexpr int kNoiseList = 4096;
// 12-bit digital noise goes through a window in slices of this many chunks (8192 samples; in the
// any-window form 33 rounds of 31 chunks), so that the list serves slices with up to half their samples
// flagged whatever the window's length.
constexpr int kNoiseSlice = 1024, kNoiseSliceAny = 1023;
// Positions a warp's ring holds: fewer than a batch wait between two batches (64 positions where a lane
// takes two at a time, else 32), and one expansion step adds at most 32. Two at a time: the plain
// kernel and the output formats; in the kernels with multi-window tiles or several variants the
// registers it takes cost more than the overlap gives.
__host__ __device__ constexpr bool noise_pairs(int mode) { return (mode & (kModeMulti | kModeAny | kModeApply | kModeCopies | kModePower)) == 0; }
// Bytes of a warp's ring: 128 positions of 16 bits (a window's samples) or 64 of 32 bits.
constexpr int kNoiseRingBytes = 256;

// Per-thread sums of x^2 and z^2 of the power-metered excision. A thread sees at most
// 65536 / 128 samples of a window, each below 2^22, so 32 bits hold its sums.
struct Pow {
    uint32_t x, z;
};

// One window to process.
struct Win {
    const uint8_t *data;  // shared memory, 16-byte aligned, sample 0 at byte off
    int32_t n;            // samples
    uint8_t *out;         // global output of sample 0
    uint32_t *mask;       // global mask block (nullable)
    int32_t mask_words;   // ceil(W / 32)
    int64_t abs_idx;      // absolute stream index of sample 0
    uint32_t sid;
    bool vec;             // out is 16-byte aligned: vector stores
    int32_t off;          // any-window form: bytes of data before sample 0 (0..15); else 0
    const TileNoise *tn;  // the tile's noise words (digital noise with the kernel's own key; else null)
    // noise of this window
    template <int BITS, class K>
    __device__ __forceinline__ NoiseRun<BITS, K> noise(const K &key) const {
        if constexpr (std::is_same<K, KeysPre>::value) {
            if (tn) return NoiseRun<BITS, K>(key, sid, static_cast<uint64_t>(abs_idx), *tn);
        }
        return NoiseRun<BITS, K>(key, sid, static_cast<uint64_t>(abs_idx), static_cast<uint64_t>(n));
    }
};

// ------------------------------------------------------------------ phase 1: histogram
// Shared atomic at histogram address kDynSmemShared + a.
__device__ __forceinline__ void red_hist8(uint32_t a) {
    asm volatile("red.shared.add.u32 [%0+1024], %1;" ::"r"(a), "r"(1u));
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// Four int8 samples.
// 256-byte rows: lp = 128*group + 4*lane; the table offset of raw byte u is u*256 + lp, which one
// byte permute assembles (byte 0 from lp, byte 1 = sample byte j, bytes 2-3 zero).
// 128-byte rows: lp = shared address of the table + 4*lane; the address is lp + u*128.
template <int ROWB>
__device__ __forceinline__ void hist8_word(uint32_t lp, uint32_t w) {
    static_assert(kDynSmemShared == 1024, "immediate offset of red_hist8");
    if (ROWB == 256) {
        red_hist8(prmt(w, lp, 0x5504u));
        red_hist8(prmt(w, lp, 0x5514u));
        red_hist8(prmt(w, lp, 0x5524u));
        red_hist8(prmt(w, lp, 0x5534u));
    } else {
        red_add_shared(lp + ((w & 0xFFu) << 7), 1u);
        red_add_shared(lp + (prmt(w, 0u, 0x4441u) << 7), 1u);
        red_add_shared(lp + (prmt(w, 0u, 0x4442u) << 7), 1u);
        red_add_shared(lp + ((w >> 24) << 7), 1u);
    }
}

// 12-bit histogram tables: copy 0 has one for the even and one for the odd windows, so that a window's
// table can be cleared while the next one's is in use; the other copies are folded into copy 0 and
// cleared before the next window.
__device__ __forceinline__ uint32_t *table12(const Shm &sm, int par) {
    return par ? sm.cum : reinterpret_cast<uint32_t *>(sm.hist);
}
__device__ __forceinline__ uint32_t copy12(const Shm &sm, int c, int par) {
    return c == 0 ? smem_addr(table12(sm, par)) : sm.hist_s + static_cast<uint32_t>(c) * 16384u;
}

// Two 12-bit samples in int16 halves. The bin x + 2048 of an in-range sample is its low 12 bits
// with bit 11 flipped; the upper half's bin sits 14 bits above its table offset. A half is in range
// iff its bits 15..11 are all equal: the caller collects w ^ (w << 1) and looks at its bits
// 0xF000F000 (kRange12) once.
constexpr uint32_t kRange12 = 0xF000F000u;
__device__ __forceinline__ void hist12_word(uint32_t copy_base, uint32_t w) {
    const uint32_t u = (w ^ 0x08000800u) & 0x0FFF0FFFu;
    red_add_shared(copy_base + ((u & 0xFFFFu) << 2), 1u);
    red_add_shared(copy_base + (u >> 14), 1u);
}

__device__ __forceinline__ uint32_t range12_bits(uint32_t w) { return w ^ (w + w); }

template <int BITS, int T, int ROWB>
__device__ __forceinline__ void phase_histogram(const Shm &sm, const Win &w, int tid, int par) {
    const int lane = tid & 31;
    const int nbytes = w.n * Geo<BITS>::kBps;
    const int nfull = nbytes >> 4;
    const uint4 *d4 = reinterpret_cast<const uint4 *>(w.data);
    if (BITS == 8) {
        const uint32_t lb = (ROWB == 256 ? sm.grp : sm.hist_s) + 4u * lane;
        int c = tid;
        for (; c + T < nfull; c += 2 * T) {
            const uint4 a = d4[c], b = d4[c + T];
            hist8_word<ROWB>(lb, a.x); hist8_word<ROWB>(lb, a.y); hist8_word<ROWB>(lb, a.z); hist8_word<ROWB>(lb, a.w);
            hist8_word<ROWB>(lb, b.x); hist8_word<ROWB>(lb, b.y); hist8_word<ROWB>(lb, b.z); hist8_word<ROWB>(lb, b.w);
        }
        if (c < nfull) {
            const uint4 a = d4[c];
            hist8_word<ROWB>(lb, a.x); hist8_word<ROWB>(lb, a.y); hist8_word<ROWB>(lb, a.z); hist8_word<ROWB>(lb, a.w);
        }
        const int rem = nbytes & 15;
        if (tid < rem) {
            const uint32_t u = static_cast<uint32_t>(w.data[nfull * 16 + tid]);
            if (ROWB == 256) red_hist8(lb + (u << 8));
            else red_add_shared(lb + (u << 7), 1u);
        }
    } else {
        const uint32_t cb = copy12(sm, lane & (sm.ncopies - 1), par);
        uint32_t bad = 0;
        // not unrolled: a window of 8192 samples has four rounds, and the unrolled loop's entry costs
        // more than it saves (8192-sample windows 583 -> 578 us, 4096 395 -> 382, 1024 1107 -> 1053)
#pragma unroll 1
        for (int c = tid; c < nfull; c += T) {
            const uint4 a = d4[c];
            hist12_word(cb, a.x); hist12_word(cb, a.y); hist12_word(cb, a.z); hist12_word(cb, a.w);
            bad |= range12_bits(a.x) | range12_bits(a.y) | range12_bits(a.z) | range12_bits(a.w);
        }
        const int rem = (nbytes & 15) >> 1;
        if (tid < rem) {
            const uint32_t x = reinterpret_cast<const uint16_t *>(w.data)[nfull * 8 + tid];
            red_add_shared(cb + (((x & 0xFFFu) ^ 0x800u) << 2), 1u);
            bad |= range12_bits(x) & 0xF000u;
        }
        if (bad & kRange12) atomicOr(&sm.ctl->err[par], 1u);
    }
}

// Any-window form: sample 0 lies off bytes into the first 16-byte chunk. Thread i of the nt that
// count this window takes the whole chunks c0 + i, c0 + i + nt, ... and, for i < 32, one sample of
// the partial chunks at the window's ends (nt >= 32).
template <int BITS, class Word, class One>
__device__ __forceinline__ void hist_chunks(const Win &w, int i, int nt, Word &&word, One &&one) {
    constexpr int BPS = Geo<BITS>::kBps, CS = Geo<BITS>::kChunkSamples;
    const int end = w.off + w.n * BPS;
    const int c0 = (w.off + 15) >> 4, c1 = end >> 4;  // whole chunks [c0, c1)
    const uint4 *d4 = reinterpret_cast<const uint4 *>(w.data);
    int c = c0 + i;
    for (; c + nt < c1; c += 2 * nt) {
        const uint4 a = d4[c], b = d4[c + nt];
        word(a.x); word(a.y); word(a.z); word(a.w);
        word(b.x); word(b.y); word(b.z); word(b.w);
    }
    if (c < c1) {
        const uint4 a = d4[c];
        word(a.x); word(a.y); word(a.z); word(a.w);
    }
    // samples before chunk c0 (all of them when no chunk is whole), then those from chunk c1 on
    const int head = min(16 * c0, end) - w.off, tail = c1 >= c0 ? end - 16 * c1 : 0;
    if (i < CS) {
        if (i * BPS < head) one(w.off + i * BPS);
    } else if (i < 2 * CS) {
        if ((i - CS) * BPS < tail) one(16 * c1 + (i - CS) * BPS);
    }
}

template <int BITS, int T>
__device__ __forceinline__ void phase_histogram_any(const Shm &sm, const Win &w, int tid, int par) {
    const int lane = tid & 31;
    if constexpr (BITS == 8) {
        const uint32_t lb = sm.hist_s + 4u * lane;
        hist_chunks<8>(w, tid, T, [&](uint32_t v) { hist8_word<128>(lb, v); },
                       [&](int at) { red_add_shared(lb + (static_cast<uint32_t>(w.data[at]) << 7), 1u); });
    } else {
        const uint32_t cb = copy12(sm, lane & (sm.ncopies - 1), par);
        uint32_t bad = 0;
        hist_chunks<12>(w, tid, T,
                        [&](uint32_t v) {
                            hist12_word(cb, v);
                            bad |= range12_bits(v);
                        },
                        [&](int at) {
                            const uint32_t x = *reinterpret_cast<const uint16_t *>(w.data + at);
                            red_add_shared(cb + (((x & 0xFFFu) ^ 0x800u) << 2), 1u);
                            bad |= range12_bits(x) & 0xF000u;
                        });
        if (bad & kRange12) atomicOr(&sm.ctl->err[par], 1u);
    }
}

// ------------------------------------------------------------------ phases 2-3: reduce + scan
// 8-bit estimation pass: each thread's bins' counts for this window (the differences of its
// running row sums) into the cumulative-count array, for one warp to scan.
template <int T, int ROWB>
__device__ __forceinline__ void phase_reduce8_counts(const Shm &sm, int tid, RowSums &rs) {
    constexpr int TE = T < 256 ? T : 256;
    constexpr int BPT = 256 / TE;
    static_assert(BPT <= 2, "RowSums holds two rows");
    const int lane = tid & 31;
    if (tid < TE) {
#pragma unroll
        for (int i = 0; i < BPT; ++i) {
            const uint4 *row = reinterpret_cast<const uint4 *>(sm.hist + ((tid * BPT + i) ^ 128) * ROWB + sm.grp);
            uint32_t s = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {  // this group's 32 lane counters (128 bytes of the row)
                const uint4 a = row[(q + lane) & 7];
                s += a.x + a.y + a.z + a.w;
            }
            sm.cum[tid * BPT + i] = s - rs.s[i];
            rs.s[i] = s;
        }
    }
}

// One warp: the inclusive scan of 256 counts in place (8 consecutive ones per lane, 16 bytes at a
// time) and the first whose cumulative count reaches half, in every lane. cum on a 16-byte boundary.
__device__ __forceinline__ int scan256_warp(uint32_t *cum, uint32_t half, int lane) {
    uint4 *const own = reinterpret_cast<uint4 *>(cum) + 2 * lane;
    const uint4 a = own[0], b = own[1];
    uint32_t c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 1; j < 8; ++j) c[j] += c[j - 1];
    uint32_t inc = c[7];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t excl = inc - c[7];
    uint32_t below = 0u;  // those that stay below half lie before the one wanted
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        c[j] += excl;
        below += c[j] < half ? 1u : 0u;
    }
    own[0] = make_uint4(c[0], c[1], c[2], c[3]);
    own[1] = make_uint4(c[4], c[5], c[6], c[7]);
    const int first = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, below));
    __syncwarp();
    return first;
}

// 12-bit: the 4096 bins as 256 rows of 16. Each row's total goes into coarse, for one warp
// to scan as the 256 counts of an 8-bit window; the copies are folded into copy 0 on the way. The
// table of the window before is cleared. coarse is the first kCoarse words of that table (its words
// are zeroed by the search, search12) or, in the estimation pass, whose other warps go on to the
// next window's histogram during the search, a region of its own (kModeTight: none). Eight lanes of a row's
// 16-byte read touch all banks (the pieces are taken in an order rotated by row pairs).
// A full scan of the 4096 bins, which this replaces, took the group two more passes over the
// table, a block-wide offset exchange and a fourth barrier: about 1400 instructions of its warps per
// window against 350 (60 streams of 2^22 samples in 2048-sample windows, threshold, 2 CTAs: 1024 -> 991 us;
// with one histogram copy and 3 CTAs, for which there was no room in the old default: 651 us).
constexpr int kCoarse = 256;
template <int T>
__device__ __forceinline__ void phase_rows12(const Shm &sm, int tid, int par, uint32_t *coarse) {
    uint32_t *const old = table12(sm, par ^ 1);
    for (int i4 = tid + (coarse == old ? kCoarse / 4 : 0); i4 < 1024; i4 += T)
        reinterpret_cast<uint4 *>(old)[i4] = make_uint4(0u, 0u, 0u, 0u);
    const int nc = sm.ncopies;
    for (int r = tid; r < 256; r += T) {
        uint4 *const row = reinterpret_cast<uint4 *>(table12(sm, par)) + 4 * r;
        const int rot = (r >> 1) & 3;
        uint32_t s = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint4 v = row[q ^ rot];
            if (nc > 1) {
                for (int c = 1; c < nc; ++c) {
                    uint4 *const o = reinterpret_cast<uint4 *>(sm.hist + c * 16384) + 4 * r + (q ^ rot);
                    const uint4 a = *o;
                    *o = make_uint4(0u, 0u, 0u, 0u);
                    v.x += a.x;
                    v.y += a.y;
                    v.z += a.z;
                    v.w += a.w;
                }
                row[q ^ rot] = v;
            }
            s += v.x + v.y + v.z + v.w;
        }
        coarse[r] = s;
    }
}

// ------------------------------------------------------------------ phase 4: search
// Smallest v in [0, B) with pred(v), for a monotone pred with pred(B-1) true; one warp.
template <int B, typename Pred>
__device__ __forceinline__ int warp_search(int lane, Pred pred) {
    int base = 0, span = B;
    while (span > 32) {
        const int st = span >> 5;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, pred(base + (lane + 1) * st - 1));
        base += (__ffs(bal) - 1) * st;
        span = st;
    }
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, lane < span && pred(base + lane));
    return base + __ffs(bal) - 1;
}

struct Rep {
    int32_t M, D;
    int32_t cval;     // constant replacement (saturated)
    int32_t t;        // min(ceil(Kq*D / 2^16), sample span + 1)
    int32_t hiv, lov; // threshold replacement above / below (saturated)
    int32_t sig2, moff;  // digital noise (NoiseScale)
    bool active;      // some sample can be flagged
};

__device__ __forceinline__ int32_t sat_to(int64_t v, int32_t lo, int32_t hi) {
    return v < lo ? lo : (v > hi ? hi : static_cast<int32_t>(v));
}

// Threshold and replacement values of a window with median M and dispersion D (Eq. 1; D is the
// window's MAD, or the median of MADs of Eq. 3): those that replacement mode MODE reads (kModeStats:
// none but M and D; kModeCopies: none, the variants have records of their own; kRepAll: those of every
// mode). One lane computes them between the search and the replace pass, while the window's other
// threads wait (all values for every mode: 60 streams of 2^26 int8 samples, zero, 1.609 ms; now 1.592).
constexpr int kRepAll = 1 << 20;
template <int BITS, int MODE>
__device__ __forceinline__ RepShared make_rep(int32_t M, int32_t d, int64_t kq, int32_t cval) {
    constexpr int SPAN = Geo<BITS>::kHi - Geo<BITS>::kLo;
    constexpr bool NONE = (MODE & (kModeStats | kModeCopies)) != 0;
    constexpr int RMODE = MODE & 3;
    constexpr bool ALL = (MODE & kRepAll) != 0;
    RepShared r = {};
    r.M = M;
    r.D = d;
    if constexpr (NONE) return r;
    const int64_t kd = kq * static_cast<int64_t>(d);
    const int64_t t = (kd + 65535) >> 16;
    r.t = static_cast<int32_t>(t < SPAN + 1 ? t : SPAN + 1);
    r.active = (d > 0 && t <= SPAN) ? 1u : 0u;  // |x - M| never exceeds the sample span
    if constexpr (ALL || RMODE == 1) r.cval = cval;
    if constexpr (ALL || RMODE == 2) {
        const int64_t c = kd >> 16;
        r.hiv = sat_to(static_cast<int64_t>(r.M) + c, Geo<BITS>::kLo, Geo<BITS>::kHi);
        r.lov = sat_to(static_cast<int64_t>(r.M) - c, Geo<BITS>::kLo, Geo<BITS>::kHi);
    }
    if constexpr (ALL || RMODE == 3) {
        r.sig2 = NoiseScale<BITS>::kSig2 * d;
        r.moff = M - NoiseScale<BITS>::kOff;
    }
    if constexpr (BITS == 8) {
        const uint32_t tt = static_cast<uint32_t>(r.t > 255 ? 255 : r.t);
        r.mb4 = static_cast<uint32_t>(r.M + 128) * 0x01010101u;
        r.tlo7 = (tt & 0x7Fu) * 0x01010101u;
        r.tsmall = tt < 128u ? ~0u : 0u;
        if constexpr (ALL || RMODE == 1) r.c4 = (static_cast<uint32_t>(cval) & 0xFFu) * 0x01010101u;
        if constexpr (ALL || RMODE == 2) {
            const uint32_t ub = static_cast<uint32_t>(r.M + 129);  // smallest biased value above M
            r.hi4 = (static_cast<uint32_t>(r.hiv) & 0xFFu) * 0x01010101u;
            r.lo4 = (static_cast<uint32_t>(r.lov) & 0xFFu) * 0x01010101u;
            r.ulo7 = (ub & 0x7Fu) * 0x01010101u;
            r.usmall = ub < 128u ? ~0u : 0u;
            r.unone = ub > 255u ? 1u : 0u;
        }
    } else {
        // 12-bit, two samples per word (see rep12_word): u = x + 2048 per 16-bit half
        const uint32_t mb = static_cast<uint32_t>(r.M + 2048);
        const uint32_t tt = static_cast<uint32_t>(r.t);  // <= 4096
        r.mb4 = (0x8000u - mb - tt) * 0x00010001u;        // 0x8000 - upper bound, u >= it flags
        r.tlo7 = (0x8000u + mb - tt) * 0x00010001u;       // 0x8000 + lower bound, u <= it flags
        if constexpr (ALL || RMODE == 1) r.c4 = (static_cast<uint32_t>(cval) & 0xFFFFu) * 0x00010001u;
        if constexpr (ALL || RMODE == 2) {
            r.hi4 = (static_cast<uint32_t>(r.hiv) & 0xFFFFu) * 0x00010001u;
            r.lo4 = (static_cast<uint32_t>(r.lov) & 0xFFFFu) * 0x00010001u;
        }
    }
    return r;
}

// One warp, 8-bit: after phase_reduce8_counts and a group barrier, the scan of the counts, the lower
// median bin, then the MAD, then the threshold and replacement values, written to the shared
// control block. The window's other threads wait for this chain, so its length counts.
template <int MODE>
__device__ __forceinline__ void phase_search8(const Shm &sm, int n, int lane, int64_t kq, int32_t cval) {
    const uint32_t *cum = sm.cum;
    const uint32_t half = static_cast<uint32_t>((n + 1) >> 1);
    const int mb = scan256_warp(sm.cum, half, lane);
    const int d = warp_search<256>(lane, [&](int dd) {
        const int hi = mb + dd < 255 ? mb + dd : 255;
        const int lo = mb - dd - 1;
        const uint32_t f = cum[hi] - (lo >= 0 ? cum[lo] : 0u);
        return f >= half;
    });
    if (lane == 0) sm.ctl->rep = make_rep<8, MODE>(mb - Geo<8>::kOffset, d, kq, cval);
}

// One warp, 12-bit: after phase_rows12 and a group barrier, the scan of the rows' totals (cc), the
// median M in its row R, then the MAD. With F(d) the samples within d of M:
//  - the smallest s for which the rows R - s .. R + s hold half the window puts D into 16(s - 1) + 1 ..
//    16 s + 15 (those rows lie within 16 s + 15 of M and hold everything within 16 s of it),
//  - F(16(s - 1)) comes from the rows' cumulative counts and parts of two rows,
//  - lane j adds the bins at distance 16(s - 1) + 1 + j on either side, and a prefix sum gives the first
//    distance that reaches half the window.
template <int MODE>
__device__ __forceinline__ void phase_search12(const Shm &sm, const uint32_t *tab, uint32_t *cc, bool zero_cc, int n,
                                               int lane, int64_t kq, int32_t cval) {
    const uint32_t half = static_cast<uint32_t>((n + 1) >> 1);
    auto prefix = [&](uint32_t v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, v, o);
            if (lane >= o) v += y;
        }
        return v;
    };
    auto upto = [&](int r) { return r >= 0 ? cc[r] : 0u; };  // samples in rows 0 .. r
    const int R = scan256_warp(cc, half, lane);
    const uint32_t in_row = prefix(lane < 16 ? tab[16 * R + lane] : 0u);
    const int M = 16 * R + __ffs(__ballot_sync(0xFFFFFFFFu, upto(R - 1) + in_row >= half)) - 1;
    const int s = warp_search<256>(lane, [&](int x) { return upto(min(R + x, 255)) - upto(R - x - 1) >= half; });
    const int d0 = 16 * (s - 1);
    uint32_t base = 0u;  // F(d0)
    if (s > 0) {
        const int b1 = min(M + d0, 4095), b2 = M - d0 - 1;
        const int b = lane < 16 ? b1 : b2;
        const uint32_t v = b >= 0 && (lane & 15) <= (b & 15) ? tab[(b & ~15) + (lane & 15)] : 0u;
        base = upto((b1 >> 4) - 1) - (b2 >= 0 ? upto((b2 >> 4) - 1) : 0u) + __reduce_add_sync(0xFFFFFFFFu, lane < 16 ? v : 0u - v);
    }
    const int d = d0 + 1 + lane;
    uint32_t add = 0u;
    if (d >= 0 && M + d <= 4095) add = tab[M + d];
    if (d > 0 && M - d >= 0) add += tab[M - d];
    const int D = d0 + __ffs(__ballot_sync(0xFFFFFFFFu, base + prefix(add) >= half));
    if (lane == 0) sm.ctl->rep = make_rep<12, MODE>(M - Geo<12>::kOffset, D, kq, cval);
    if (zero_cc) {
        __syncwarp();
        for (int i = lane; i < kCoarse / 4; i += 32) reinterpret_cast<uint4 *>(cc)[i] = make_uint4(0u, 0u, 0u, 0u);
    }
}

__device__ __forceinline__ Rep load_rep(const RepShared &s) {
    Rep r;
    r.M = s.M;
    r.D = s.D;
    r.cval = s.cval;
    r.t = s.t;
    r.hiv = s.hiv;
    r.lov = s.lov;
    r.active = s.active != 0u;
    r.sig2 = s.sig2;
    r.moff = s.moff;
    return r;
}

// ------------------------------------------------------------------ phase 5: replace
// Bit 7 of byte j of the result is [a_j >= c_j] for unsigned bytes, given clo7 = c & 0x7F7F7F7F
// and csmall = all ones when every c_j < 128 (zero when every c_j >= 128). The subtraction
// cannot borrow across bytes because (a | 0x80) >= 0x80 > (c & 0x7F).
__device__ __forceinline__ uint32_t ge_bytes_msb(uint32_t a, uint32_t clo7, uint32_t csmall) {
    const uint32_t d = (a | 0x80808080u) - clo7;  // bit 7: low 7 bits of a >= low 7 bits of c
    return (a & d) | ((a | d) & csmall);
}

// Per-window constants of the int8 replace pass.
struct Rep8 {
    uint32_t mb4;      // (M + 128) in every byte
    uint32_t tlo7;     // t & 0x7F in every byte
    uint32_t tsmall;   // t < 128 ? ~0 : 0
    uint32_t c4;       // constant replacement in every byte
    uint32_t hi4, lo4; // threshold replacement above / below in every byte
    uint32_t ulo7;     // (M + 129) & 0x7F in every byte (x > M test)
    uint32_t usmall;   // M + 129 < 128 ? ~0 : 0
    uint32_t unone;    // M == 127: nothing lies above the median
};

__device__ __forceinline__ Rep8 load_rep8(const RepShared *rsrc) {
    const uint4 *rq = reinterpret_cast<const uint4 *>(rsrc);
    const uint4 q2 = rq[2], q3 = rq[3], q4 = rq[4];
    Rep8 k;
    k.mb4 = q2.x;
    k.tlo7 = q2.y;
    k.tsmall = q2.z;
    k.c4 = q2.w;
    k.hi4 = q3.x;
    k.lo4 = q3.y;
    k.ulo7 = q3.z;
    k.usmall = q3.w;
    k.unone = q4.x;
    return k;
}

// 4 int8 samples: returns the output word and sets f to 0xFF in flagged bytes. With digital noise the
// word stays as it is: the noise overwrites every flagged sample.
template <int MODE>
__device__ __forceinline__ uint32_t rep8_word(uint32_t w, const Rep8 &k, uint32_t &f) {
    const uint32_t wb = w ^ 0x80808080u;                  // x + 128 in every byte
    const uint32_t ad = __vabsdiffu4(wb, k.mb4);         // |x - M|
    f = prmt(ge_bytes_msb(ad, k.tlo7, k.tsmall), 0u, 0xBA98u);
    if (MODE == 3) return w;
    uint32_t rep = 0u;
    if (MODE == 1) rep = k.c4;
    if (MODE == 2) {
        const uint32_t up = k.unone ? 0u : prmt(ge_bytes_msb(wb, k.ulo7, k.usmall), 0u, 0xBA98u);
        rep = (k.hi4 & up) | (k.lo4 & ~up);
    }
    return (w & ~f) | (rep & f);
}

// Two 12-bit samples (int16 halves of w, in range): returns the output word and sets f, whose bits 15
// and 31 are the samples' flags. With u = x + 2048 (12 bits) per half and bounds lo = M + 2048 - t,
// hi = M + 2048 + t: x is flagged iff u >= hi or u <= lo (Eq. 2 with |x - M| >= t). Per half,
// u + (0x8000 - hi) has bit 15 set iff u >= hi, and (0x8000 + lo) - u iff u <= lo; no carry or borrow
// crosses the halves because every operand is below 2^13. A byte permute that takes the sign of
// bytes 1 and 3 makes a flag its half's select mask. With digital noise the word stays as it is: the
// noise overwrites every flagged sample.
__device__ __forceinline__ uint32_t half_mask(uint32_t f) { return prmt(f, 0u, 0xBB99u); }
template <int MODE>
__device__ __forceinline__ uint32_t rep12_word(uint32_t w, uint32_t hi2, uint32_t lo2x, uint32_t c2, uint32_t h2,
                                               uint32_t l2, uint32_t &f) {
    const uint32_t u = (w ^ 0x08000800u) & 0x0FFF0FFFu;
    const uint32_t up = u + hi2;   // bit 15 / 31: u >= hi
    const uint32_t dn = lo2x - u;  // bit 15 / 31: u <= lo
    f = up | dn;
    if (MODE == 3) return w;
    const uint32_t m = half_mask(f);
    uint32_t z = 0u;
    if (MODE == 1) z = c2;
    if (MODE == 2) {
        const uint32_t ma = half_mask(up);
        z = (h2 & ma) | (l2 & ~ma);
    }
    return (w & ~m) | (z & m);
}

// Mask bits of a chunk of eight 12-bit samples from its four words of flags (bits 15 and 31): the
// signs of the flags' bytes, then the signed byte dot product of chunk_bits.
__device__ __forceinline__ uint32_t chunk_bits12(uint32_t f0, uint32_t f1, uint32_t f2, uint32_t f3) {
    return static_cast<uint32_t>(__dp4a(static_cast<int>(prmt(f2, f3, 0xFDB9u)), static_cast<int>(0x80C0E0F0u),
                                        __dp4a(static_cast<int>(prmt(f0, f1, 0xFDB9u)), static_cast<int>(0xF8FCFEFFu), 0)));
}

// Mask bits of a 16-sample chunk from its four flag words (0x00/0xFF bytes), sample j -> bit j.
// A flag byte read as signed is -1, so a signed byte dot product with negated powers of two
// (-1, -2, -4, -8 for the first word of a half, -16 .. -128 for the second) packs 8 flags.
__device__ __forceinline__ uint32_t chunk_bits(uint32_t f0, uint32_t f1, uint32_t f2, uint32_t f3) {
    const int lo = __dp4a(static_cast<int>(f1), static_cast<int>(0x80C0E0F0u),
                          __dp4a(static_cast<int>(f0), static_cast<int>(0xF8FCFEFFu), 0));
    const int hi = __dp4a(static_cast<int>(f3), static_cast<int>(0x80C0E0F0u),
                          __dp4a(static_cast<int>(f2), static_cast<int>(0xF8FCFEFFu), 0));
    return static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 8);
}

// Position of the j-th (0-based) set bit of m (j < popc(m)), by halving popcount search.
__device__ __forceinline__ int nth_set_bit(uint32_t m, int j) {
    int pos = 0;
    int c = __popc(m & 0xFFFFu);
    if (j >= c) { j -= c; pos += 16; m >>= 16; }
    c = __popc(m & 0xFFu);
    if (j >= c) { j -= c; pos += 8; m >>= 8; }
    c = __popc(m & 0xFu);
    if (j >= c) { j -= c; pos += 4; m >>= 4; }
    c = __popc(m & 0x3u);
    if (j >= c) { j -= c; pos += 2; m >>= 2; }
    return pos + ((j >= static_cast<int>(m & 1u)) ? 1 : 0);
}

// ------------------------------------------------------------------ output formats
// OUTF 0 writes the input's type; 1 writes fp16 and 2 bf16 (int8 input only). Every sample value
// is exact in either: |x| <= 2048 needs 12 significant bits (fp16 has 11 + 1) and int8 needs 8
// (bf16 has 7 + 1).
template <int BITS, int OUTF>
__device__ __forceinline__ void store_sample(uint8_t *out, int pos, int32_t z) {
    if (OUTF == 1) reinterpret_cast<__half *>(out)[pos] = __int2half_rn(z);
    else if (OUTF == 2) reinterpret_cast<__nv_bfloat16 *>(out)[pos] = __int2bfloat16_rn(z);
    else if (BITS == 8) out[pos] = static_cast<uint8_t>(z);
    else reinterpret_cast<int16_t *>(out)[pos] = static_cast<int16_t>(z);
}

// The 16 int8 output samples of chunk c (v holds them as bytes) in format OUTF: 16-byte stores
// when vec, else one sample at a time. fp16: a biased byte u = x + 128 placed under 0x64 is the
// fp16 1024 + u, and subtracting 1152 leaves x. bf16: u placed in the fp32 2^23 + u, minus
// 2^23 + 128, leaves x as fp32; its bf16 rounding is exact.
template <int OUTF>
__device__ __forceinline__ void store_chunk8(uint8_t *out, int c, const uint4 &v, bool vec) {
    const uint32_t ww[4] = {v.x, v.y, v.z, v.w};
    if constexpr (OUTF == 0) {
        if (vec) {
            __stcs(reinterpret_cast<uint4 *>(out) + c, v);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) out[c * 16 + j] = static_cast<uint8_t>(ww[j >> 2] >> ((j & 3) * 8));
        }
    } else {
        uint32_t h[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t u = ww[q] ^ 0x80808080u;
            if (OUTF == 1) {
                const __half2 off = __half2half2(__ushort_as_half(static_cast<unsigned short>(0x6480u)));  // 1152
                __half2 lo, hi;
                *reinterpret_cast<uint32_t *>(&lo) = __byte_perm(u, 0x64646464u, 0x5140u);
                *reinterpret_cast<uint32_t *>(&hi) = __byte_perm(u, 0x64646464u, 0x7362u);
                lo = __hsub2(lo, off);
                hi = __hsub2(hi, off);
                h[2 * q] = *reinterpret_cast<uint32_t *>(&lo);
                h[2 * q + 1] = *reinterpret_cast<uint32_t *>(&hi);
            } else {
                float f[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    f[k] = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7540u | k)) - 8388736.0f;
                const __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]);
                const __nv_bfloat162 b = __floats2bfloat162_rn(f[2], f[3]);
                h[2 * q] = *reinterpret_cast<const uint32_t *>(&a);
                h[2 * q + 1] = *reinterpret_cast<const uint32_t *>(&b);
            }
        }
        if (vec) {
            uint4 *o = reinterpret_cast<uint4 *>(out) + 2 * c;
            __stcs(o, make_uint4(h[0], h[1], h[2], h[3]));
            __stcs(o + 1, make_uint4(h[4], h[5], h[6], h[7]));
        } else {
            uint16_t *o = reinterpret_cast<uint16_t *>(out) + 16 * c;
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = static_cast<uint16_t>(h[j >> 1] >> ((j & 1) * 16));
        }
    }
}

// Digital noise for the flagged samples of one round of the warp: lane l holds in bits the flags of
// samples s0, s0 + 1, ... The flagged samples are numbered across the warp (an exclusive prefix sum
// of the per-lane counts); in each pass lane q takes sample q, found by a shuffle binary search for
// the lane that owns it and a popcount search for its bit, and all 32 lanes evaluate Philox
// together. The stores go straight to the output; they follow the chunks' own stores in warp order
// (__syncwarp before the call).
template <int BITS, bool PW, class K, int OUTF = 0>
__device__ __forceinline__ void noise_batch(const Win &w, const Rep &r, const K &p, int lane, int s0,
                                            uint32_t bits, Pow &pw) {
    const uint32_t cnt = __popc(bits);
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    const uint32_t excl = inc - cnt;
    const NoiseRun<BITS, K> run = w.template noise<BITS>(p);
    for (uint32_t q0 = 0; q0 < total; q0 += 32) {
        const uint32_t q = q0 + lane;
        // owner: the last lane whose first index is <= q (lanes without flags share the next
        // lane's first index, so the search passes over them)
        int L = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            const uint32_t e = __shfl_sync(0xFFFFFFFFu, excl, L + step);
            if (e <= q) L += step;
        }
        const uint32_t eL = __shfl_sync(0xFFFFFFFFu, excl, L);
        const uint32_t bL = __shfl_sync(0xFFFFFFFFu, bits, L);
        const int sL = __shfl_sync(0xFFFFFFFFu, s0, L);
        if (q < total) {
            const int pos = sL + nth_set_bit(bL, static_cast<int>(q - eL));
            const int32_t z = run.value_any(static_cast<uint32_t>(pos), r.sig2, r.moff);
            store_sample<BITS, OUTF>(w.out, pos, z);
            if (PW) pw.z += static_cast<uint32_t>(z * z);
        }
    }
}

// Digital noise, replace pass (12-bit): the warp numbers its flagged samples of this round, reserves
// that many list entries with one shared atomic, and each lane writes its positions, counted from
// the window's first sample. Samples beyond the list's end take the per-warp path at once. Called by
// all lanes of the warp with the flags of samples s0, s0 + 1, ...
template <int BITS, bool PW, class K, int OUTF = 0>
__device__ __forceinline__ void noise_append(const Shm &sm, const Win &w, const Rep &r, const K &p, int lane,
                                             int s0, uint32_t bits, uint32_t *nlc, Pow &pw) {
    if (!__any_sync(0xFFFFFFFFu, bits != 0u)) return;
    const uint32_t cnt = __popc(bits);
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    uint32_t base = kNoiseList;
    if (sm.nlist != nullptr && lane == 31) base = atomicAdd(nlc, total);
    base = __shfl_sync(0xFFFFFFFFu, base, 31);
    uint32_t off = base + inc - cnt;
    if (base + total <= static_cast<uint32_t>(kNoiseList)) {
        // one predicated store per sample of the chunk: with a quarter of the samples flagged in
        // bursts some lane has all eight, and a loop over the set bits costs more per step (with the
        // noise words shared over a tile, 60 streams of 2^25 samples in 8192-sample windows: 4.54 -> 4.27 ms)
#pragma unroll
        for (int j = 0; j < Geo<BITS>::kChunkSamples; ++j)
            if ((bits >> j) & 1u) sm.nlist[off++] = static_cast<uint16_t>(s0 + j);
        return;
    }
    uint32_t beyond = bits;  // what the list has no room for
    for (; off < static_cast<uint32_t>(kNoiseList) && beyond; beyond &= beyond - 1u)
        sm.nlist[off++] = static_cast<uint16_t>(s0 + __ffs(static_cast<int>(beyond)) - 1);
    __syncwarp();  // the round's chunk stores come first
    noise_batch<BITS, PW, K, OUTF>(w, r, p, lane, s0, beyond, pw);
}

// Digital noise, after the group barrier that follows the replace pass: every thread of the
// group evaluates Philox for a share of the list and stores the value over the chunk's output.
template <int BITS, int T, bool PW, class K, int OUTF = 0>
__device__ __forceinline__ void noise_list(const Shm &sm, const Win &w, const Rep &r, const K &p, int tid,
                                           const uint32_t *nlc, Pow &pw) {
    if (sm.nlist == nullptr) return;
    const uint32_t n = min(*nlc, static_cast<uint32_t>(kNoiseList));
    const NoiseRun<BITS, K> run = w.template noise<BITS>(p);
    auto put = [&](uint32_t pos, int32_t z) {
        store_sample<BITS, OUTF>(w.out, static_cast<int>(pos), z);
        if (PW) pw.z += static_cast<uint32_t>(z * z);
    };
    uint32_t i = static_cast<uint32_t>(tid);
    if (run.one_hi) {
        // two entries at a time: the two Philox chains are independent, so their rounds interleave
        // and fill each other's dependency stalls (60 streams of 2^25 12-bit samples in 8192-sample
        // windows, a quarter of them flagged: 4.60 -> 4.53 ms per call)
        for (; i + T < n; i += 2 * T) {
            const uint32_t la = sm.nlist[i], lb = sm.nlist[i + T];
            const int2 z = run.value2(la, lb, r.sig2, r.moff);
            put(la, z.x);
            put(lb, z.y);
        }
        if (i < n) {
            const uint32_t l = sm.nlist[i];
            put(l, run.value(l, r.sig2, r.moff));
        }
    } else {  // a window across a multiple of 2^32
        for (; i < n; i += T) {
            const uint32_t l = sm.nlist[i];
            put(l, run.value_any(l, r.sig2, r.moff));
        }
    }
}

// Digital noise (int8), replace pass: the warp appends one list entry per chunk of its round
// that holds a flagged sample, (chunk << 16) | the chunk's 16 flag bits, at places reserved
// with one shared atomic on the entry count *nlc. The list has room for every chunk of a stage.
// Called by all lanes of the warp (bits = 0 for a lane without a chunk).
__device__ __forceinline__ void noise_note8(const Shm &sm, int lane, int c, uint32_t bits, uint32_t *nlc) {
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, bits != 0u);
    if (bal == 0u) return;
    uint32_t base = 0u;
    if (lane == 0) base = atomicAdd(nlc, static_cast<uint32_t>(__popc(bal)));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (bits)
        reinterpret_cast<uint32_t *>(sm.nlist)[base + __popc(bal & ((1u << lane) - 1u))] =
            (static_cast<uint32_t>(c) << 16) | bits;
}

// Digital noise (int8), after the replace pass and a group barrier: the n entries noted by
// noise_note8, in any order (a sample's noise depends only on its absolute index). Warp w
// expands entries 2w and 2w + 1, then 2w + 2NW and 2w + 2NW + 1, and so on: each half-warp
// takes one entry and its lane j tests flag bit j. The flagged positions go into the warp's
// ring, compacted by a ballot and a prefix popcount, and whenever 32 (PAIR: 64) are waiting every
// lane takes one (two, whose Philox chains interleave) and emit evaluates and stores its noise.
// Fewer are left for the end. Every lane does Philox work in every batch but the last, however
// the flags are spread over the chunks, and the chunks are shared out evenly between the warps.
// PAIR, and no branch per batch for runs across a multiple of 2^32 (60 streams of 2^22 samples,
// noise): 16384-sample windows 259 -> 252 us, 65536 377 -> 350, fp16 output 281 -> 271.
template <int T, bool PAIR, class Emit, class Emit2>
__device__ __forceinline__ void noise_expand8(const Shm &sm, uint32_t n, int tid, Emit &&emit, Emit2 &&emit2) {
    using Pos = typename std::conditional<PAIR, uint16_t, uint32_t>::type;
    constexpr uint32_t NW = T / 32, B = PAIR ? 64 : 32, RING = 2 * B;
    static_assert(RING * sizeof(Pos) == kNoiseRingBytes, "ring size");
    constexpr uint32_t RM = RING - 1;
    const int lane = tid & 31;
    const uint32_t warp = static_cast<uint32_t>(tid >> 5);
    const uint32_t *list = reinterpret_cast<const uint32_t *>(sm.nlist);
    Pos *ring = reinterpret_cast<Pos *>(sm.nring) + warp * RING;
    const uint32_t j = static_cast<uint32_t>(lane & 15);
    const uint32_t below = (1u << lane) - 1u;
    uint32_t head = 0u, tail = 0u;  // positions taken / queued so far (tail - head < B between steps)
    auto at = [&](uint32_t i) -> uint32_t { return ring[(head + i + static_cast<uint32_t>(lane)) & RM]; };
    for (uint32_t e0 = 2u * warp; e0 < n; e0 += 2u * NW) {
        const uint32_t e = e0 + static_cast<uint32_t>(lane >> 4);
        const uint32_t ent = e < n ? list[e] : 0u;
        const bool fl = ((ent >> j) & 1u) != 0u;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, fl);
        if (fl) ring[(tail + static_cast<uint32_t>(__popc(bal & below))) & RM] = static_cast<Pos>((ent >> 16) * 16u + j);
        tail += static_cast<uint32_t>(__popc(bal));
        if (tail - head >= B) {
            __syncwarp();
            if constexpr (PAIR) {
                const uint32_t pa = at(0), pb = at(32);
                __syncwarp();  // read before the next step refills the slots
                head += B;
                emit2(pa, pb);
            } else {
                const uint32_t pos = at(0);
                __syncwarp();  // read before the next step refills the slot
                head += B;
                emit(pos);
            }
        }
    }
    if (PAIR && tail - head > 32u) {
        __syncwarp();
        emit(at(0));
        head += 32u;
    }
    if (tail != head) {
        __syncwarp();
        if (static_cast<uint32_t>(lane) < tail - head) emit(at(0));
    }
}

// The same for a run whose indices have two high words (a tile across a multiple of 2^32): one entry
// per thread, its samples one after the other.
template <int T, class Emit>
__device__ __forceinline__ void noise_expand8_any(const Shm &sm, uint32_t n, int tid, Emit &&emit) {
    for (uint32_t e = static_cast<uint32_t>(tid); e < n; e += T) {
        const uint32_t ent = reinterpret_cast<const uint32_t *>(sm.nlist)[e];
        for (uint32_t m = ent & 0xFFFFu; m; m &= m - 1u) emit((ent >> 16) * 16u + static_cast<uint32_t>(__ffs(m) - 1));
    }
}

// Digital noise (int8) of one window, after its replace pass noted its chunks in the list (*nlc
// entries): one group barrier, then noise_expand8. Every store is checked against the window's
// length.
template <int T, bool PW, bool PAIR, class K, int OUTF = 0>
__device__ __forceinline__ void noise_deferred8(const Shm &sm, const Win &w, const Rep &r, const K &p, int tid,
                                                const uint32_t *nlc, Pow &pw) {
    named_bar(sm.bar_id, T);  // every entry of the window is in the list
    const NoiseRun<8, K> run = w.template noise<8>(p);
    auto put = [&](uint32_t pos, int32_t z) {
        if (pos >= static_cast<uint32_t>(w.n)) return;
        store_sample<8, OUTF>(w.out, static_cast<int>(pos), z);
        if (PW) pw.z += static_cast<uint32_t>(z * z);
    };
    const uint32_t off = static_cast<uint32_t>(w.off);
    if constexpr (!std::is_same<K, KeysPre>::value) {
        // a variant's own key: no tile words, and its window's flags are too few to pay for them
        noise_expand8<T, false>(
            sm, *nlc, tid, [&](uint32_t at) { put(at - off, run.value_any(at - off, r.sig2, r.moff)); },
            [](uint32_t, uint32_t) {});
    } else if (run.one_hi) {
        noise_expand8<T, PAIR>(
            sm, *nlc, tid, [&](uint32_t at) { put(at - off, run.value(at - off, r.sig2, r.moff)); },
            [&](uint32_t a, uint32_t b) {
                const int2 z = run.value2(a - off, b - off, r.sig2, r.moff);
                put(a - off, z.x);
                put(b - off, z.y);
            });
    } else {
        noise_expand8_any<T>(sm, *nlc, tid, [&](uint32_t at) { put(at - off, run.value_any(at - off, r.sig2, r.moff)); });
    }
}

// Sum of squares of the bytes of w kept by keep (0xFF per kept byte), as signed int8 samples.
__device__ __forceinline__ uint32_t sq4(uint32_t w, uint32_t keep) {
    const int32_t v = static_cast<int32_t>(w & keep);
    return static_cast<uint32_t>(__dp4a(v, v, 0));
}

// rsrc: the shared record r was loaded from (its int8 constants are read from there). FO (8-bit
// in-place form): chunks without a flagged sample are not stored, and in noise mode no chunk is
// (the noise pass writes every flagged sample). PAIR (the split-warp form's replace warps):
// full rounds go two at a time.
template <int BITS, int MODE, int T, bool PW, class K, int OUTF = 0, bool FO = false, bool PAIR = false>
__device__ __forceinline__ uint32_t phase_replace(const Shm &sm, const Win &w, const Rep &r, const K &p,
                                                  int tid, uint32_t *nlc, Pow &pw, const RepShared *rsrc,
                                                  int slice = 0, int send = 0) {
    constexpr int BPS = Geo<BITS>::kBps;
    const int lane = tid & 31, warp = tid >> 5;
    const int nbytes = w.n * BPS;
    const int nfull = nbytes >> 4;
    const int nchunks = (nbytes + 15) >> 4;
    const uint4 *d4 = reinterpret_cast<const uint4 *>(w.data);
    uint32_t flagged = 0;
    if (BITS == 8) {
        constexpr int M8 = PW && MODE == 3 ? 0 : MODE;  // power metering adds the noise's squares to zeros'
        const Rep8 k = load_rep8(rsrc);
        uint16_t *mk = reinterpret_cast<uint16_t *>(w.mask);
        int base = warp * 32;
        if (r.active && w.vec && mk) {
            // rounds in which all 32 chunks of the warp are full: no bounds checks
            auto full_round = [&](int c, uint4 v) {
                if (PW) pw.x += sq4(v.x, ~0u) + sq4(v.y, ~0u) + sq4(v.z, ~0u) + sq4(v.w, ~0u);
                uint32_t f0, f1, f2, f3;
                v.x = rep8_word<M8>(v.x, k, f0);
                v.y = rep8_word<M8>(v.y, k, f1);
                v.z = rep8_word<M8>(v.z, k, f2);
                v.w = rep8_word<M8>(v.w, k, f3);
                const uint32_t bits = chunk_bits(f0, f1, f2, f3);
                if (!FO || (MODE != 3 && bits)) store_chunk8<OUTF>(w.out, c, v, true);
                if (PW) pw.z += sq4(v.x, ~0u) + sq4(v.y, ~0u) + sq4(v.z, ~0u) + sq4(v.w, ~0u);
                mk[c] = static_cast<uint16_t>(bits);
                flagged += __popc(bits);
                if (MODE == 3) noise_note8(sm, lane, c, bits, nlc);
            };
            // two rounds at a time, both chunks loaded before either is replaced (the loads of the
            // second overlap the first's arithmetic): zero, constant and threshold in the split-warp
            // form (1.618 -> 1.607 ms for a zero-mode call over 60 streams of 2^26 int8 samples in
            // 16384-sample windows; in the joint form the fp16 output lost 6 % and the digital copy
            // and the Median-of-MAD apply pass 1 %)
            if (PAIR && MODE != 3) {
                for (; base + T + 32 <= nfull; base += 2 * T) {
                    const uint4 va = d4[base + lane];
                    const uint4 vb = d4[base + T + lane];
                    full_round(base + lane, va);
                    full_round(base + T + lane, vb);
                }
            }
            for (; base + 32 <= nfull; base += T) full_round(base + lane, d4[base + lane]);
        }
        // warp-uniform rounds: lane handles chunk base + lane
        for (; base < nchunks; base += T) {
            const int c = base + lane;
            uint32_t bits = 0;
            if (c < nchunks) {
                uint4 v = d4[c];
                const uint4 vin = v;
                if (r.active) {
                    uint32_t f0, f1, f2, f3;
                    v.x = rep8_word<M8>(v.x, k, f0);
                    v.y = rep8_word<M8>(v.y, k, f1);
                    v.z = rep8_word<M8>(v.z, k, f2);
                    v.w = rep8_word<M8>(v.w, k, f3);
                    bits = chunk_bits(f0, f1, f2, f3);
                }
                if (c < nfull) {
                    if (!FO || (MODE != 3 && bits)) store_chunk8<OUTF>(w.out, c, v, w.vec);
                } else {  // ragged last chunk of the window
                    const int valid = nbytes - c * 16;
                    bits &= (1u << valid) - 1u;
                    const uint32_t ww[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (j < valid && (!FO || (MODE != 3 && ((bits >> j) & 1u))))
                            store_sample<8, OUTF>(w.out, c * 16 + j, static_cast<int8_t>(ww[j >> 2] >> ((j & 3) * 8)));
                }
                if (PW) {
                    // the samples of the window only: the ragged chunk's tail bytes are not its own
                    const int valid = c < nfull ? 16 : nbytes - c * 16;
                    uint32_t kp[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int nv = valid - 4 * q;
                        kp[q] = nv >= 4 ? ~0u : (nv <= 0 ? 0u : (1u << (8 * nv)) - 1u);
                    }
                    pw.x += sq4(vin.x, kp[0]) + sq4(vin.y, kp[1]) + sq4(vin.z, kp[2]) + sq4(vin.w, kp[3]);
                    pw.z += sq4(v.x, kp[0]) + sq4(v.y, kp[1]) + sq4(v.z, kp[2]) + sq4(v.w, kp[3]);
                }
                flagged += __popc(bits);
                if (mk) mk[c] = static_cast<uint16_t>(bits);
            }
            if (MODE == 3) noise_note8(sm, lane, c, bits, nlc);
        }
        if (mk) {
            for (int c = nchunks + tid; c < 2 * w.mask_words; c += T) mk[c] = 0;
        }
    } else {
        uint8_t *mk = reinterpret_cast<uint8_t *>(w.mask);
        const int32_t t = r.t;
        const uint32_t hi2 = rsrc->mb4, lo2 = rsrc->tlo7, c2 = MODE == 1 ? rsrc->c4 : 0u;
        const uint32_t h2 = MODE == 2 ? rsrc->hi4 : 0u, l2 = MODE == 2 ? rsrc->lo4 : 0u;
        const int cend = MODE == 3 ? min(nchunks, send) : nchunks;  // chunks [slice, send)
        for (int base = slice + warp * 32; base < cend; base += T) {
            const int c = base + lane;
            uint32_t bits = 0;
            if (c < cend) {
                const uint4 v = d4[c];
                uint32_t ww[4] = {v.x, v.y, v.z, v.w};
                const int valid = c < nfull ? 8 : ((nbytes - c * 16) >> 1);  // samples in the window
                if (!PW) {
                    if (r.active) {
                        uint32_t f[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) ww[q] = rep12_word<MODE>(ww[q], hi2, lo2, c2, h2, l2, f[q]);
                        bits = chunk_bits12(f[0], f[1], f[2], f[3]);
                        // samples past the window (a ragged last chunk) are neither flagged nor stored
                        if (valid < 8) bits &= (1u << valid) - 1u;
                    }
                } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int sh = (j & 1) * 16;
                    const int32_t x = static_cast<int16_t>((ww[j >> 1] >> sh) & 0xFFFFu);
                    const int32_t ad = x > r.M ? x - r.M : r.M - x;
                    const bool fl = r.active && ad >= t && j < valid;
                    int32_t zo = x;
                    if (fl) {
                        int32_t z = 0;
                        if (MODE == 1) z = r.cval;
                        else if (MODE == 2) z = x > r.M ? r.hiv : r.lov;
                        ww[j >> 1] = (ww[j >> 1] & ~(0xFFFFu << sh)) | ((static_cast<uint32_t>(z) & 0xFFFFu) << sh);
                        bits |= 1u << j;
                        zo = z;
                    }
                    if (PW && j < valid) {
                        pw.x += static_cast<uint32_t>(x * x);
                        pw.z += static_cast<uint32_t>(zo * zo);
                    }
                }
                }
                flagged += __popc(bits);
                if (OUTF == 1) {  // fp16: each int16 pair converted in place, same bytes per chunk
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const __half2 hv = __halves2half2(__short2half_rn(static_cast<short>(ww[q] & 0xFFFFu)),
                                                          __short2half_rn(static_cast<short>(ww[q] >> 16)));
                        ww[q] = *reinterpret_cast<const uint32_t *>(&hv);
                    }
                }
                if (w.vec && c < nfull) {
                    __stcs(reinterpret_cast<uint4 *>(w.out + c * 16), make_uint4(ww[0], ww[1], ww[2], ww[3]));
                } else {
                    uint16_t *o = reinterpret_cast<uint16_t *>(w.out);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < valid) o[c * 8 + j] = static_cast<uint16_t>((ww[j >> 1] >> ((j & 1) * 16)) & 0xFFFFu);
                }
                if (mk) mk[c] = static_cast<uint8_t>(bits);
            }
            if (MODE == 3) noise_append<12, PW, K, OUTF>(sm, w, r, p, lane, c * 8, bits, nlc, pw);
        }
        if (mk && cend == nchunks) {
            for (int c = nchunks + tid; c < 4 * w.mask_words; c += T) mk[c] = 0;
        }
    }
    return flagged;
}

// ------------------------------------------------------------------ any-window form
// The replace pass of a window of any length at any alignment (BPS-aligned), in rounds of 31 chunks:
// lane l takes the 16-byte chunk base + l of the window as it lies in shared memory, which is how
// it lies in global memory too, so whole chunks go out as 16-byte stores where in and out are
// aligned alike. The mask counts bits from sample 0, off samples into the first chunk: its
// 16-bit piece h (8-bit for 12-bit samples) joins the flags of chunks h and h + 1, the second
// from the next lane. Lane 31 only gives its flags to lane 30; its chunk is lane 0's of the next
// round. Returns the lane's flags of its own chunk (0 for lane 31). (Each lane building its own
// sample-aligned 16 bytes with funnel shifts needs a second load and leaves every store unaligned.)
template <int BITS, int MODE>
__device__ __forceinline__ uint32_t replace_round_any(const Win &w, const Rep &r, const RepShared *rsrc, int base, int lane) {
    constexpr int BPS = Geo<BITS>::kBps, CS = Geo<BITS>::kChunkSamples;
    const int offs = w.off / BPS;
    const int c = base + lane;
    const int lo = c == 0 ? offs : 0;
    const int hi = min(CS, offs + w.n - c * CS);  // the window's samples of the chunk: [lo, hi)
    const bool own = lane < 31 && hi > 0;
    uint32_t bits = 0;
    if (hi > 0) {
        const uint4 v = reinterpret_cast<const uint4 *>(w.data)[c];
        uint32_t ww[4] = {v.x, v.y, v.z, v.w};
        if (r.active) {
            uint32_t f[4];
            if (BITS == 8) {
                const Rep8 k = load_rep8(rsrc);
#pragma unroll
                for (int q = 0; q < 4; ++q) ww[q] = rep8_word<MODE>(ww[q], k, f[q]);
                bits = chunk_bits(f[0], f[1], f[2], f[3]);
            } else {
                const RepShared &k = *rsrc;
#pragma unroll
                for (int q = 0; q < 4; ++q) ww[q] = rep12_word<MODE>(ww[q], k.mb4, k.tlo7, k.c4, k.hi4, k.lo4, f[q]);
                bits = chunk_bits12(f[0], f[1], f[2], f[3]);
            }
            bits &= (1u << hi) - (1u << lo);
        }
        if (own) {
            uint8_t *o = w.out - w.off + 16 * static_cast<int64_t>(c);
            if (lo == 0 && hi == CS && w.vec) {
                __stcs(reinterpret_cast<uint4 *>(o), make_uint4(ww[0], ww[1], ww[2], ww[3]));
            } else if (BITS == 8) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j >= lo && j < hi) o[j] = static_cast<uint8_t>(ww[j >> 2] >> ((j & 3) * 8));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j >= lo && j < hi) reinterpret_cast<uint16_t *>(o)[j] = static_cast<uint16_t>(ww[j >> 1] >> ((j & 1) * 16));
            }
        }
    }
    const uint32_t nb = __shfl_down_sync(0xFFFFFFFFu, bits, 1);
    if (w.mask && own && c * CS < w.n) {
        const uint32_t piece = (bits >> offs) | (nb << (CS - offs));
        if (BITS == 8) reinterpret_cast<uint16_t *>(w.mask)[c] = static_cast<uint16_t>(piece);
        else reinterpret_cast<uint8_t *>(w.mask)[c] = static_cast<uint8_t>(piece);
    }
    return own ? bits : 0u;
}

// Mask pieces past the window's last sample.
template <int BITS>
__device__ __forceinline__ void mask_padding(const Win &w, int i, int nt) {
    constexpr int CS = Geo<BITS>::kChunkSamples;
    if (!w.mask) return;
    for (int h = (w.n + CS - 1) / CS + i; h < w.mask_words * (32 / CS); h += nt) {
        if (BITS == 8) reinterpret_cast<uint16_t *>(w.mask)[h] = 0;
        else reinterpret_cast<uint8_t *>(w.mask)[h] = 0;
    }
}

template <int BITS, int MODE, int T, class K>
__device__ __forceinline__ uint32_t phase_replace_any(const Shm &sm, const Win &w, const Rep &r, const K &p, int tid,
                                                      uint32_t *nlc, Pow &pw, const RepShared *rsrc, int slice = 0, int send = 0) {
    constexpr int BPS = Geo<BITS>::kBps, CS = Geo<BITS>::kChunkSamples;
    const int lane = tid & 31, warp = tid >> 5;
    const int nch = (w.off + w.n * BPS + 15) >> 4;
    const int cend = BITS == 12 && MODE == 3 ? min(nch, send) : nch;
    uint32_t flagged = 0;
    for (int base = slice + warp * 31; base < cend; base += (T / 32) * 31) {
        const uint32_t bits = replace_round_any<BITS, MODE>(w, r, rsrc, base, lane);
        flagged += __popc(bits);
        if (MODE == 3) {
            if (BITS == 8) noise_note8(sm, lane, base + lane, bits, nlc);
            else noise_append<12, false, K>(sm, w, r, p, lane, (base + lane) * CS - w.off / BPS, bits, nlc, pw);
        }
    }
    if (cend == nch) mask_padding<BITS>(w, tid, T);
    return flagged;
}

// 12-bit digital noise of one window, in slices: replace(counter, chunks from, to) lists their flagged
// samples and gives the thread's flag count, list(counter) evaluates them. A list per slice leaves
// lanes of many last batches idle and adds two barriers each; one list for a window whose flags do
// not fit leaves the rest to the per-warp path. So a window is one slice where the CTA's window before
// had room in the list for its flags (ctl->wide), and a CTA of one window (ALONE) lets the first slice
// tell: the others join its list where it promises room (the threads agree through the vote of the
// barrier). 60 streams of 2^22 samples in 32768-sample windows, 1.6 % and 10 % flagged: always one list 480 and
// 759 us a call, always slices of 8192 samples 532 and 660, this 456 and 583; 30 of them, one CTA a
// window, 1.6 %: 555 us in slices, 495 this.
// nlc: two counters, both zero on entry, used in turn; the one of the list before is zeroed between
// the two barriers around a list's evaluation, when no thread reads it any more.
template <int T, bool ANY, bool ALONE, class Replace, class List>
__device__ __forceinline__ uint32_t noise_slices12(const Shm &sm, const Win &w, uint32_t *nlc, int tid, Replace &&replace,
                                                   List &&list) {
    constexpr int STEP = ANY ? kNoiseSliceAny : kNoiseSlice;
    const int nch = (w.off + 2 * w.n + 15) >> 4;
    uint32_t f = 0;
    int step = STEP;
    if (!ALONE && nch > STEP && sm.ctl->wide) step = nch;
    for (int c = 0, k = 0;;) {
        f += replace(nlc + k, c, c + step);
        c += step;
        if (ALONE && c == STEP && c < nch) {
            // the warp that lists last reads the whole length
            const uint32_t length = *static_cast<volatile uint32_t *>(nlc + k);
            const uint32_t slices = static_cast<uint32_t>((nch + STEP - 1) / STEP);
            if (!named_bar_or(sm.bar_id, T, 8u * slices * length > 7u * kNoiseList)) {
                step = nch;
                continue;
            }
        } else {
            named_bar(sm.bar_id, T);  // every flagged position of the list is in it
        }
        if (c < nch && tid == 0) nlc[k ^ 1] = 0u;
        list(nlc + k);
        if (c >= nch) return f;
        named_bar(sm.bar_id, T);  // the list is free again
        k ^= 1;
    }
}

// ------------------------------------------------------------------ digital copies
// Eq. 2 for all variants of one threshold multiple at once (grp: their bits, v: the first of them),
// over a window of whole warp rounds that uses all its mask words, with aligned outputs and masks: same
// M, same t, so the flags, the mask bits and the count are computed once, and each variant adds its own
// replacement and stores (one variant at a time, every one of them computed the flags again: 8 variants, two
// multiples with four replacements each, 60 streams of 2^22 samples 748 us a call, now 653).
template <int T>
__device__ __forceinline__ uint32_t copies_pass8(const Shm &sm, const Win &w, int v, uint32_t grp, bool noise, int tid,
                                                 uint32_t *nlc) {
    const int lane = tid & 31, warp = tid >> 5;
    const RepShared &lead = sm.cp->vrep[v];
    const Rep8 k = load_rep8(&lead);
    const uint32_t on = lead.active ? ~0u : 0u;
    const uint4 *d4 = reinterpret_cast<const uint4 *>(w.data);
    const int nchunks = w.n >> 4;
    uint32_t flagged = 0;
    // two chunks of a lane at a time, so that a variant's mode, addresses and constants are read once
    // for both
    for (int c = warp * 32 + lane; c < nchunks; c += 2 * T) {
        const bool two = c + T < nchunks;  // the same for the whole warp
        uint32_t x[2][4], f[2][4], bits[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 a = h == 0 || two ? d4[c + h * T] : make_uint4(0u, 0u, 0u, 0u);
            x[h][0] = a.x;
            x[h][1] = a.y;
            x[h][2] = a.z;
            x[h][3] = a.w;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t ad = __vabsdiffu4(x[h][q] ^ 0x80808080u, k.mb4);
                f[h][q] = prmt(ge_bytes_msb(ad, k.tlo7, k.tsmall) & on, 0u, 0xBA98u);
            }
            bits[h] = chunk_bits(f[h][0], f[h][1], f[h][2], f[h][3]);
        }
        flagged += __popc(bits[0]) + (two ? __popc(bits[1]) : 0);
        for (uint32_t g = grp; g; g &= g - 1u) {
            const int u = __ffs(static_cast<int>(g)) - 1;
            const uint32_t mode = sm.pass->mode[u];
            const uint32_t c4 = mode == 1u ? sm.cp->vrep[u].c4 : 0u;
            uint4 *const out = reinterpret_cast<uint4 *>(sm.pass->out[u]) + c;
            uint16_t *const mk = sm.pass->mask[u] + c;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && !two) break;
                uint32_t o[4];
                if (mode == 3u) {  // the noise overwrites every flagged sample
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[q] = x[h][q];
                } else if (mode == 2u) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint32_t up =
                            k.unone ? 0u : prmt(ge_bytes_msb(x[h][q] ^ 0x80808080u, k.ulo7, k.usmall), 0u, 0xBA98u);
                        o[q] = (x[h][q] & ~f[h][q]) | (((k.hi4 & up) | (k.lo4 & ~up)) & f[h][q]);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[q] = (x[h][q] & ~f[h][q]) | (c4 & f[h][q]);
                }
                __stcs(out + h * T, make_uint4(o[0], o[1], o[2], o[3]));
                mk[h * T] = static_cast<uint16_t>(bits[h]);
            }
        }
        if (noise) {
            noise_note8(sm, lane, c, bits[0], nlc);
            if (two) noise_note8(sm, lane, c + T, bits[1], nlc);
        }
    }
    return flagged;
}

// ------------------------------------------------------------------ one window
// All T threads of the group call this. The 12-bit tables must be zero at a group's first window.
// Uses the group's named barrier after the histogram, after the reduce and after the search. There is no barrier at the end: each warp adds its flag count and marks itself done,
// and the last warp of the window (window parity `par`) writes the count, median and MAD to
// slot `widx` of the segment and, when release_bar != 0, releases the stage through it.
// `stage_ok` is this thread's result of waiting for the stage (false: timed out); the first
// barrier combines it, and the function returns false if any thread of the group timed out.
//
// MODE & 3 is the replacement mode (rfi_mode); the other bits select a form of the pass. For
// the Median-of-MAD variant (Eq. 3), kModeStats runs phases 1-4 only and writes M and D, and
// kModeApply skips phases 1-4, reads the window's M from sg.med and its dispersion from sg.mad
// and runs phase 5 (amd, when given, holds the window's {M, dispersion} in shared memory).
// kModePower also sums x^2 and z^2 over the window into sg.power.
template <int BITS, int MODE, int T, int ROWB, bool ALONE = false>
__device__ bool process_window(const Shm &sm, const Win &w, const Seg &sg, int64_t widx, const Params &p,
                               int tid, int par, uint32_t release_bar, bool stage_ok, RowSums &rs,
                               const int2 *amd = nullptr, const Seg *vsegs = nullptr) {
    constexpr int NW = T / 32;
    constexpr bool STATS = (MODE & kModeStats) != 0;
    constexpr bool APPLY = (MODE & kModeApply) != 0;
    constexpr bool PW = (MODE & kModePower) != 0;
    constexpr bool COPIES = (MODE & kModeCopies) != 0;
    constexpr int OUTF = (MODE & kModeF16) ? 1 : ((MODE & kModeBF16) ? 2 : 0);
    constexpr int RMODE = MODE & 3;
    constexpr bool ANY = (MODE & kModeAny) != 0;
    constexpr bool TIGHT = (MODE & kModeTight) != 0;
    const int lane = tid & 31;
    if (STATS) {
        // Estimation only (the first pass of Eq. 3): M and D of the window. Nothing reads the
        // stage after the histogram, so the tile's last window releases it there; the search
        // warp writes M and D itself while the other warps go on to the next window. sg lives in
        // the stage's descriptor, which the copy warp rewrites once the stage is released: its
        // output pointers are taken first.
        int32_t *const med = sg.med, *const mad = sg.mad;
        if (stage_ok) {
            if constexpr (ANY) phase_histogram_any<BITS, T>(sm, w, tid, par);
            else phase_histogram<BITS, T, ROWB>(sm, w, tid, par);
        }
        if (named_bar_or(sm.bar_id, T, !stage_ok)) return false;
        if (tid == 0 && release_bar) mbar_arrive(release_bar);
        // int8: the counts go to one warp, which scans them and searches while the other warps
        // start the next window (one group barrier fewer than a block-wide scan)
        if constexpr (BITS == 8) phase_reduce8_counts<T, ROWB>(sm, tid, rs);
        else phase_rows12<T>(sm, tid, par, TIGHT ? table12(sm, par ^ 1) : sm.coarse);
        named_bar(sm.bar_id, T);
        if (tid < 32) {
            if constexpr (BITS == 8) {
                phase_search8<MODE>(sm, w.n, lane, p.kq, p.cval);
            } else {
                phase_search12<MODE>(sm, table12(sm, par), TIGHT ? table12(sm, par ^ 1) : sm.coarse, TIGHT, w.n, lane, p.kq,
                                     p.cval);
            }
            if (lane == 0) {  // the lane that wrote the record
                if (med) med[widx] = sm.ctl->rep.M;
                if (mad) mad[widx] = sm.ctl->rep.D;
                if (BITS == 12 && atomicExch(&sm.ctl->err[par], 0u)) atomicOr(p.status, kStatusSampleRange);
            }
        }
        if (TIGHT) named_bar(sm.bar_id, T);  // the search worked in the next window's table
        return true;
    }
    if (!APPLY) {
        if (stage_ok) {
            if constexpr (ANY) phase_histogram_any<BITS, T>(sm, w, tid, par);
            else phase_histogram<BITS, T, ROWB>(sm, w, tid, par);
        }
        if (named_bar_or(sm.bar_id, T, !stage_ok)) return false;
        if constexpr (BITS == 8) phase_reduce8_counts<T, ROWB>(sm, tid, rs);
        else phase_rows12<T>(sm, tid, par, table12(sm, par ^ 1));
        named_bar(sm.bar_id, T);
        if (tid < 32) {
            if constexpr (BITS == 8) {
                phase_search8<MODE>(sm, w.n, lane, p.kq, p.cval);
            } else {
                phase_search12<MODE>(sm, table12(sm, par), table12(sm, par ^ 1), true, w.n, lane, p.kq, p.cval);
            }
        }
    } else {
        // every thread has read the previous window's values before this barrier
        if (named_bar_or(sm.bar_id, T, !stage_ok)) return false;
        if (tid == 0) {  // from the stage's copy (amd) when the copy warp brought it along
            const int2 md = amd ? *amd : make_int2(sg.med[widx], sg.mad[widx]);
            sm.ctl->rep = make_rep<BITS, MODE>(md.x, md.y, p.kq, p.cval);
        }
    }
    named_bar(sm.bar_id, T);
    const Rep r = load_rep(sm.ctl->rep);
    uint32_t f = 0;
    Pow pw = {0u, 0u};
    const KeysPre key{p};
    // the replace pass, and the digital noise of the samples it listed
    auto replace = [&](uint32_t *nlc, int slice, int send) {
        if constexpr (ANY) return phase_replace_any<BITS, RMODE, T, KeysPre>(sm, w, r, key, tid, nlc, pw, &sm.ctl->rep, slice, send);
        else return phase_replace<BITS, RMODE, T, PW, KeysPre, OUTF, (MODE & kModeFlaggedOnly) != 0>(sm, w, r, key, tid, nlc, pw,
                                                                                                    &sm.ctl->rep, slice, send);
    };
    if constexpr (!STATS && !COPIES) {
        uint32_t *const nlc = &sm.ctl->ncount[2 * par];
        if constexpr (BITS == 12 && RMODE == 3) {
            f = noise_slices12<T, ANY, ALONE>(sm, w, nlc, tid, replace, [&](const uint32_t *c) {
                noise_list<12, T, PW, KeysPre, OUTF>(sm, w, r, key, tid, c, pw);
            });
        } else {
            f = replace(nlc, 0, 0);
            if constexpr (RMODE == 3) noise_deferred8<T, PW, noise_pairs(MODE), KeysPre, OUTF>(sm, w, r, key, tid, nlc, pw);
        }
    }
    if (COPIES) {
        // every variant's values from the window's M and D, then its replace pass
        const int nvar = params_nvar(p);
        // variants share passes over whole rounds with aligned buffers and masks and without mask words past the
        // window's last sample (the shared pass writes none); where the first variant's are not so, warp 0
        // gathers nothing for it
        const bool may = BITS == 8 && params_share(p) && w.vec && w.mask && (w.n & 511) == 0 && w.n == 32 * w.mask_words;
        if (tid < 32) {
            bool slow = !may;
            if (tid < nvar) {
                const Variant vr = params_var(p)[tid];
                sm.cp->vrep[tid] = make_rep<BITS, kRepAll>(r.M, r.D, vr.kq, vr.cval);
                if (BITS == 8 && may) {
                    const Seg &sv = vsegs[static_cast<int64_t>(tid) * params_seg_stride(p)];
                    uint32_t grp = 0u;
                    for (int u = 0; u < nvar; ++u) grp |= params_var(p)[u].kq == vr.kq ? 1u << u : 0u;
                    sm.pass->group[tid] = grp;
                    sm.pass->mode[tid] = static_cast<uint32_t>(vr.mode);
                    sm.pass->out[tid] = sv.out + widx * sv.W;
                    sm.pass->mask[tid] = reinterpret_cast<uint16_t *>(sv.mask + widx * sv.mask_words);
                    slow = sv.vec == 0 || sv.mask == nullptr;
                }
            }
            const bool any_slow = __any_sync(0xFFFFFFFFu, slow);
            if (BITS == 8 && tid == 0) sm.pass->fast = any_slow ? 0u : 1u;
        }
        named_bar(sm.bar_id, T);
        uint32_t todo = BITS == 8 && sm.pass->fast ? (1u << nvar) - 1u : 0u;
        const bool grouped = todo != 0u;
        while (todo) {
            const int v = __ffs(static_cast<int>(todo)) - 1;
            const uint32_t grp = sm.pass->group[v];
            todo &= ~grp;
            uint32_t noise = 0u;
            for (int u = v; u < nvar; ++u) noise |= ((grp >> u) & 1u) != 0u && sm.pass->mode[u] == 3u ? 1u << u : 0u;
            uint32_t *nc = &sm.cp->ncount[4 * v + 2 * par];
            uint32_t fv = copies_pass8<T>(sm, w, v, grp, noise != 0u, tid, nc);
            fv = __reduce_add_sync(0xFFFFFFFFu, fv);
            if (lane < nvar && ((grp >> lane) & 1u) && fv) atomicAdd(&sm.cp->vcount[lane][par], fv);
            __syncwarp();  // lane 0 announces the window for every lane that counted
            for (uint32_t m = noise; m; m &= m - 1u) {  // the same list, each with its own key
                const int u = __ffs(static_cast<int>(m)) - 1;
                Win wu = w;
                wu.out = sm.pass->out[u];
                const uint64_t seed = params_var(p)[u].seed;
                noise_deferred8<T, false, false>(sm, wu, load_rep(sm.cp->vrep[u]),
                                                 KeysSeed{static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32)}, tid, nc,
                                                 pw);
            }
            if (noise && todo) named_bar(sm.bar_id, T);  // the next group lists its own
        }
        if (!grouped)
        for (int v = 0; v < params_nvar(p); ++v) {
            uint32_t *nc = &sm.cp->ncount[4 * v + 2 * par];
            const Variant vr = params_var(p)[v];
            const Seg &sv = vsegs[static_cast<int64_t>(v) * params_seg_stride(p)];
            Win wv = w;
            wv.out = sv.out + widx * sv.W * Geo<BITS>::kBps;
            wv.mask = sv.mask ? sv.mask + widx * sv.mask_words : nullptr;
            wv.vec = sv.vec != 0;
            const Rep rv = load_rep(sm.cp->vrep[v]);
            const KeysSeed vkey{static_cast<uint32_t>(vr.seed), static_cast<uint32_t>(vr.seed >> 32)};
            uint32_t fv;
            switch (vr.mode) {
                case 0: fv = phase_replace<BITS, 0, T, false>(sm, wv, rv, vkey, tid, nc, pw, &sm.cp->vrep[v]); break;
                case 1: fv = phase_replace<BITS, 1, T, false>(sm, wv, rv, vkey, tid, nc, pw, &sm.cp->vrep[v]); break;
                case 2: fv = phase_replace<BITS, 2, T, false>(sm, wv, rv, vkey, tid, nc, pw, &sm.cp->vrep[v]); break;
                default:
                    if constexpr (BITS == 12) {
                        fv = noise_slices12<T, false, false>(
                            sm, wv, nc, tid,
                            [&](uint32_t *c, int slice, int send) {
                                return phase_replace<BITS, 3, T, false>(sm, wv, rv, vkey, tid, c, pw, &sm.cp->vrep[v], slice, send);
                            },
                            [&](const uint32_t *c) { noise_list<BITS, T, false>(sm, wv, rv, vkey, tid, c, pw); });
                    } else {
                        fv = phase_replace<BITS, 3, T, false>(sm, wv, rv, vkey, tid, nc, pw, &sm.cp->vrep[v]);
                        noise_deferred8<T, false, false>(sm, wv, rv, vkey, tid, nc, pw);
                    }
                    // the noise work area and the first indices are reused by the next variant
                    if (v + 1 < params_nvar(p)) named_bar(sm.bar_id, T);
                    break;
            }
            fv = __reduce_add_sync(0xFFFFFFFFu, fv);
            if (lane == 0 && fv) atomicAdd(&sm.cp->vcount[v][par], fv);
        }
    }
    f = __reduce_add_sync(0xFFFFFFFFu, f);
    unsigned long long px = 0ull, pz = 0ull;
    if (PW) {  // warp sums in two 16-bit halves, so that no partial sum overflows 32 bits
        px = (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, pw.x >> 16)) << 16) +
             __reduce_add_sync(0xFFFFFFFFu, pw.x & 0xFFFFu);
        pz = (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, pw.z >> 16)) << 16) +
             __reduce_add_sync(0xFFFFFFFFu, pw.z & 0xFFFFu);
    }
    if (lane == 0) {
        if (f) atomicAdd(&sm.ctl->count[par], f);
        if (PW) {
            atomicAdd(&sm.ctl->pw[par][0], px);
            atomicAdd(&sm.ctl->pw[par][1], pz);
        }
        __threadfence_block();
        if (atomicAdd(&sm.ctl->done[par], 1u) == NW - 1) {
            // last warp of this window: every count is in and every read of the stage is done
            __threadfence_block();
            const uint32_t cnt = atomicExch(&sm.ctl->count[par], 0u);
            sm.ctl->done[par] = 0u;
            if (RMODE == 3 && !COPIES) {  // every warp has read them
                sm.ctl->ncount[2 * par] = 0u;
                if (BITS == 12) {
                    sm.ctl->ncount[2 * par + 1] = 0u;
                    sm.ctl->wide = 8u * cnt <= 7u * kNoiseList;
                }
            }
            if (COPIES) {
                uint32_t most = 0u;
                for (int v = 0; v < params_nvar(p); ++v) {
                    const uint32_t cv = atomicExch(&sm.cp->vcount[v][par], 0u);
                    most = cv > most ? cv : most;
                    sm.cp->ncount[4 * v + 2 * par] = 0u;
                    sm.cp->ncount[4 * v + 2 * par + 1] = 0u;
                    const Seg &sv = vsegs[static_cast<int64_t>(v) * params_seg_stride(p)];
                    if (sv.counts) sv.counts[widx] = cv;
                    sm.ctl->flagged += cv;
                }
                if (BITS == 12) sm.ctl->wide = 8u * most <= 7u * kNoiseList;
            }
            if (PW) {
                const unsigned long long sx = atomicExch(&sm.ctl->pw[par][0], 0ull);
                const unsigned long long sz = atomicExch(&sm.ctl->pw[par][1], 0ull);
                if (sg.power) {
                    sg.power[2 * widx] = sx;
                    sg.power[2 * widx + 1] = sz;
                }
            }
            if (!COPIES && sg.counts) sg.counts[widx] = cnt;
            if (!APPLY && sg.med) sg.med[widx] = r.M;
            if (!APPLY && sg.mad) sg.mad[widx] = r.D;
            sm.ctl->flagged += cnt;
            if (BITS == 12 && atomicExch(&sm.ctl->err[par], 0u)) atomicOr(p.status, kStatusSampleRange);
            if (release_bar) mbar_arrive(release_bar);
        }
    }
    return true;
}

// ------------------------------------------------------------------ replace pass over a tile
// Eq. 1 and Eq. 2 over a whole tile of nw full int8 windows of one segment, W = 2^lw samples
// each, 16-byte aligned, window k (of the tile) with the thresholds reps[k] already in shared
// memory: the replace pass over all of the tile's chunks (a warp's round of 32 chunks lies in
// one window, whose flag count takes one shared atomic), then the digital noise of the listed
// chunks as in noise_deferred8, each sample taking its window's M and spread. The last warp
// writes the windows' counts from cnt (and zeroes them) and, when release_bar != 0, releases
// the stage. Windows start at window w0 of the segment.
template <int RMODE, int T>
__device__ void replace_tile8(const Shm &sm, const uint8_t *stage, const Seg &sg, uint32_t w0, int nw, int lw,
                              const RepShared *reps, uint32_t *cnt, const Params &p, int tid, int par,
                              uint32_t release_bar, const TileNoise &tn) {
    constexpr int NW = T / 32;
    const int lane = tid & 31, warp = tid >> 5;
    const int lcw = lw - 4;  // log2 of the chunks per window
    const int nchunks = nw << lcw;
    const uint4 *d4 = reinterpret_cast<const uint4 *>(stage);
    uint8_t *out = sg.out + (static_cast<int64_t>(w0) << lw);
    uint16_t *mk = sg.mask ? reinterpret_cast<uint16_t *>(sg.mask + static_cast<int64_t>(w0) * sg.mask_words)
                           : nullptr;
    for (int c0 = warp * 32; c0 < nchunks; c0 += T) {
        const int k = c0 >> lcw;
        const RepShared &rk = reps[k];
        const Rep8 k8 = load_rep8(&rk);
        const int c = c0 + lane;
        uint4 v = d4[c];
        uint32_t bits = 0;
        if (rk.active) {
            uint32_t f0, f1, f2, f3;
            v.x = rep8_word<RMODE>(v.x, k8, f0);
            v.y = rep8_word<RMODE>(v.y, k8, f1);
            v.z = rep8_word<RMODE>(v.z, k8, f2);
            v.w = rep8_word<RMODE>(v.w, k8, f3);
            bits = chunk_bits(f0, f1, f2, f3);
        }
        store_chunk8<0>(out, c, v, true);
        if (mk) mk[c] = static_cast<uint16_t>(bits);
        if (RMODE == 3) noise_note8(sm, lane, c, bits, &sm.ctl->ncount[2 * par]);
        const uint32_t wf = __reduce_add_sync(0xFFFFFFFFu, __popc(bits));
        if (lane == 0 && wf) atomicAdd(&cnt[k], wf);
    }

    if (RMODE == 3) {
        named_bar(sm.bar_id, T);  // every entry of the tile is in the list
        const KeysPre key{p};
        const NoiseRun<8, KeysPre> run(key, sg.stream_id, static_cast<uint64_t>(sg.abs0 + (static_cast<int64_t>(w0) << lw)), tn);
        const uint32_t n = sm.ctl->ncount[2 * par];
        if (run.one_hi) {
            noise_expand8<T, false>(
                sm, n, tid,
                [&](uint32_t pos) {
                    const RepShared &rk = reps[pos >> lw];
                    out[pos] = static_cast<uint8_t>(run.value(pos, rk.sig2, rk.moff));
                },
                [](uint32_t, uint32_t) {});
        } else {
            noise_expand8_any<T>(sm, n, tid, [&](uint32_t pos) {
                const RepShared &rk = reps[pos >> lw];
                out[pos] = static_cast<uint8_t>(run.value_any(pos, rk.sig2, rk.moff));
            });
        }
    }

    if (lane == 0) {
        __threadfence_block();
        if (atomicAdd(&sm.ctl->done[par], 1u) == NW - 1) {
            // last warp of the tile: every count is in and every read of the stage is done
            __threadfence_block();
            sm.ctl->done[par] = 0u;
            if (RMODE == 3) sm.ctl->ncount[2 * par] = 0u;  // every warp has read it
            unsigned long long tot = 0ull;
            for (int k = 0; k < nw; ++k) {
                const uint32_t ck = cnt[k];
                cnt[k] = 0u;
                if (sg.counts) sg.counts[w0 + k] = ck;
                tot += ck;
            }
            sm.ctl->flagged += tot;
            if (release_bar) mbar_arrive(release_bar);
        }
    }
}

// ------------------------------------------------------------------ apply pass over a tile
// The apply pass (Eq. 1 and Eq. 2 around each window's given M with its given dispersion, as
// for the median of MADs of Eq. 3) over a whole tile of nw full int8 windows of one segment,
// W = 2^lw >= 512 samples each, 16-byte aligned: one barrier for the tile's thresholds (thread
// k builds window k's), then replace_tile8. Against one window at a time this saves three
// barriers per window and keeps every thread busy on windows of 4096 samples, which give 256
// threads one chunk each.
template <int MODE, int T>
__device__ bool process_tile_apply8(const Shm &sm, const uint8_t *stage, const Tile &tl, const Seg &sg,
                                    const int2 *amd, const Params &p, int tid, int par, int lw,
                                    uint32_t release_bar, bool stage_ok, const TileNoise &tn) {
    const int nw = static_cast<int>(tl.nw);
    // every thread has finished the previous tile or window (its thresholds, counts, noise
    // work area) before this barrier
    if (named_bar_or(sm.bar_id, T, !stage_ok)) return false;
    RepShared *reps = sm.at->rep;
    if (tid < nw) reps[tid] = make_rep<8, MODE>(amd[tid].x, amd[tid].y, p.kq, p.cval);
    named_bar(sm.bar_id, T);
    replace_tile8<MODE & 3, T>(sm, stage, sg, tl.w0, nw, lw, reps, sm.at->count, p, tid, par, release_bar, tn);
    return true;
}

// ------------------------------------------------------------------ multi-window tiles
// Histogram of up to K windows of 2^lw samples at once: window slot g (< nw) is counted by the
// 32/K lanes (32/K)g .. of every warp into their own columns of the lane-striped table, so the
// atomics stay conflict-free and the slots never mix.
template <int T, int K>
__device__ __forceinline__ void hist8_multi(const Shm &sm, const uint8_t *stage, int lw, int nw, int tid) {
    constexpr int LPS = 32 / K;  // lanes per slot
    constexpr int TS = T / K;    // threads per slot
    const int lane = tid & 31, warp = tid >> 5;
    const int g = lane / LPS;
    if (g >= nw) return;
    const int i = warp * LPS + (lane % LPS);
    const uint32_t lb = sm.hist_s + 4u * lane;
    const uint4 *d4 = reinterpret_cast<const uint4 *>(stage + (g << lw));
    const int nch = 1 << (lw - 4);
    int c = i;
    for (; c + TS < nch; c += 2 * TS) {
        const uint4 a = d4[c], b = d4[c + TS];
        hist8_word<128>(lb, a.x); hist8_word<128>(lb, a.y); hist8_word<128>(lb, a.z); hist8_word<128>(lb, a.w);
        hist8_word<128>(lb, b.x); hist8_word<128>(lb, b.y); hist8_word<128>(lb, b.z); hist8_word<128>(lb, b.w);
    }
    if (c < nch) {
        const uint4 a = d4[c];
        hist8_word<128>(lb, a.x); hist8_word<128>(lb, a.y); hist8_word<128>(lb, a.z); hist8_word<128>(lb, a.w);
    }
}

// Counts of every slot from the table, which is zeroed as it is read (the 128-byte row of raw
// byte u holds lane l's count at word l; a slot's lanes are 8/K of the row's eight 16-byte
// groups). The eight threads tid & ~7 .. tid | 7 read the eight groups of the same row, so the
// reads and clears are free of bank conflicts; with four slots, thread pairs combine their
// groups by a shuffle. A warp takes four neighbouring rows at a time, so that its 16-bit stores fall
// into two neighbouring words of each slot (rows 8 apart met in a bank four ways). Counts go to 16-bit arrays, 264 entries apart (slot g's array starts
// on bank 4g, so the stores of one row's slots do not collide either, and on a 16-byte boundary).
template <int T, int K>
__device__ __forceinline__ void reduce8_multi(const Shm &sm, int tid) {
    static_assert(K == 4 || K == 8, "four or eight window slots");
    constexpr int RPT = 256 / (T / 8);  // rows per thread
    const int p = tid & 7;
    uint4 *tab = reinterpret_cast<uint4 *>(sm.hist);
    uint16_t *cumg = reinterpret_cast<uint16_t *>(sm.cum) + (K == 8 ? p : (p >> 1)) * Geo<8>::kCumWords;
#pragma unroll 4
    for (int k = 0; k < RPT; ++k) {
        const int row = (tid >> 3) + k * (T / 8);
        uint4 *a = tab + row * 8 + p;
        const uint4 v = *a;
        *a = make_uint4(0u, 0u, 0u, 0u);
        uint32_t sum = v.x + v.y + v.z + v.w;
        if (K == 4) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
        if (K == 8 || (p & 1) == 0) cumg[row ^ 128] = static_cast<uint16_t>(sum);
    }
}

// One warp: the inclusive scan of a slot's 256 counts in place (8 consecutive bins per lane, one
// 16-byte load and store), then its lower median bin and MAD (as phase_search8), and the threshold and replacement values into *rep (lane 0). The counts and
// cumulative counts are 16-bit (a window of this form has at most 8192 samples).
template <int MODE>
__device__ __forceinline__ void scan_search8(uint16_t *cum, int n, int lane, int64_t kq, int32_t cval,
                                             RepShared *rep) {
    uint4 *const own = reinterpret_cast<uint4 *>(cum) + lane;
    const uint4 h = *own;
    const uint32_t hw[4] = {h.x, h.y, h.z, h.w};
    uint32_t c[8];
    uint32_t run = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        run += hw[j] & 0xFFFFu;
        c[2 * j] = run;
        run += hw[j] >> 16;
        c[2 * j + 1] = run;
    }
    uint32_t inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t excl = inc - run;
    const uint32_t half = static_cast<uint32_t>((n + 1) >> 1);
    // bins whose cumulative count stays below half the window lie below the median bin
    uint32_t below = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        c[j] += excl;
        below += c[j] < half ? 1u : 0u;
    }
    *own = make_uint4(c[0] | (c[1] << 16), c[2] | (c[3] << 16), c[4] | (c[5] << 16), c[6] | (c[7] << 16));
    const int mb = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, below));
    __syncwarp();
    const int d = warp_search<256>(lane, [&](int dd) {
        const int hi = mb + dd < 255 ? mb + dd : 255;
        const int lo = mb - dd - 1;
        const uint32_t f = static_cast<uint32_t>(cum[hi]) - (lo >= 0 ? static_cast<uint32_t>(cum[lo]) : 0u);
        return f >= half;
    });
    if (lane == 0) *rep = make_rep<8, MODE>(mb - Geo<8>::kOffset, d, kq, cval);
}

// A tile of nw (1 <= nw <= K) full int8 windows of 2^lw samples, 16-byte aligned, in shared
// memory at stage, for the plain excision modes (MODE 0..3) or the estimation pass of the
// Median of MAD (kModeStats). The histogram table must be zero on entry and is zero again
// after the reduce. Barriers: after the histogram (a bar.red.or that also agrees on a timeout),
// after the reduce, and, for excision, after the searches; warp w searches windows w, w + NW,
// ... M and D go straight to the segment's arrays. release_bar (nonzero for the tile's last
// windows) releases the stage: after the histogram for kModeStats, else after the replace pass.
template <int MODE, int T, int K>
__device__ bool process_tile_multi8(const Shm &sm, const uint8_t *stage, const Seg &sg, uint32_t w0, int nw, int lw,
                                    const Params &p, int tid, int par, uint32_t release_bar, bool stage_ok,
                                    const TileNoise &tn) {
    constexpr bool STATS = (MODE & kModeStats) != 0;
    constexpr int NW = T / 32;
    const int lane = tid & 31, warp = tid >> 5;
    int32_t *const med = sg.med, *const mad = sg.mad;  // sg lives in the stage descriptor
    if (stage_ok) hist8_multi<T, K>(sm, stage, lw, nw, tid);
    if (named_bar_or(sm.bar_id, T, !stage_ok)) return false;
    if (STATS && tid == 0 && release_bar) mbar_arrive(release_bar);
    reduce8_multi<T, K>(sm, tid);
    named_bar(sm.bar_id, T);
    for (int g = warp; g < nw; g += NW) {
        RepShared *rep = &sm.mt->rep[g];
        scan_search8<MODE>(reinterpret_cast<uint16_t *>(sm.cum) + g * Geo<8>::kCumWords, 1 << lw, lane, p.kq, p.cval, rep);
        __syncwarp();
        if (lane == 0) {
            if (med) med[w0 + g] = rep->M;
            if (mad) mad[w0 + g] = rep->D;
        }
    }
    if (STATS) return true;
    named_bar(sm.bar_id, T);
    replace_tile8<MODE & 3, T>(sm, stage, sg, w0, nw, lw, sm.mt->rep, sm.mt->count, p, tid, par, release_bar, tn);
    return true;
}

// ------------------------------------------------------------------ multi-window tiles of any windows
// nw (1 <= nw <= K) windows of up to 8192 samples each, of any length at any alignment: window slot g
// starts off + g * W bytes into the stage, the last one may be shorter. As process_tile_multi8 with
// the histogram and replace rounds of the any-window form; a warp's replace round is 31 chunks of
// one window. A noise-list entry's chunk number holds the slot above bit 10 (a window of 8192
// samples has at most 514 chunks).
template <int MODE, int T, int K>
__device__ bool process_tile_any8(const Shm &sm, const uint8_t *stage, int off, const Seg &sg, uint32_t w0, int nw,
                                  const Params &p, int tid, int par, uint32_t release_bar, const TileNoise &tn) {
    constexpr bool STATS = (MODE & kModeStats) != 0;
    constexpr int RMODE = MODE & 3;
    constexpr int NW = T / 32, LPS = 32 / K, TS = T / K;
    static_assert(TS >= 32, "hist_chunks needs 32 threads per window");
    const int lane = tid & 31, warp = tid >> 5;
    int32_t *const med = sg.med, *const mad = sg.mad;  // sg lives in the stage descriptor
    const int W = sg.W;
    const int64_t left = sg.len - static_cast<int64_t>(w0) * W;
    auto window = [&](int g) {
        Win w;
        const int64_t k = static_cast<int64_t>(w0) + g;
        const int64_t left = sg.len - k * W;
        const int at = off + g * W;
        w.data = stage + (at & ~15);
        w.off = at & 15;
        w.n = static_cast<int32_t>(left < W ? left : W);
        w.out = sg.out + k * W;
        w.mask = sg.mask ? sg.mask + k * sg.mask_words : nullptr;
        w.mask_words = sg.mask_words;
        w.abs_idx = sg.abs0 + k * W;
        w.sid = sg.stream_id;
        w.tn = &tn;
        w.vec = ((reinterpret_cast<uintptr_t>(w.out) - w.off) & 15u) == 0u;
        return w;
    };
    if (lane / LPS < nw) {
        const Win w = window(lane / LPS);
        const uint32_t lb = sm.hist_s + 4u * lane;
        hist_chunks<8>(w, warp * LPS + lane % LPS, TS, [&](uint32_t v) { hist8_word<128>(lb, v); },
                       [&](int at) { red_add_shared(lb + (static_cast<uint32_t>(w.data[at]) << 7), 1u); });
    }
    if (named_bar_or(sm.bar_id, T, false)) return false;
    if (STATS && tid == 0 && release_bar) mbar_arrive(release_bar);
    reduce8_multi<T, K>(sm, tid);
    named_bar(sm.bar_id, T);
    for (int g = warp; g < nw; g += NW) {
        RepShared *rep = &sm.mt->rep[g];
        const int64_t lg = left - static_cast<int64_t>(g) * W;
        scan_search8<MODE>(reinterpret_cast<uint16_t *>(sm.cum) + g * Geo<8>::kCumWords, static_cast<int>(lg < W ? lg : W), lane,
                     p.kq, p.cval, rep);
        __syncwarp();
        if (lane == 0) {
            if (med) med[w0 + g] = rep->M;
            if (mad) mad[w0 + g] = rep->D;
        }
    }
    if (STATS) return true;
    named_bar(sm.bar_id, T);
    if constexpr (!STATS) {
        const RepShared *reps = sm.mt->rep;
        const int rpw = ((15 + W + 15) / 16 + 30) / 31;  // rounds of a window
        for (int q = warp; q < nw * rpw; q += NW) {
            const int g = q / rpw, base = (q - g * rpw) * 31;
            const Win w = window(g);
            const uint32_t bits = replace_round_any<8, RMODE>(w, load_rep(reps[g]), &reps[g], base, lane);
            if (RMODE == 3) noise_note8(sm, lane, (g << 10) + base + lane, bits, &sm.ctl->ncount[2 * par]);
            const uint32_t wf = __reduce_add_sync(0xFFFFFFFFu, __popc(bits));
            if (lane == 0 && wf) atomicAdd(&sm.mt->count[g], wf);
            if (base == 0) mask_padding<8>(w, lane, 32);
        }
        if (RMODE == 3) {
            named_bar(sm.bar_id, T);  // every entry of the windows is in the list
            const KeysPre key{p};
            uint8_t *const out = sg.out + static_cast<int64_t>(w0) * W;
            const NoiseRun<8, KeysPre> run(key, sg.stream_id, static_cast<uint64_t>(sg.abs0 + static_cast<int64_t>(w0) * W), tn);
            const uint32_t n = sm.ctl->ncount[2 * par];
            auto where = [&](uint32_t at, int g) {  // entry position -> sample of the tile
                return static_cast<uint32_t>(g * W + static_cast<int>(at & 16383u) - ((off + g * W) & 15));
            };
            if (run.one_hi) {
                noise_expand8<T, false>(
                    sm, n, tid,
                    [&](uint32_t at) {
                        const int g = static_cast<int>(at >> 14);
                        const uint32_t pos = where(at, g);
                        out[pos] = static_cast<uint8_t>(run.value(pos, reps[g].sig2, reps[g].moff));
                    },
                    [](uint32_t, uint32_t) {});
            } else {
                noise_expand8_any<T>(sm, n, tid, [&](uint32_t at) {
                    const int g = static_cast<int>(at >> 14);
                    const uint32_t pos = where(at, g);
                    out[pos] = static_cast<uint8_t>(run.value_any(pos, reps[g].sig2, reps[g].moff));
                });
            }
        }
        if (lane == 0) {
            __threadfence_block();
            if (atomicAdd(&sm.ctl->done[par], 1u) == NW - 1) {
                // last warp: every count is in and every read of the stage is done
                __threadfence_block();
                sm.ctl->done[par] = 0u;
                if (RMODE == 3) sm.ctl->ncount[2 * par] = 0u;  // every warp has read it
                unsigned long long tot = 0ull;
                for (int g = 0; g < nw; ++g) {
                    const uint32_t cg = sm.mt->count[g];
                    sm.mt->count[g] = 0u;
                    if (sg.counts) sg.counts[w0 + g] = cg;
                    tot += cg;
                }
                sm.ctl->flagged += tot;
                if (release_bar) mbar_arrive(release_bar);
            }
        }
    }
    return true;
}

}  // namespace dev
}  // namespace rfi
