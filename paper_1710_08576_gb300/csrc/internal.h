// Internal interface between the plan (host C++) and the excision kernels (CUDA).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rfi {

// Bits that kernels OR into the plan's device status word.
constexpr uint32_t kStatusSampleRange = 1u;  // reported as RFI_ERR_SAMPLE_RANGE
constexpr uint32_t kStatusTimeout = 2u;      // reported as RFI_ERR_TIMEOUT
constexpr uint32_t kStatusLayout = 4u;       // unexpected shared-memory window: RFI_ERR_UNSUPPORTED

// Kernel modes beyond the four replacement modes (rfi_mode 0..3), for the Median-of-MAD
// variant (Eq. 3): a pass that only estimates M and D per window, and passes that apply Eq. 1
// and Eq. 2 with a per-window centre and dispersion read from memory (kModeApply + rfi_mode).
constexpr int kModeStats = 4;
constexpr int kModeApply = 8;
constexpr int kApplyTileWindows = 32;  // at most this many windows per tile in apply passes
// Flag bit of the power-metered excision: the kernel also sums x^2 and z^2 over every window
// (the detected power of the unfiltered and filtered signal, for the improvement metric of
// Section III-A) and writes them to Seg::power.
constexpr int kModePower = 16;
// Flag bit of the digital-copy pass (Section III-A): one histogram, median and MAD per window and
// up to kMaxCopies (k, replacement) variants written to their own outputs. The variants come
// from Params::var; variant v of segment s is segment v * Params::seg_stride + s.
constexpr int kModeCopies = 32;
// Flag bits of the fused output format: write the excised samples as fp16 (int8 and 12-bit
// input) or bf16 (int8 input), the real-valued input a channeliser FFT reads. Both are exact.
constexpr int kModeF16 = 64;
constexpr int kModeBF16 = 128;
constexpr int kMaxCopies = 8;
// Flag bit of the multi-window form (8-bit, one consumer group; plain excision or the estimation
// pass): tiles of several small windows of 2^l samples (512..8192) are histogrammed together and
// share one reduce and one set of barriers. A separate instantiation, so that plans without such
// windows keep the plain kernel's shared-memory layout and code.
constexpr int kModeMulti = 256;
// Flag bit of the in-place form that writes back only what changes (RFI_PLAN_WRITE_FLAGGED):
// chunks without a flagged sample are not stored, and with digital noise no chunk is (the noise
// pass writes every flagged sample). Its own instantiation, like kModeMulti.
constexpr int kModeFlaggedOnly = 512;
// Flag bit of the split-warp form (8-bit zero, constant and threshold modes, also write-flagged,
// one group of 8 consumer warps): warps 0-3 histogram, reduce and search window n + 1 while
// warps 4-7 replace window n, handing each window's thresholds over through a ring of slots with
// mbarriers. Its own instantiation, chosen by the launch shape (Shape::warp_split == 2).
constexpr int kModeWarpSplit = 1024;

// Flag bit of the any-window form (plain excision, the estimation pass and the apply passes; one
// group of 8 consumer warps): the copy warp stages a tile's bytes as they lie in global memory,
// rounded out to 16-byte chunks, and the window phases take windows that start and end anywhere in
// a chunk; several 8-bit windows of up to kMultiMaxWindow samples of any length share a histogram
// table as in the multi-window form. For plans with windows that the aligned forms serve badly
// (any_form_gain). 24 int8 streams of 2^18..2^22 samples in windows of 1000..40000, threshold: 200 -> 65
// us a call (host included); 24 x 2466361 int8 samples in 2000-sample windows: 126 -> 77 us; 1.04 G
// 12-bit samples in 829-sample windows, noise: 28.8 -> 14.7 ms.
constexpr int kModeAny = 2048;
constexpr int kMultiMaxWindow = 8192;  // largest window that shares a table (16-bit counts, list entries)

// Windows of 2^l = 512..8192 int8 samples share a table in the multi-window form.
inline bool multi_window(int bits, int32_t W) {
    return bits == 8 && W >= 512 && W <= kMultiMaxWindow && (W & (W - 1)) == 0;
}
// Flag bit of the 12-bit estimation pass in shapes that leave no room for the rows' counts (fit_mode): they
// lie over the idle table, and the other warps wait for the search. Its own instantiation: as a
// branch of the usual one it cost that 2 % (1024-sample windows 1229 -> 1260 us a call).
constexpr int kModeTight = 4096;

// What the any-window form saves on a sample of a stream of windows W, in us per call of 60 x 2^22 samples
// (negative: what it costs). noise: digital noise in the excision kernel; mom: Median of MAD.
//  - Windows whose bytes are no multiple of 16 are loaded byte by byte by the aligned forms' consumers with
//    no copy in flight and stored byte by byte, one window a tile (int8, noise: 1001 samples 2112 aligned, 445
//    any; 8001: 1476, 296; 50001: 3392, 262; 12-bit 1001: 3096, 1291; Median of MAD 1001: 2582, 758).
//  - Other int8 windows of up to 8192 samples that are no power of two go one at a time through the
//    histogram's reduce and the barriers there (zero: 528 samples 1326 and 553, 1600: 468 and 315, 3200: 279
//    and 238, 4000: 233 and 221, 4800: 205 and 228, 8000: 152 and 239; noise: 528 samples 2133 and 657, 4800: 329
//    and 277, 8000: 231 and 287; Median of MAD 1600: 622 and 480, 4000: 300 and 281, 4800: 282 and 275).
//  - Windows of the multi-window form lose its fixed layout (zero: 512 samples 380 and 531, 2048: 166 and 257,
//    4096: 154 and 250; Median of MAD: 411 and 1121, -, 179 and 285), the rest a lane in 32 and the
//    stages' tighter fit (zero, 16384 samples: 118 and 142; 65536: 123 and 171; 12-bit 16384: 267 and 297;
//    Median of MAD 16384: 173 and 187).
inline int64_t any_form_gain(int bits, bool noise, bool mom, int32_t W, int64_t len) {
    const int bps = bits == 8 ? 1 : 2;
    if (static_cast<int64_t>(W) * bps % 16 != 0) return len <= 16 ? 0 : (mom ? 1800 : 1200);
    if (bits != 8) return -50;
    if (W > kMultiMaxWindow || len < 2 * static_cast<int64_t>(W)) return mom ? -15 : -40;
    if (multi_window(bits, W)) return mom ? -30 - 350000 / W : -100 - 25000 / W;
    return noise ? 860000 / W - 150 : 480000 / W - (mom ? 95 : 117);
}
// Windows per tile of a stage: as many whole ones as fit (the any-window form keeps 16 bytes for
// the tile's distance to the 16-byte boundary before it).
inline int64_t tile_windows(int bits, int mode, int32_t W, int stage_bytes) {
    const int64_t wb = static_cast<int64_t>(W) * (bits == 8 ? 1 : 2);
    if (mode & kModeAny) return (stage_bytes - 16) / wb > 1 ? (stage_bytes - 16) / wb : 1;
    return wb % 16 == 0 && stage_bytes / wb > 1 ? stage_bytes / wb : 1;
}
// Smallest stage for windows of up to wb bytes.
inline int min_stage_bytes(int mode, int64_t wb) {
    return static_cast<int>((wb + ((mode & kModeAny) ? 16 : 0) + 127) / 128 * 128);
}

// One variant of a digital-copy pass.
struct Variant {
    int64_t kq;     // round(k * 1.4826 * 2^16)
    uint64_t seed;  // noise key
    int32_t cval;   // constant replacement, already saturated
    int32_t mode;   // rfi_mode
};

// Device counters of one kernel pass, reset before it.
struct DevCounters {
    unsigned tile_counter;       // dynamic work-list cursor
    uint32_t status;             // kStatus* bits
    unsigned long long flagged;  // flagged samples of the pass
    unsigned fill_counter;       // work cursor of the digital-noise pass
    unsigned pad;
};

// One contiguous run of windows of one stream, starting on a window boundary.
struct Seg {
    const uint8_t *in;    // sample 0 of the run
    uint8_t *out;         // output sample 0
    uint32_t *mask;       // mask block of window 0 (nullable)
    uint32_t *counts;     // flagged count of window 0 (nullable)
    int32_t *med;         // median of window 0 (nullable)
    int32_t *mad;         // MAD of window 0 (nullable)
    int64_t len;          // samples in the run
    int64_t abs0;         // absolute stream index of sample 0 (multiple of W)
    int32_t W;            // window length
    uint32_t stream_id;   // Philox stream key
    int32_t mask_words;   // ceil(W / 32)
    int32_t vec;          // in/out 16-byte aligned and W * bytes_per_sample % 16 == 0
    uint64_t *power;      // detected power of window 0: {sum x^2, sum z^2} (nullable)
    uint32_t nwords;      // mask words of the run (set for the digital-noise pass)
    int32_t tidx;         // not of the table: a stage descriptor's tile index
};

// Work-list entry of the persistent kernel: windows [w0, w0 + nw) of segment seg.
struct Tile {
    uint32_t seg;
    uint32_t w0;
    uint32_t nw;
    uint32_t bytes;       // input bytes covered by the tile
};

// Method parameters shared by every window of a call.
struct Params {
    int64_t kq;                   // round(k * 1.4826 * 2^16)
    uint64_t seed;                // noise key
    int32_t cval;                 // constant replacement, already saturated
    int32_t ncopies;              // 12-bit histogram copies (1, 2 or 4)
    uint32_t *status;             // device status word (atomicOr of kStatus*)
    unsigned long long *flagged;  // device total of flagged samples
    uint32_t rk0[10], rk1[10];    // Philox4x32-10 round keys of `seed` (see set_round_keys)
    // Digital copy: the number of variants (bits 0-3), whether those of one multiple share a pass (bit
    // 4, copies_share), the distance between one variant's segment table and the next (bits 5-31), and the byte offset of the variant table from the
    // status word (both live in the plan's workspace). Packed into 8 bytes: a larger parameter
    // block changes the register allocation of every excision kernel for the worse.
    int32_t copies;
    int32_t var_off;
};

__host__ __device__ inline int params_nvar(const Params &p) { return p.copies & 15; }
__host__ __device__ inline bool params_share(const Params &p) { return (p.copies & 16) != 0; }
__host__ __device__ inline int params_seg_stride(const Params &p) { return p.copies >> 5; }
// Whether digital copies of n variants, variant v of multiple kq(v), run one pass per multiple. A variant that
// shares a pass saves 24 us of a call on 60 streams of 2^22 samples, but the pass that chooses its
// variants' replacements as it stores costs each multiple 15 us over the pass built for one (two multiples of
// four variants 626 us apart, 480 shared; one of two 208, 196; one of one 157, 171; eight of one 591, 708).
template <class Multiple>
inline bool copies_share(int n, Multiple &&kq) {
    int groups = 0;
    for (int v = 0; v < n; ++v) {
        bool first = true;
        for (int u = 0; u < v; ++u) first = first && kq(u) != kq(v);
        groups += first ? 1 : 0;
    }
    return 24 * (n - groups) > 15 * groups;
}
__host__ __device__ inline const Variant *params_var(const Params &p) {
    return reinterpret_cast<const Variant *>(reinterpret_cast<const char *>(p.status) + p.var_off);
}

// Philox4x32-10 key schedule: round r uses (seed_lo + r * 0x9E3779B9, seed_hi + r * 0xBB67AE85)
// (the Weyl increments of Salmon et al., SC'11), precomputed so kernels read them as constants.
inline void set_round_keys(Params &p) {
    uint32_t k0 = static_cast<uint32_t>(p.seed), k1 = static_cast<uint32_t>(p.seed >> 32);
    for (int r = 0; r < 10; ++r) {
        p.rk0[r] = k0;
        p.rk1[r] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

struct Shape {
    int consumer_warps;   // 4, 8 or 16
    int stages;           // 1..8
    int ctas_per_sm;      // 1..4
    int stage_bytes;      // multiple of 128, >= the largest tile
    int dynamic_tiles;    // 1: atomic counter, 2: static round robin
    int hist_copies;      // 12-bit histogram copies
    int groups;           // consumer groups per CTA (1 or 2)
    int warp_split;       // 2: the split-warp form (kModeWarpSplit) where it runs; 0 or 1: joint
};

// The mode a persistent launch of this shape runs: mode | kModeWarpSplit when the shape asks for
// the split-warp form and the mode and shape allow it.
inline bool warp_split_runs(int bits, int mode, const Shape &s) {
    const int base = mode & ~kModeFlaggedOnly;  // the write-flagged form splits too
    return bits == 8 && base >= 0 && base <= 2 && s.consumer_warps == 8 && s.groups == 1;
}
inline int shape_mode(int bits, int mode, const Shape &s) {
    return s.warp_split == 2 && warp_split_runs(bits, mode, s) ? (mode | kModeWarpSplit) : mode;
}

// Whether a call of a plan that took the split-warp form unasked runs the joint form instead: tiles that
// are not 16-byte aligned are loaded byte by byte by the consumers and stored so, by half the threads
// in the split form. 60 streams of 2^22 samples, zero, 16384-sample windows: unaligned 1306 us a call
// joint, 2002 split, aligned 118 and 112; 65536-sample windows 3427, 5766, 123 and 116. So it pays
// from about a hundredth of the samples on.
inline bool joint_for_unaligned(uint64_t unaligned, uint64_t total) { return 128 * unaligned > total; }

// Bytes of dynamic shared memory the kernels need.
size_t persistent_smem_bytes(int bits, int mode, const Shape &s);
size_t stream_smem_bytes(int bits, int mode, int consumer_warps, int ncopies, int window_bytes);

// Maximum resident CTAs per SM of the persistent kernel for this shape (0 if it cannot run).
int persistent_occupancy(int bits, int mode, const Shape &s);

// 12-bit histogram copies where nothing asks for a number: more copies spread a warp's same-bin
// atomics, but take 16 KiB each from the CTAs and are folded every window (60 streams of 2^22 samples, sigma
// 120, 8192-sample windows, 1 and 2 copies: noise 358 us a call with 3 CTAs per SM, 488 with 2, zero 275 and
// 376; 65536-sample windows, one CTA either way: 318 and 329). Narrow data, whose atomics meet in a few
// bins, does not pay for them either (sigma 0.7, zero: 218 and 320; 32768-sample windows, one CTA: 234 and 257).
constexpr int kDefaultHistCopies = 1;

// Persistent batched kernel over a device work list. counter: one zeroed uint32 (dynamic tiles).
cudaError_t launch_persistent(int bits, int mode, const Shape &s, int grid, const Seg *segs,
                              const Tile *tiles, int ntiles, const Params &p, unsigned *counter,
                              int inject_timeout, cudaStream_t st);

// Plain kernel: one CTA per window of one segment (windows [w_begin, w_begin + nw)).
cudaError_t launch_stream(int bits, int mode, int consumer_warps, const Seg &seg, int64_t w_begin,
                          int64_t nw, const Params &p, cudaStream_t st);

// Median of MAD (Eq. 3): windows [a, b) of the stream whose window 0 is entry `base` of the
// per-window MAD and MoM arrays. Mm[base + j] = lower median of D[base + max(0, j-kmom+1) .. j].
constexpr int kMomChunk = 128;
struct MomChunk {
    int64_t base;
    int32_t a, b;
};
cudaError_t launch_mom(int bits, const MomChunk *chunks, int nchunks, const int32_t *D, int32_t *Mm, int kmom,
                       cudaStream_t st);

// Digital noise as a second pass over segments whose excision pass wrote 0 at the flagged
// samples, the flag mask, every window's count and every window's M and D (segments of fewer
// than 2^31 samples). The pass's units are `unit` words of a segment's mask (nwin * ceil(W / 32)
// words), unit = 32, 64, 128 or 256; segment s holds units [fwin[s], fwin[s + 1]), nunits =
// fwin[nseg]. counter: one zeroed uint32, the cursor that the warps take units from.
constexpr int kFillUnitMin = 32, kFillUnitMax = 256;
constexpr int kFillWarps = 8;  // warps per CTA
int noise_fill_grid(int sm_count);
cudaError_t launch_noise_fill(int bits, const Seg *segs, int nseg, const uint32_t *fwin, uint32_t nunits, int unit,
                              const Params &p, unsigned *counter, int grid, cudaStream_t st);

// Write n (<= kSegBatch) segment descriptors to dst (device) from kernel parameters.
constexpr int kSegBatch = 32;
cudaError_t launch_write_segs(Seg *dst, const Seg *src_host, int n, cudaStream_t st);

}  // namespace rfi
