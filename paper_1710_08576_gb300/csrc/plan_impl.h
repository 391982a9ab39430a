// Host-side plan state shared by plan.cpp, host_pipe.cpp and autotune.cpp.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "rfi.h"
#include "internal.h"

namespace rfi {

// Buffers of the chunked host pipeline (rfi_excise_host), allocated on first use.
struct HostPipe {
    static constexpr int kSlots = 3;
    int64_t chunk_bytes = 0;     // input bytes per slot
    uint8_t *in[kSlots] = {};
    uint8_t *out[kSlots] = {};
    uint32_t *mask[kSlots] = {};
    uint32_t *counts[kSlots] = {};
    cudaEvent_t h2d[kSlots] = {}, comp[kSlots] = {}, d2h[kSlots] = {};
    cudaStream_t s_comp = nullptr, s_d2h = nullptr;
    bool ready = false;
};

}  // namespace rfi

struct rfi_plan_s {
    int bits = 8, S = 0, mode = 0;
    uint32_t flags = 0;
    double k = 0;
    int64_t kq = 0;
    int32_t cval = 0;
    uint64_t seed = 0;
    std::vector<int64_t> len;
    std::vector<int32_t> W;
    std::vector<uint32_t> sid;
    std::vector<int64_t> nwin, woff;
    uint64_t total_windows = 0, total_samples = 0, last_windows = 0;
    int device = 0, sm_count = 0;
    rfi::Shape shape{};
    bool given_stage = false;  // the caller's shape gives the stage size
    bool split_by_rule = false;  // the split-warp form was neither asked for nor tuned
    std::vector<rfi::Tile> tiles_host;
    int ntiles = 0, grid = 0;
    int grid_apply = 0;  // Median of MAD: grid of the apply pass (no histogram: more CTAs fit)
    // device workspace
    void *ws = nullptr;
    size_t ws_bytes = 0;
    rfi::DevCounters *d_ctr = nullptr;
    rfi::Seg *d_segs = nullptr;
    rfi::Tile *d_tiles = nullptr;
    int32_t *d_med = nullptr, *d_mad = nullptr;
    // Median of MAD (Eq. 3): kmom >= 2; segment table holds 2S entries (stats pass, apply pass)
    int kmom = 0;
    int32_t *d_mom = nullptr;
    // RFI_PLAN_POWER: {sum x^2, sum z^2} per window
    bool power = false;
    // some stream has windows of 2^l samples, 512 <= 2^l <= 8192: the multi-window form
    bool multi = false;
    // windows that the aligned forms serve badly: the any-window form (any_form_gain)
    bool any = false;
    // RFI_PLAN_WRITE_FLAGGED: in place, only changed chunks are stored
    bool write_flagged = false;
    uint64_t *d_pow = nullptr;
    int out_format = RFI_OUT_SAME;  // fused output format
    // digital noise as a second pass (noise_fill): the excision pass replaces with 0, then the
    // fill kernel writes the noise of every flagged sample; d_fwin: S + 1 unit offsets
    bool fill = false;
    uint32_t *d_fwin = nullptr;
    uint32_t nfwin = 0;
    int fill_grid = 0, fill_unit = 0;  // CTAs, mask words of a unit
    uint32_t *d_fmask = nullptr;  // flag masks of streams called without one (allocated on demand)
    std::vector<int64_t> fmask_off;
    // digital copy: the variants (segment table holds ncopy * S entries)
    int ncopy = 0;
    std::vector<rfi::Variant> variants;
    rfi::Variant *d_var = nullptr;
    rfi::MomChunk *d_mchunks = nullptr;
    std::vector<rfi::MomChunk> mchunks;
    std::vector<rfi::Seg> segs_host;
    bool segs_valid = false;
    int last_seg_writes = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t gexec = nullptr;
    rfi::HostPipe pipe;
    size_t host_pipe_bytes = 0;
    // a plan split by window-size class: one internal plan per class and its stream indices
    std::vector<rfi_plan_s *> parts;
    // parts after the first run on their own streams, forked from and joined back into the
    // caller's stream with events, so that one part's tail overlaps the next part's kernels
    std::vector<cudaStream_t> part_st;
    std::vector<cudaEvent_t> part_ev;  // [0]: the fork; [k]: part k's end
    std::vector<std::vector<int>> part_streams;
};

namespace rfi {

rfi_status plan_choose_shape(rfi_plan_s *P, const rfi_launch_shape *req);
// Whether the split-warp form (kModeWarpSplit) can run this plan with shape s.
bool plan_warp_split_runs(const rfi_plan_s *P, const Shape &s);
rfi_status plan_build_tiles(rfi_plan_s *P);
rfi_status plan_alloc_workspace(rfi_plan_s *P);
rfi_status plan_enqueue_batched(rfi_plan_s *P, cudaStream_t st, bool joint = false);
rfi_status plan_build_graph(rfi_plan_s *P);
rfi_status plan_autotune(rfi_plan_s *P, const rfi_launch_shape *req);
void plan_release_host_pipe(rfi_plan_s *P);
Params plan_params(const rfi_plan_s *P);
std::vector<Seg> plan_segs(const rfi_plan_s *P, const void *const *in, void *const *out, uint32_t *const *mask,
                           uint32_t *const *counts);
rfi_status plan_check_buffers(const rfi_plan_s *P, const void *const *in, void *const *out,
                              uint32_t *const *mask, uint32_t *const *counts);
rfi_status plan_run_batched(rfi_plan_s *P, const std::vector<Seg> &segs, cudaStream_t st);
inline int plan_nsegs(const rfi_plan_s *P) {
    return P->kmom >= 2 ? 2 * P->S : (P->ncopy > 0 ? P->ncopy * P->S : P->S);
}
// Whether a plan of one window size takes its tiles from the cursor and not round robin. SMs differ in
// pace, which the cursor evens out, but its round trips cost a plan of few tiles. us a call, round robin
// and cursor, int8 noise in 16384-sample windows (12-bit noise, 8192 samples; fp16 output): 5.3 tiles a CTA
// 33.2 and 33.3 (37.5 and 38.6; 32.8 and 33.1), 9.1 tiles 51.8 and 53.5 (58.5 and 59.7; 51.4 and 50.8), 12
// tiles 66.0 and 64.1 (74.2 and 74.2; 64.0 and 62.9), 16 tiles 84.7 and 82.8 (96.0 and 94.3; 81.9 and
// 79.2), 40 tiles 197 and 190 (225 and 218; 189 and 180).
inline bool many_tiles(int64_t tiles, int64_t ctas) { return tiles >= 12 * ctas; }
// Windows per tile of each stream: as many as a stage holds, fewer in a small plan, which spreads its
// windows: tiles are halved as long as all of them still run at once on `room` CTAs (2^20 int8 samples
// in 4096-sample windows: 64 tiles of four 9.6 us a call, 256 of one 8.2, with noise 12.3 and 8.8;
// 2^22 samples: 256 tiles 10.3 us, 512 on 456 CTAs 12.4). whole: a stage size that the caller gave
// stands for its tiles. The tuner times the same lists.
inline std::vector<int64_t> windows_per_tile(int bits, int mode, bool mom, bool whole, const std::vector<int64_t> &nwin,
                                             const std::vector<int32_t> &W, int stage_bytes, int64_t room) {
    std::vector<int64_t> per(W.size());
    auto set = [&](int64_t div) {  // the tiles
        int64_t n = 0;
        for (size_t i = 0; i < W.size(); ++i) {
            int64_t p = tile_windows(bits, mode, W[i], stage_bytes);
            if (mom) p = p < kApplyTileWindows ? p : kApplyTileWindows;
            per[i] = p / div > 1 ? p / div : 1;
            n += (nwin[i] + per[i] - 1) / per[i];
        }
        return n;
    };
    int64_t div = 1;
    for (int64_t n = set(1); !whole && div < 64 && n < room; div *= 2) {
        const int64_t more = set(2 * div);
        if (more == n || more > room) break;
        n = more;
    }
    set(div);
    return per;
}
// Key of a tuned shape, after the device's name: what the candidates and their times depend on. A stream
// shorter than its window counts with its length, which its stage is sized for; a shape tuned under
// the caller's constraints is kept apart from others.
inline std::string tune_key(int bits, int mode, const std::vector<int64_t> &len, const std::vector<int32_t> &W,
                            const rfi_launch_shape *req) {
    std::string k = "|" + std::to_string(bits) + "|" + std::to_string(mode) + "|" + std::to_string(len.size()) + "|";
    for (size_t i = 0; i < len.size(); ++i) {
        k += std::to_string(W[i]) + ":" + std::to_string(len[i] / W[i]);
        k += len[i] < W[i] ? "/" + std::to_string(len[i]) + "," : ",";
    }
    if (req) {
        const int32_t f[] = {req->consumer_warps, req->stages, req->ctas_per_sm, req->stage_bytes,
                             req->dynamic_tiles, bits == 12 ? req->hist_copies : 0, req->groups, req->warp_split};
        bool any = false;
        for (int32_t v : f) any = any || v != 0;
        if (any)
            for (int32_t v : f) k += "|" + std::to_string(v);
    }
    return k;
}
// Whether a shape from the cache is one that the tuner could have made for windows that need min_stage bytes.
inline bool tuned_shape_fits(const Shape &s, int min_stage) {
    return (s.consumer_warps == 4 || s.consumer_warps == 8 || s.consumer_warps == 16) && s.stages >= 1 && s.stages <= 8 &&
           s.ctas_per_sm >= 1 && s.ctas_per_sm <= 4 && s.stage_bytes >= min_stage && s.stage_bytes <= 227 * 1024 &&
           s.stage_bytes % 128 == 0 && (s.dynamic_tiles == 1 || s.dynamic_tiles == 2) &&
           (s.hist_copies == 1 || s.hist_copies == 2 || s.hist_copies == 4) && (s.groups == 1 || s.groups == 2) &&
           (s.warp_split == 1 || s.warp_split == 2);
}
// Stage class of a window of wb bytes: 0 up to 16 KiB, 1 up to 32 KiB, 2 larger.
inline int window_class(int64_t wb) { return wb <= 16384 ? 0 : (wb <= 32768 ? 1 : 2); }
// Per-part pointer arrays of a split plan (entries in the part's stream order).
template <class T>
std::vector<T> part_args(const rfi_plan_s *P, size_t k, T const *all) {
    std::vector<T> v;
    for (int i : P->part_streams[k]) v.push_back(all ? all[i] : T());
    return v;
}
// Kernel mode of a per-window MAD plan (the power-metered form when RFI_PLAN_POWER is set).
inline int plan_kernel_mode(const rfi_plan_s *P) {
    const int fmt = P->out_format == RFI_OUT_F16 ? kModeF16 : (P->out_format == RFI_OUT_BF16 ? kModeBF16 : 0);
    if (P->ncopy > 0) return kModeCopies;
    const int m = (P->fill && P->kmom < 2 ? 0 : P->mode) | (P->power ? kModePower : 0) | fmt;
    if (P->write_flagged) return m | kModeFlaggedOnly;
    if (P->any) return m | kModeAny;
    return m | (P->multi && m < 4 ? kModeMulti : 0);
}
// Kernel mode of the estimation pass of a Median-of-MAD plan.
inline int plan_stats_mode(const rfi_plan_s *P) {
    return kModeStats | (P->any ? kModeAny : (P->multi ? kModeMulti : 0));
}
// Kernel mode of the apply pass of a Median-of-MAD plan.
inline int plan_apply_mode(const rfi_plan_s *P) {
    return (kModeApply + (P->fill ? 0 : P->mode)) | (P->any ? kModeAny : 0);
}
// The mode that the plan's stages and tiles are sized for.
inline int plan_tile_mode(const rfi_plan_s *P) { return P->any ? kModeAny : 0; }

}  // namespace rfi
