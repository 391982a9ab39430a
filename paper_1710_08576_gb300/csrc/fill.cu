// Digital noise as a second pass (Eq. 2's noise replacement, value as in NoiseScale).
//
// The excision pass of a noise plan created with RFI_PLAN_NOISE_PASS runs as a zero-replacement
// pass: it writes 0 at every flagged sample, the flag mask and every window's M and D. This
// kernel then overwrites the flagged samples with M + the Philox noise of spread 1.4826·D, keyed
// by the absolute sample index as always, so the result is the same bits as the one-pass form.
//
// Work: a segment's mask is one array of words, window k's at k * mw (mw = ceil(W / 32)), cut into
// units of up to 256 words regardless of the windows; segment s holds units [fwin[s], fwin[s + 1]).
// The warps take units in order from a cursor, so that at any time they read masks and write
// samples close to one another (giving each warp a run of consecutive units instead made the
// k = 3 call of the 60-stream benchmark 40 % slower) and a warp that met dense units takes fewer. Per unit:
//  1. the lanes load the words (lane l words l, l + 32, ...) and list the nonzero ones,
//  2. per group of 32 nonzero words, lane l takes one: its window (M, D, first sample) and, by a
//     prefix sum of the flag counts, where its flags go in the warp's position list,
//  3. the group's words are expanded one by one: lane j tests bit j and a popcount of the bits
//     below gives its place; an entry is 16 bits, the word's slot in its group and the bit,
//  4. every lane takes an entry of the list and evaluates its noise, 32 at a time. The fewer than
//     32 entries left over go in front of the next group's, so only the last batch of a unit is
//     not full. Two entries of a lane at a time: their Philox chains interleave.
// What bounds it: the Philox products. A 32 x 32 -> 64-bit product takes four cycles of a quarter of
// an SM's multiplier for a warp (measured), so the 18 of a batch of 32 samples and the other multiply
// instructions come to about 90 cycles; step 3 costs 8 instructions per nonzero word (no vote, branch or
// carried counter per word) and steps 1 and 2 about 400 per unit. On 60 streams of 2^26 int8 samples in
// 16384-sample windows (k = 3, 6.3 % flagged) the pass takes 1.13 ms; 1.70 ms with a ring filled
// word by word under a ballot, a static share of the units and 20 products a value. Measured and not
// kept: the next unit's words loaded while one is worked on (56 registers, 1.5 % slower), the
// left-over samples kept in registers across units (57 registers, 1.7 % slower), a sixth CTA per
// SM (40 registers, 1 % slower).

#include "core.cuh"

namespace rfi {
namespace dev {

constexpr int kFillThreads = kFillWarps * 32;
constexpr int kFillWords = kFillUnitMax / 32;  // mask words per lane of the largest unit

// One warp's work area.
struct FillWarp {
    uint2 word[kFillUnitMax];    // the unit's nonzero words and their indices, in order
    uint2 ent[64];               // two groups of 32 words: {word, place of its flags in the list}
    uint4 win[64];               // of the same words: {first sample, sig2 and moff of its window (NoiseScale), -}
    uint16_t list[32 + 32 * 32]; // flagged samples waiting: slot in ent * 32 + bit
};

template <int BITS>
__device__ __forceinline__ void fill_store(uint8_t *out, uint32_t pos, int32_t z) {
    if (BITS == 8) out[pos] = static_cast<uint8_t>(z);
    else reinterpret_cast<int16_t *>(out)[pos] = static_cast<int16_t>(z);
}

// Segments hold fewer than 2^31 samples (the plan routes longer ones through the one-pass form),
// so every segment-relative index below fits 32 bits.
template <int BITS>
__global__ void __launch_bounds__(kFillThreads) noise_fill_kernel(const Seg *__restrict__ segs, int nseg,
                                                                 const uint32_t *__restrict__ fwin, uint32_t nunits,
                                                                 uint32_t unit, Params p, unsigned *counter) {
    __shared__ FillWarp area[kFillWarps];
    FillWarp &a = area[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t below = (1u << lane) - 1u, bit = 1u << lane;
    const KeysPre key{p};
    int s = 0;
    // the first unit of a warp is its own (spread over the CTAs, so that few units take many SMs),
    // the others come from the cursor, fetched while the unit before is worked on. Where every unit
    // has a warp of its own nobody asks the cursor: thousands of additions to one word at once took 2 us
    // (2^22 int8 samples, few flagged: 16.7 us a call with them, 14.5 without)
    const uint32_t nwarps = gridDim.x * kFillWarps;
    uint32_t u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (; u < nunits;) {
        uint32_t next = nunits;
        if (nunits > nwarps && lane == 0) next = nwarps + atomicAdd(counter, 1u);
        while (s + 1 < nseg && fwin[s + 1] <= u) ++s;  // a warp's units ascend
        const Seg &g = segs[s];
        const uint32_t W = static_cast<uint32_t>(g.W), mw = static_cast<uint32_t>(g.mask_words);
        const uint32_t jfirst = (u - fwin[s]) * unit;
        const uint32_t jend = min(jfirst + unit, g.nwords), j0 = jfirst + lane;
        const uint32_t *mk = g.mask;
        uint32_t m[kFillWords];
#pragma unroll
        for (int i = 0; i < kFillWords; ++i) m[i] = j0 + 32 * i < jend ? mk[j0 + 32 * i] : 0u;
        uint32_t n = 0;  // nonzero words
#pragma unroll
        for (int i = 0; i < kFillWords; ++i) {
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, m[i] != 0u);
            if (m[i]) a.word[n + __popc(bal & below)] = make_uint2(m[i], j0 + 32 * i);
            n += static_cast<uint32_t>(__popc(bal));
        }
        if (n == 0u) {
            u = __shfl_sync(0xFFFFFFFFu, next, 0);
            continue;
        }
        __syncwarp();
        const int lg = (mw & (mw - 1u)) == 0u ? __ffs(static_cast<int>(mw)) - 1 : -1;  // log2 mw, or -1
        const NoiseRun<BITS, KeysPre> run(key, g.stream_id, static_cast<uint64_t>(g.abs0), static_cast<uint64_t>(g.len));
        uint8_t *const out = g.out;
        auto emit = [&](uint32_t code) {
            const uint4 e = a.win[code >> 5];
            const uint32_t pos = e.x + (code & 31u);
            const int32_t sig2 = static_cast<int32_t>(e.y), moff = static_cast<int32_t>(e.z);
            fill_store<BITS>(out, pos, run.one_hi ? run.value(pos, sig2, moff) : run.value_any(pos, sig2, moff));
        };
        // two entries of a lane at a time: their Philox chains are independent and interleave
        auto emit2 = [&](uint32_t c0, uint32_t c1) {
            if (!run.one_hi) {
                emit(c0);
                emit(c1);
                return;
            }
            const uint4 e0 = a.win[c0 >> 5], e1 = a.win[c1 >> 5];
            const uint32_t p0 = e0.x + (c0 & 31u), p1 = e1.x + (c1 & 31u);
            const uint32_t s0 = run.sum(p0), s1 = run.sum(p1);
            fill_store<BITS>(out, p0, NoiseScale<BITS>::value(s0, static_cast<int32_t>(e0.y), static_cast<int32_t>(e0.z)));
            fill_store<BITS>(out, p1, NoiseScale<BITS>::value(s1, static_cast<int32_t>(e1.y), static_cast<int32_t>(e1.z)));
        };
        uint32_t have = 0;  // entries waiting at the front of the list
        for (uint32_t e0 = 0, grp = 0; e0 < n; e0 += 32, grp ^= 32u) {
            const uint32_t ne = min(32u, n - e0);
            uint32_t w = 0u, cnt = 0u;
            if (lane < ne) {
                const uint2 wj = a.word[e0 + lane];
                w = wj.x;
                cnt = static_cast<uint32_t>(__popc(w));
                const uint32_t k = lg >= 0 ? wj.y >> lg : wj.y / mw;
                a.win[grp + lane] = make_uint4(k * W + ((wj.y - k * mw) << 5),
                                               static_cast<uint32_t>(NoiseScale<BITS>::kSig2 * g.mad[k]),
                                               static_cast<uint32_t>(g.med[k] - NoiseScale<BITS>::kOff), 0u);
            }
            uint32_t inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= static_cast<uint32_t>(o)) inc += y;
            }
            a.ent[grp + lane] = make_uint2(w, have + inc - cnt);
            const uint32_t total = have + __shfl_sync(0xFFFFFFFFu, inc, 31);
            __syncwarp();
            // a full group (the other lanes' words are zero) in steps of four words
            uint32_t code = grp * 32u + lane;
            for (uint32_t e = 0; e < ne; e += 4) {
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint2 wo = a.ent[grp + e + q];
                    if (wo.x & bit) a.list[wo.y + __popc(wo.x & below)] = static_cast<uint16_t>(code + 32u * q);
                }
                code += 128u;
            }
            __syncwarp();
            uint32_t h = 0;
            for (; h + 64u <= total; h += 64u) emit2(a.list[h + lane], a.list[h + 32u + lane]);
            if (h + 32u <= total) {
                emit(a.list[h + lane]);
                h += 32u;
            }
            have = total - h;
            const uint32_t left = lane < have ? a.list[h + lane] : 0u;
            __syncwarp();
            if (e0 + 32 < n) {
                // a full group fills at least one batch, so what is left over is this group's: the
                // next one may take the other half of ent
                if (lane < have) a.list[lane] = static_cast<uint16_t>(left);
            } else if (lane < have) {
                emit(left);
            }
            __syncwarp();
        }
        u = __shfl_sync(0xFFFFFFFFu, next, 0);
    }
}

}  // namespace dev

int noise_fill_grid(int sm_count) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dev::noise_fill_kernel<8>, dev::kFillThreads, 0) != cudaSuccess ||
        n < 1) {
        cudaGetLastError();
        n = 1;
    }
    return sm_count * n;
}

cudaError_t launch_noise_fill(int bits, const Seg *segs, int nseg, const uint32_t *fwin, uint32_t nunits, int unit,
                              const Params &p, unsigned *counter, int grid, cudaStream_t st) {
    if (nunits == 0) return cudaSuccess;
    if (nunits < static_cast<uint32_t>(grid)) grid = static_cast<int>(nunits);
    if (bits == 8) dev::noise_fill_kernel<8><<<grid, dev::kFillThreads, 0, st>>>(segs, nseg, fwin, nunits, static_cast<uint32_t>(unit), p, counter);
    else dev::noise_fill_kernel<12><<<grid, dev::kFillThreads, 0, st>>>(segs, nseg, fwin, nunits, static_cast<uint32_t>(unit), p, counter);
    return cudaGetLastError();
}

}  // namespace rfi
