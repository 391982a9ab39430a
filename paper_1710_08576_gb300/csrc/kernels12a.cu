// 12-bit instantiations of the any-window form of the persistent kernel (plain excision, the
// estimation and the apply passes of the Median of MAD), one consumer group of 8 warps.
#include "kernels_impl.cuh"

namespace rfi {

static_assert(kModeAny == 2048 && kModeStats == 4 && kModeApply == 8, "mode numbers of the cases below");

#define RFI_DISPATCH_ANY(FN, MODE, CW, G, ...)                                                        \
    do {                                                                                              \
        switch (MODE * 1000 + CW * 10 + G) {                                                          \
            RFI_CASE_MCG(12, FN, 2048, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2049, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2050, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2051, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2052, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2056, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2057, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2058, 8, 1, __VA_ARGS__)                                             \
            RFI_CASE_MCG(12, FN, 2059, 8, 1, __VA_ARGS__)                                             \
            default: break;                                                                           \
        }                                                                                             \
    } while (0)

cudaError_t launch_persistent_any_b12(int mode, const Shape &s, int grid, const Seg *segs, const Tile *tiles,
                                     int ntiles, const Params &p, unsigned *counter, int inject, cudaStream_t st) {
    RFI_DISPATCH_ANY(dev::persistent_launch_t, mode, s.consumer_warps, s.groups, s, grid, segs, tiles, ntiles, p,
                     counter, inject, st);
    return cudaErrorInvalidValue;
}

int persistent_occupancy_any_b12(int mode, const Shape &s) {
    RFI_DISPATCH_ANY(dev::persistent_occ_t, mode, s.consumer_warps, s.groups, s);
    return 0;
}

}  // namespace rfi
