// Instantiations of the tent kernels with FP32 arithmetic, the Taylor sum of each tent carried
// as an FP32 pair hi + lo (two-sum) and the state between tents stored in FP64 (MTP_FP32_SPLIT).
// In 3D the items are those of shape variant 1, one patch element each: with the second sum in shared
// memory few CTAs fit an SM, and twice the items at half the work keep more warps of a CTA busy.  The
// results are the same bits.  25 layers of the graded 32^3 mesh (3259 tents per layer), paired items ->
// these, on a GB300: p = 1 9.5 -> 7.5 ms, p = 2 25.3 -> 18.1, p = 3 66 -> 54, p = 4 247 -> 206, p = 5 883 -> 775;
// 60 layers of 16^3 cubes (143 per layer): 2.2 -> 1.7, 5.7 -> 3.8, 13.3 -> 10.0, 32 -> 27, 116 -> 105.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_split(KernelEntry e[2][5]) {
    e[0][0] = MTP_KERNEL_ENTRY(float, 2, 1, 3);
    e[0][1] = MTP_KERNEL_ENTRY(float, 2, 2, 3);
    e[0][2] = MTP_KERNEL_ENTRY(float, 2, 3, 3);
    e[0][3] = MTP_KERNEL_ENTRY(float, 2, 4, 3);
    e[0][4] = MTP_KERNEL_ENTRY(float, 2, 5, 3);
    e[1][0] = MTP_KERNEL_ENTRY(float, 3, 17, 3);
    e[1][1] = MTP_KERNEL_ENTRY(float, 3, 18, 3);
    e[1][2] = MTP_KERNEL_ENTRY(float, 3, 19, 3);
    e[1][3] = MTP_KERNEL_ENTRY(float, 3, 20, 3);
    e[1][4] = MTP_KERNEL_ENTRY(float, 3, 21, 3);
}
}  // namespace mtp
