// FP32 instantiations of the general tent kernel in shape variant 1: one patch element per stage
// item (twice the items of the paired default at half the work each) for layers that hold fewer
// tents than the GPU has CTA slots; the degree argument carries the variant as p + 16.  In 3D up
// to kApexMaxDegree the apex tent kernel is the faster one for every layer width (16^3 cavity,
// p = 3: 92 ms per 0.25 time units against 214 ms for variant 2), so the variant selects it.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f32_v1(KernelEntry e[2][5]) {
    e[0][0] = MTP_KERNEL_ENTRY(float, 2, 17, 0);
    e[0][1] = MTP_KERNEL_ENTRY(float, 2, 18, 0);
    e[0][2] = MTP_KERNEL_ENTRY(float, 2, 19, 0);
    e[0][3] = MTP_KERNEL_ENTRY(float, 2, 20, 0);
    e[0][4] = MTP_KERNEL_ENTRY(float, 2, 21, 0);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f32(p);
    e[1][4] = MTP_KERNEL_ENTRY(float, 3, 21, 0);
}
}  // namespace mtp
