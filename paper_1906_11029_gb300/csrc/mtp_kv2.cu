// FP32 instantiations of the general tent kernel in shape variant 2: one patch element and one
// basis function (or facet mode) per item, 512 threads per CTA in 3D, for the shortest tents on
// layers that hold fewer tents than the GPU has CTA slots; the degree argument carries the variant
// as p + 32.  In 3D up to kApexMaxDegree the variant selects the apex tent kernel (see mtp_kv.cu).
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f32_v2(KernelEntry e[2][5]) {
    e[0][0] = MTP_KERNEL_ENTRY(float, 2, 33, 0);
    e[0][1] = MTP_KERNEL_ENTRY(float, 2, 34, 0);
    e[0][2] = MTP_KERNEL_ENTRY(float, 2, 35, 0);
    e[0][3] = MTP_KERNEL_ENTRY(float, 2, 36, 0);
    e[0][4] = MTP_KERNEL_ENTRY(float, 2, 37, 0);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f32(p);
    e[1][4] = MTP_KERNEL_ENTRY(float, 3, 37, 0);
}
}  // namespace mtp
