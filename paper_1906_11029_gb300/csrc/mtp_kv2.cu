// Shape variant 2 of the general FP32 tent kernel: one patch element and one basis function (or facet
// mode) per item, 512 threads per CTA in 3D, for the shortest tents on layers that hold fewer tents
// than the GPU has CTA slots; the degree argument carries the variant as p + 32.  Where the apex tent
// kernels run the variant selects them (see mtp_kv.cu).
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f32_v2(KernelEntry e[2][5]) {
    for (int p = 1; p <= 5; ++p) e[0][p - 1] = apex2_entry_f32(p);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f32(p);
    e[1][4] = MTP_KERNEL_ENTRY(float, 3, 37, 0);
}
}  // namespace mtp
