// Shape variant 1 of the general FP32 tent kernel: one patch element per stage item (twice the items
// of the paired default at half the work each) for layers that hold fewer tents than the GPU has
// CTA slots; the degree argument carries the variant as p + 16.  Where the apex tent kernels run they
// are the faster ones for every layer width (16^3 cavity, p = 3: 92 ms per 0.25 time units against
// 214 ms for variant 2), so there the variant selects them.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f32_v1(KernelEntry e[2][5]) {
    for (int p = 1; p <= 5; ++p) e[0][p - 1] = apex2_entry_f32(p);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f32(p);
    e[1][4] = MTP_KERNEL_ENTRY(float, 3, 21, 0);
}
}  // namespace mtp
