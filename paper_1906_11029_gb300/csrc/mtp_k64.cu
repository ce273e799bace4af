// FP64 instantiations of the general tent kernel: 2D, and 3D beyond the apex tent kernel's degrees.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f64(KernelEntry e[2][5]) {
    e[0][0] = MTP_KERNEL_ENTRY(double, 2, 1, 0);
    e[0][1] = MTP_KERNEL_ENTRY(double, 2, 2, 0);
    e[0][2] = MTP_KERNEL_ENTRY(double, 2, 3, 0);
    e[0][3] = MTP_KERNEL_ENTRY(double, 2, 4, 0);
    e[0][4] = MTP_KERNEL_ENTRY(double, 2, 5, 0);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f64(p);
    e[1][4] = MTP_KERNEL_ENTRY(double, 3, 5, 0);
}
}  // namespace mtp
