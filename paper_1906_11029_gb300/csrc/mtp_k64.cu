// FP64 kernel table: the apex tent kernels, and the general one in 3D beyond their degrees.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_f64(KernelEntry e[2][5]) {
    for (int p = 1; p <= 5; ++p) e[0][p - 1] = apex2_entry_f64(p);
    for (int p = 1; p <= 4; ++p) e[1][p - 1] = apex_entry_f64(p);
    e[1][4] = MTP_KERNEL_ENTRY(double, 3, 5, 0);
}
}  // namespace mtp
