// FP64 instantiations of the general tent kernels: 3D p = 5, and stretched meshes at every degree.
#include "mtp_launch.cuh"
namespace mtp {
MTP_KERNEL_TABLE(kernel_table_f64, double, 0)
}
