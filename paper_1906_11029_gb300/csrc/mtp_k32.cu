// FP32 instantiations of the general tent kernels (geometry and the causality test in FP64): 3D p = 5, and
// stretched meshes at every degree (see kMaxStretch).
#include "mtp_launch.cuh"
namespace mtp {
MTP_KERNEL_TABLE(kernel_table_f32, float, 0)
}
