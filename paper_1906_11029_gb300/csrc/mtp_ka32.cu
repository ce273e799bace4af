// FP32 instantiations of the apex tent kernel.
#include "mtp_apex_launch.cuh"
namespace mtp {
KernelEntry apex_entry_f32(int p) {
    return p == 1 ? apex_entry<float, 1>() : p == 2 ? apex_entry<float, 2>() : p == 3 ? apex_entry<float, 3>() : apex_entry<float, 4>();
}
}  // namespace mtp
