// FP64 instantiations of the apex tent kernel.
#include "mtp_apex_launch.cuh"
namespace mtp {
KernelEntry apex_entry_f64(int p) {
    return p == 1 ? apex_entry<double, 1>() : p == 2 ? apex_entry<double, 2>() : p == 3 ? apex_entry<double, 3>() : apex_entry<double, 4>();
}
}  // namespace mtp
