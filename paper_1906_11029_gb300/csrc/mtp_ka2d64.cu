// FP64 instantiations of the 2D apex tent kernel.
#include "mtp_apex2_launch.cuh"
namespace mtp {
KernelEntry apex2_entry_f64(int p) { return apex2_entry_of<double>(p); }
BatchEntry apex2_batch_f64() { return apex2_batch_of<double>(); }
}  // namespace mtp
