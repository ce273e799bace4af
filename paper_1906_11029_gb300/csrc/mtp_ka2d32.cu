// FP32 instantiations of the 2D apex tent kernel.
#include "mtp_apex2_launch.cuh"
namespace mtp {
KernelEntry apex2_entry_f32(int p) { return apex2_entry_of<float>(p); }
BatchEntry apex2_batch_f32() { return apex2_batch_of<float>(); }
}  // namespace mtp
