// FP32 instantiations of the many-instance apex kernel, by the largest degree of the batch.
#include "mtp_apex_launch.cuh"
namespace mtp {
BatchEntry apex_batch_f32(int pmax) {
    return pmax <= 2 ? apex_batch<float, 2>() : pmax == 3 ? apex_batch<float, 3>() : apex_batch<float, 4>();
}
}  // namespace mtp
