// FP64 instantiations of the many-instance apex kernel, by the largest degree of the batch.
#include "mtp_apex_launch.cuh"
namespace mtp {
BatchEntry apex_batch_f64(int pmax) {
    return pmax <= 2 ? apex_batch<double, 2>() : pmax == 3 ? apex_batch<double, 3>() : apex_batch<double, 4>();
}
}  // namespace mtp
