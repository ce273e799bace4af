// Split precision (mtp_ks.cu) in 3D, p = 1..3, with the items of shape variant 2: one patch element and
// one basis function (or facet mode), 512 threads per CTA; for layers of at most a tent per SM.
#include "mtp_launch.cuh"
namespace mtp {
void kernel_table_split_narrow(KernelEntry e[3]) {
    e[0] = MTP_KERNEL_ENTRY(float, 3, 33, 3);
    e[1] = MTP_KERNEL_ENTRY(float, 3, 34, 3);
    e[2] = MTP_KERNEL_ENTRY(float, 3, 35, 3);
}
}  // namespace mtp
