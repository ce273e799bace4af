// FP64 instantiations of the 2D apex tent kernel.
#include "mtp_apex2.cuh"
#include "mtp_launch.cuh"

namespace mtp {
namespace {

using Real = double;

template <int P>
cudaError_t prepare_layer(int, size_t* smem_bytes) {
    *smem_bytes = Apex2<Real, P>::BYTES;
    return cudaFuncSetAttribute(apex2_layer_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem_bytes);
}
template <int P>
cudaError_t launch_layer(const KArgs& a, int64_t t0, int n_tents, int n_rhs, cudaStream_t st) {
    apex2_layer_kernel<Real, P><<<dim3(n_tents, n_rhs), Apex2<Real, P>::NT, Apex2<Real, P>::BYTES, st>>>(a, t0);
    return cudaGetLastError();
}
template <int P>
cudaError_t prepare_persistent(int, int* blocks_per_sm) {
    constexpr size_t bytes = Apex2<Real, P>::BYTES;
    cudaError_t e = cudaFuncSetAttribute(apex2_persistent_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex2_persistent_kernel<Real, P>,
                                                         Apex2<Real, P>::NT, bytes);
}
template <int P>
cudaError_t launch_persistent(const KArgs& a, const PArgs& pa, int grid, cudaStream_t st) {
    apex2_persistent_kernel<Real, P><<<grid, Apex2<Real, P>::NT, Apex2<Real, P>::BYTES, st>>>(a, pa);
    return cudaGetLastError();
}
template <int P>
KernelEntry entry() {
    return {launch_layer<P>, prepare_layer<P>, launch_persistent<P>, prepare_persistent<P>};
}

cudaError_t prepare_batch(size_t smem, int* blocks_per_sm) {
    cudaError_t e = cudaFuncSetAttribute(apex2_batch_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex2_batch_kernel<Real>, 256, smem);
}
cudaError_t launch_batch(const BatchArgs& b, int grid, size_t smem, cudaStream_t st) {
    apex2_batch_kernel<Real><<<grid, 256, smem, st>>>(b);
    return cudaGetLastError();
}
size_t batch_smem(int p, int) {
    return p == 1 ? Apex2<Real, 1>::BYTES : p == 2 ? Apex2<Real, 2>::BYTES : p == 3 ? Apex2<Real, 3>::BYTES
         : p == 4 ? Apex2<Real, 4>::BYTES : Apex2<Real, 5>::BYTES;
}

}  // namespace

KernelEntry apex2_entry_f64(int p) {
    return p == 1 ? entry<1>() : p == 2 ? entry<2>() : p == 3 ? entry<3>() : p == 4 ? entry<4>() : entry<5>();
}
BatchEntry apex2_batch_f64() { return {launch_batch, prepare_batch, batch_smem}; }

}  // namespace mtp
