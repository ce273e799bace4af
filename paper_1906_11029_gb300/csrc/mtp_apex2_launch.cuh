// Launch wrappers of the 2D apex tent kernel, instantiated per precision in mtp_ka2d32.cu / mtp_ka2d64.cu.
#pragma once

#include "mtp_apex2.cuh"
#include "mtp_launch.cuh"

namespace mtp {

template <typename Real, int P>
cudaError_t prepare_apex2_layer(int, size_t* smem_bytes) {
    *smem_bytes = Apex2<Real, P>::BYTES;
    return cudaFuncSetAttribute(apex2_layer_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem_bytes);
}
template <typename Real, int P>
cudaError_t launch_apex2_layer(const KArgs& a, int64_t t0, int n_tents, int n_rhs, cudaStream_t st) {
    apex2_layer_kernel<Real, P><<<dim3(n_tents, n_rhs), Apex2<Real, P>::NT, Apex2<Real, P>::BYTES, st>>>(a, t0);
    return cudaGetLastError();
}
template <typename Real, int P>
cudaError_t prepare_apex2_persistent(int, int* blocks_per_sm) {
    constexpr size_t bytes = Apex2<Real, P>::BYTES;
    cudaError_t e = cudaFuncSetAttribute(apex2_persistent_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex2_persistent_kernel<Real, P>,
                                                         Apex2<Real, P>::NT, bytes);
}
template <typename Real, int P>
cudaError_t launch_apex2_persistent(const KArgs& a, const PArgs& pa, int grid, cudaStream_t st) {
    apex2_persistent_kernel<Real, P><<<grid, Apex2<Real, P>::NT, Apex2<Real, P>::BYTES, st>>>(a, pa);
    return cudaGetLastError();
}
template <typename Real, int P>
KernelEntry apex2_entry() {
    return {launch_apex2_layer<Real, P>, prepare_apex2_layer<Real, P>, launch_apex2_persistent<Real, P>, prepare_apex2_persistent<Real, P>};
}

template <typename Real>
cudaError_t prepare_apex2_batch(size_t smem, int* blocks_per_sm) {
    cudaError_t e = cudaFuncSetAttribute(apex2_batch_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex2_batch_kernel<Real>, 256, smem);
}
template <typename Real>
cudaError_t launch_apex2_batch(const BatchArgs& b, int grid, size_t smem, cudaStream_t st) {
    apex2_batch_kernel<Real><<<grid, 256, smem, st>>>(b);
    return cudaGetLastError();
}
template <typename Real>
size_t apex2_batch_smem(int p, int) {
    return p == 1 ? Apex2<Real, 1>::BYTES : p == 2 ? Apex2<Real, 2>::BYTES : p == 3 ? Apex2<Real, 3>::BYTES
         : p == 4 ? Apex2<Real, 4>::BYTES : Apex2<Real, 5>::BYTES;
}

template <typename Real>
KernelEntry apex2_entry_of(int p) {
    return p == 1 ? apex2_entry<Real, 1>() : p == 2 ? apex2_entry<Real, 2>() : p == 3 ? apex2_entry<Real, 3>()
         : p == 4 ? apex2_entry<Real, 4>() : apex2_entry<Real, 5>();
}
template <typename Real>
BatchEntry apex2_batch_of() { return {launch_apex2_batch<Real>, prepare_apex2_batch<Real>, apex2_batch_smem<Real>}; }

}  // namespace mtp
