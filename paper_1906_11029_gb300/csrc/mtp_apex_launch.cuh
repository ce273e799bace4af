// Launch wrappers of the apex tent kernel, instantiated per precision in mtp_ka32.cu / mtp_ka64.cu.
#pragma once

#include "mtp_apex.cuh"
#include "mtp_launch.cuh"

namespace mtp {

template <typename Real, int P>
cudaError_t prepare_apex_layer(int, size_t* smem_bytes) {
    *smem_bytes = ApexShape<Real, P>::BYTES;
    if (!smem_fits(*smem_bytes)) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(apex_layer_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem_bytes);
}
template <typename Real, int P>
cudaError_t launch_apex_layer(const KArgs& a, int64_t t0, int n_tents, int n_rhs, cudaStream_t st) {
    apex_layer_kernel<Real, P><<<dim3(n_tents, n_rhs), ApexShape<Real, P>::NT, ApexShape<Real, P>::BYTES, st>>>(a, t0);
    return cudaGetLastError();
}
template <typename Real, int P>
cudaError_t prepare_apex_persistent(int, int* blocks_per_sm) {
    constexpr size_t bytes = ApexShape<Real, P>::BYTES;
    if (!smem_fits(bytes)) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(apex_persistent_kernel<Real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex_persistent_kernel<Real, P>,
                                                         ApexShape<Real, P>::NT, bytes);
}
template <typename Real, int P>
cudaError_t launch_apex_persistent(const KArgs& a, const PArgs& pa, int grid, cudaStream_t st) {
    apex_persistent_kernel<Real, P><<<grid, ApexShape<Real, P>::NT, ApexShape<Real, P>::BYTES, st>>>(a, pa);
    return cudaGetLastError();
}

template <typename Real, int P>
KernelEntry apex_entry() {
    return {launch_apex_layer<Real, P>, prepare_apex_layer<Real, P>, launch_apex_persistent<Real, P>,
            prepare_apex_persistent<Real, P>};
}

template <typename Real, int PM>
cudaError_t prepare_apex_batch(size_t smem, int* blocks_per_sm) {
    if (!smem_fits(smem)) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(apex_batch_kernel<Real, PM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, apex_batch_kernel<Real, PM>, 192, smem);
}
template <typename Real, int PM>
cudaError_t launch_apex_batch(const BatchArgs& b, int grid, size_t smem, cudaStream_t st) {
    apex_batch_kernel<Real, PM><<<grid, 192, smem, st>>>(b);
    return cudaGetLastError();
}
template <typename Real>
size_t apex_batch_smem(int p, int) {
    return p == 1 ? ApexShape<Real, 1>::BYTES : p == 2 ? ApexShape<Real, 2>::BYTES : p == 3 ? ApexShape<Real, 3>::BYTES : ApexShape<Real, 4>::BYTES;
}
template <typename Real, int PM>
BatchEntry apex_batch() {
    return {launch_apex_batch<Real, PM>, prepare_apex_batch<Real, PM>, apex_batch_smem<Real>};
}

}  // namespace mtp
