// Lattice exchange and energy (see include/mtp.h): y(x_k) = (1/sqrt|det J|) sum_a V[k][a] Y_a, its
// inverse, and 1/2 sum (|Y_E|^2 / eps + |Y_H|^2 / mu) of a flat front.
//
// A CTA takes 32 elements: warp = field, lane = element.  The element blocks are copied through
// shared memory (rows of odd length), so global accesses are contiguous in both layouts, and a
// thread holds its field's coefficients in registers and runs the straight-line products of
// LatticeOps.  The products are FP64 and bound these kernels (1.7 FP64 multiply-adds a clock and
// SM).  Measured on a GB300 for 196 608 elements of degree 4 in FP32 (826 MB in and out, 0.12 ms of
// HBM): lattice to state, energy and state to lattice take 3.5 ms together; a thread per
// coefficient with strided reads, dense products and a division each took 9.5 ms.
#include <string>

#include <cuda_runtime.h>

#include "mtp_device.h"
#include "mtp_internal.h"
#include "mtp_lattice_ops.h"

namespace mtp {

namespace {

constexpr int kLatElems = 32;

template <int DIM, int P>
struct LatShape {
    static constexpr int NF = DIM == 2 ? 3 : 6;
    static constexpr int NB = DIM == 2 ? (P + 1) * (P + 2) / 2 : (P + 1) * (P + 2) * (P + 3) / 6;
    static constexpr int NC = NF * NB, SP = NC | 1, NT = 32 * NF;
};

template <typename Real, int DIM, int P>
__global__ void __launch_bounds__(LatShape<DIM, P>::NT) to_lattice_kernel(const Real* state, double* vals, const double* geo,
                                                                          int64_t ne, int64_t n) {
    using Sh = LatShape<DIM, P>;
    constexpr int NF = Sh::NF, NB = Sh::NB, NC = Sh::NC, SP = Sh::SP, NT = Sh::NT;
    extern __shared__ __align__(16) unsigned char smem[];
    double* out = (double*)smem;
    Real* in = (Real*)smem;
    const int lane = threadIdx.x & 31, f = threadIdx.x >> 5;
    for (int64_t e0 = (int64_t)blockIdx.x * kLatElems; e0 < n; e0 += (int64_t)gridDim.x * kLatElems) {
        const int ns = (int)(n - e0 < kLatElems ? n - e0 : kLatElems);
        const Real* src = state + e0 * NC;
        for (int i = threadIdx.x; i < ns * NC; i += NT) in[i / NC * SP + i % NC] = src[i];
        __syncthreads();
        const int k = lane < ns ? lane : ns - 1;
        double x[NB];
#pragma unroll
        for (int a = 0; a < NB; ++a) x[a] = (double)in[k * SP + f * NB + a];
        const double is = geo[(e0 + k) % ne * kGeoStride + 28];
        __syncthreads();
        LatticeOps<DIM, P>::to(x, [&](int p, double v) { out[lane * SP + p * NF + f] = is * v; });
        __syncthreads();
        double* dst = vals + e0 * NC;
        for (int i = threadIdx.x; i < ns * NC; i += NT) dst[i] = out[i / NC * SP + i % NC];
        __syncthreads();
    }
}

template <typename Real, int DIM, int P>
__global__ void __launch_bounds__(LatShape<DIM, P>::NT) from_lattice_kernel(const double* vals, Real* state, const double* geo,
                                                                            int64_t ne, int64_t n) {
    using Sh = LatShape<DIM, P>;
    constexpr int NF = Sh::NF, NB = Sh::NB, NC = Sh::NC, SP = Sh::SP, NT = Sh::NT;
    extern __shared__ __align__(16) unsigned char smem[];
    double* in = (double*)smem;
    Real* out = (Real*)smem;
    const int lane = threadIdx.x & 31, f = threadIdx.x >> 5;
    for (int64_t e0 = (int64_t)blockIdx.x * kLatElems; e0 < n; e0 += (int64_t)gridDim.x * kLatElems) {
        const int ns = (int)(n - e0 < kLatElems ? n - e0 : kLatElems);
        const double* src = vals + e0 * NC;
        for (int i = threadIdx.x; i < ns * NC; i += NT) in[i / NC * SP + i % NC] = src[i];
        __syncthreads();
        const int k = lane < ns ? lane : ns - 1;
        double v[NB];
#pragma unroll
        for (int p = 0; p < NB; ++p) v[p] = in[k * SP + p * NF + f];
        const double sq = 1.0 / geo[(e0 + k) % ne * kGeoStride + 28];
        __syncthreads();
        auto put = [&](int a, double y) { out[lane * SP + f * NB + a] = (Real)(sq * y); };
        LatticeOps<DIM, P>::from(v, put);
        __syncthreads();
        Real* dst = state + e0 * NC;
        for (int i = threadIdx.x; i < ns * NC; i += NT) dst[i] = out[i / NC * SP + i % NC];
        __syncthreads();
    }
}

// Few elements: a thread per value with the dense products, in the order of the points or functions, which
// spreads them over all SMs.  The kernels above take as long for one CTA as for one on every SM: in FP32
// at degree 4, 40 / 46 us to / from the lattice (device time); these take 14 / 10 us for 384 elements.
template <typename Real>
__global__ void __launch_bounds__(128) to_lattice_small_kernel(const Real* state, double* vals, const double* geo, const double* V,
                                                               int64_t ne, int nf, int nb, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const int64_t ek = i / nf, e = ek / nb;
    const int f = (int)(i - ek * nf), k = (int)(ek - e * nb);
    const Real* x = state + (e * nf + f) * nb;
    double acc = 0;
#pragma unroll 8
    for (int a = 0; a < nb; ++a) acc += V[k * nb + a] * (double)x[a];
    vals[i] = geo[e % ne * kGeoStride + 28] * acc;
}

template <typename Real>
__global__ void __launch_bounds__(128) from_lattice_small_kernel(const double* vals, Real* state, const double* geo,
                                                                 const double* Vinv, int64_t ne, int nf, int nb, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const int64_t ef = i / nb, e = ef / nf;
    const int a = (int)(i - ef * nb), f = (int)(ef - e * nf);
    const double* v = vals + e * nb * nf + f;
    const double sq = 1.0 / geo[e % ne * kGeoStride + 28];
    double acc = 0;
#pragma unroll 8
    for (int k = 0; k < nb; ++k) acc += Vinv[a * nb + k] * v[k * nf];
    state[i] = (Real)(sq * acc);
}

// DENSE states of many elements: a thread per (element, function), products in the order of the points.  A
// split-precision evolve turns a change in the last bit of its FP64 state into one of its FP32
// arithmetic, so its states keep this order.  (34 992 elements of degree 4: 465 us; a warp per field with the
// dense products in registers takes 582 us, a thread per value 513 us.)
template <typename Real>
__global__ void __launch_bounds__(256) from_lattice_dense_kernel(const double* vals, Real* state, const double* geo,
                                                                 const double* Vinv, int64_t ne, int nf, int nb, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / nb;
        const int a = (int)(i - e * nb);
        const double sq = 1.0 / geo[e % ne * kGeoStride + 28];
        const double* v = vals + e * nb * nf;
        for (int f = 0; f < nf; ++f) {
            double acc = 0;
            for (int k = 0; k < nb; ++k) acc += Vinv[a * nb + k] * v[k * nf + f];
            state[(e * nf + f) * nb + a] = (Real)(sq * acc);
        }
    }
}

constexpr int kEnergyBlocks = 304;

// squares summed per (element, field), then one division, in a fixed order
template <typename Real, int DIM, int P>
__global__ void __launch_bounds__(LatShape<DIM, P>::NT) energy_partial_kernel(const Real* state, const double* geo, int64_t ne,
                                                                              double* partial) {
    using Sh = LatShape<DIM, P>;
    constexpr int NF = Sh::NF, NB = Sh::NB, NC = Sh::NC, SP = Sh::SP, NT = Sh::NT;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[NT];
    Real* in = (Real*)smem;
    const int lane = threadIdx.x & 31, f = threadIdx.x >> 5;
    const Real* st = state + (int64_t)blockIdx.y * ne * NC;
    const int word = f < (DIM == 3 ? 3 : 2) ? 29 : 30;   // E fields first, then H
    double acc = 0;
    for (int64_t e0 = (int64_t)blockIdx.x * kLatElems; e0 < ne; e0 += (int64_t)gridDim.x * kLatElems) {
        const int ns = (int)(ne - e0 < kLatElems ? ne - e0 : kLatElems);
        const Real* src = st + e0 * NC;
        for (int i = threadIdx.x; i < ns * NC; i += NT) in[i / NC * SP + i % NC] = src[i];
        __syncthreads();
        if (lane < ns) {
            double s0 = 0, s1 = 0;
#pragma unroll
            for (int a = 0; a < NB; ++a) {
                const double y = (double)in[lane * SP + f * NB + a];
                if (a & 1) s1 = __fma_rn(y, y, s1); else s0 = __fma_rn(y, y, s0);
            }
            acc += (s0 + s1) / geo[(e0 + lane) * kGeoStride + word];
        }
        __syncthreads();
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double s = red[threadIdx.x];
#pragma unroll
        for (int w = 1; w < NF; ++w) s += red[threadIdx.x + 32 * w];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

constexpr int kFinalThreads = 256;
__global__ void energy_final_kernel(const double* partial, int nblocks, double* out) {
    __shared__ double red[kFinalThreads];
    const int rhs = blockIdx.x;
    double acc = 0;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) acc += partial[rhs * nblocks + i];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[rhs] = 0.5 * red[0];
}

cudaError_t sm_count(int* n) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
}

// CTAs for n elements: no more than can be resident, so that a CTA's loop amortises its launch
int lattice_grid(int64_t n, int nsm) {
    const int64_t g = (n + kLatElems - 1) / kLatElems;
    return (int)(g < nsm * 32 ? g : nsm * 32);
}

// Elements per SM up to which the small kernels run.  They are as fast as the others, in 3D at degrees 3, 4 and 5 on
// 152 SMs, for about 2700 elements (18 per SM), from the lattice in both precisions and to the lattice in FP64: 14 | 14,
// 36 | 37, 86 | 88 us for 2688 elements with the small | the other kernel, to the lattice in FP64; 19 | 19, 45 | 46,
// 106 | 105 us from it in FP32.  To the lattice in FP32 every product of theirs converts its coefficient, and the
// line is at 1300 elements: 13 | 15, 34 | 40, 81 | 93 us for 1152, 19 | 15, 54 | 41, 134 | 93 us for 1920.
template <typename Real>
constexpr int kSmallTo = sizeof(Real) == 4 ? 8 : 16;
constexpr int kSmallFrom = 16;

template <typename K>
cudaError_t lattice_smem(K kernel, size_t bytes) {
    return bytes > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : cudaSuccess;
}

template <typename Real, int DIM, int P, bool DENSE>
struct Lattice {
    using Sh = LatShape<DIM, P>;
    static cudaError_t to(const Mesh& m, const void* state, double* vals, cudaStream_t st) {
        constexpr size_t bytes = (size_t)kLatElems * Sh::SP * sizeof(double);
        const int64_t n = (int64_t)m.n_rhs * m.ne;
        int nsm = 0;
        cudaError_t e = sm_count(&nsm);
        if (e != cudaSuccess) return e;
        if (n <= (int64_t)kSmallTo<Real> * nsm) {
            to_lattice_small_kernel<Real><<<(unsigned)((n * Sh::NC + 127) / 128), 128, 0, st>>>(
                (const Real*)state, vals, device_geo(m), device_lattice_tables(m)[0], m.ne, Sh::NF, Sh::NB, n * Sh::NC);
            return cudaGetLastError();
        }
        e = lattice_smem(to_lattice_kernel<Real, DIM, P>, bytes);
        if (e != cudaSuccess) return e;
        to_lattice_kernel<Real, DIM, P><<<lattice_grid(n, nsm), Sh::NT, bytes, st>>>((const Real*)state, vals, device_geo(m), m.ne, n);
        return cudaGetLastError();
    }
    static cudaError_t from(const Mesh& m, const double* vals, void* state, cudaStream_t st) {
        constexpr size_t bytes = (size_t)kLatElems * Sh::SP * sizeof(double);
        const int64_t n = (int64_t)m.n_rhs * m.ne;
        int nsm = 0;
        cudaError_t e = sm_count(&nsm);
        if (e != cudaSuccess) return e;
        if (n <= (int64_t)kSmallFrom * nsm) {
            from_lattice_small_kernel<Real><<<(unsigned)((n * Sh::NC + 127) / 128), 128, 0, st>>>(
                vals, (Real*)state, device_geo(m), device_lattice_tables(m)[1], m.ne, Sh::NF, Sh::NB, n * Sh::NC);
            return cudaGetLastError();
        }
        if constexpr (DENSE) {
            const int64_t rows = n * Sh::NB, g = (rows + 255) / 256;
            from_lattice_dense_kernel<Real><<<(unsigned)(g < 65535 ? g : 65535), 256, 0, st>>>(
                vals, (Real*)state, device_geo(m), device_lattice_tables(m)[1], m.ne, Sh::NF, Sh::NB, rows);
        } else {
            e = lattice_smem(from_lattice_kernel<Real, DIM, P>, bytes);
            if (e != cudaSuccess) return e;
            from_lattice_kernel<Real, DIM, P><<<lattice_grid(n, nsm), Sh::NT, bytes, st>>>(vals, (Real*)state, device_geo(m), m.ne, n);
        }
        return cudaGetLastError();
    }
    static cudaError_t energy(const Mesh& m, const void* state, double* partial, cudaStream_t st) {
        constexpr size_t bytes = (size_t)kLatElems * Sh::SP * sizeof(Real);
        const cudaError_t e = lattice_smem(energy_partial_kernel<Real, DIM, P>, bytes);
        if (e != cudaSuccess) return e;
        energy_partial_kernel<Real, DIM, P><<<dim3(kEnergyBlocks, m.n_rhs), Sh::NT, bytes, st>>>((const Real*)state, device_geo(m),
                                                                                                m.ne, partial);
        return cudaGetLastError();
    }
};

struct LatticeEntry {
    cudaError_t (*to)(const Mesh&, const void*, double*, cudaStream_t);
    cudaError_t (*from)(const Mesh&, const double*, void*, cudaStream_t);
    cudaError_t (*energy)(const Mesh&, const void*, double*, cudaStream_t);
};
template <typename Real, int DIM, int P, bool DENSE>
LatticeEntry entry() {
    using L = Lattice<Real, DIM, P, DENSE>;
    return {L::to, L::from, L::energy};
}
template <typename Real, int DIM, bool DENSE = false>
LatticeEntry entry_p(int p) {
    return p == 1 ? entry<Real, DIM, 1, DENSE>() : p == 2 ? entry<Real, DIM, 2, DENSE>() : p == 3 ? entry<Real, DIM, 3, DENSE>()
         : p == 4 ? entry<Real, DIM, 4, DENSE>() : entry<Real, DIM, 5, DENSE>();
}
LatticeEntry lattice_entry(const Mesh& m) {
    if (m.precision == MTP_FP32_SPLIT) return m.dim == 2 ? entry_p<double, 2, true>(m.p) : entry_p<double, 3, true>(m.p);
    if (m.precision == MTP_FP64) return m.dim == 2 ? entry_p<double, 2>(m.p) : entry_p<double, 3>(m.p);
    return m.dim == 2 ? entry_p<float, 2>(m.p) : entry_p<float, 3>(m.p);
}

}  // namespace

size_t energy_scratch_doubles(const Mesh& m) { return (size_t)(kEnergyBlocks + 1) * m.n_rhs; }

int device_from_lattice(Mesh& m, const double* vals, void* state, void* stream) {
    MTP_TRY(device_mesh_upload(m));
    CUDA_TRY(lattice_entry(m).from(m, vals, state, (cudaStream_t)stream));
    return MTP_OK;
}

int device_to_lattice(Mesh& m, const void* state, double* vals, void* stream) {
    MTP_TRY(device_mesh_upload(m));
    CUDA_TRY(lattice_entry(m).to(m, state, vals, (cudaStream_t)stream));
    return MTP_OK;
}

int device_energy(Mesh& m, const void* state, double* out_host, void* stream) {
    MTP_TRY(device_mesh_upload(m));
    cudaStream_t st = (cudaStream_t)stream;
    double* partial = device_energy_scratch(m);
    CUDA_TRY(lattice_entry(m).energy(m, state, partial, st));
    double* out_dev = partial + (size_t)kEnergyBlocks * m.n_rhs;
    energy_final_kernel<<<m.n_rhs, kFinalThreads, 0, st>>>(partial, kEnergyBlocks, out_dev);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaMemcpyAsync(out_host, out_dev, sizeof(double) * m.n_rhs, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return MTP_OK;
}

}  // namespace mtp
