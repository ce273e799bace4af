// Shared pieces of the device-side translation units.
#pragma once

#include <string>

#include <cuda_runtime.h>

#include "mtp_internal.h"

#define CUDA_TRY(call)                                                                       \
    do {                                                                                     \
        cudaError_t _e = (call);                                                             \
        if (_e != cudaSuccess)                                                               \
            return set_error(_e == cudaErrorMemoryAllocation ? MTP_ENOMEM : MTP_ECUDA,       \
                             std::string(#call) + ": " + cudaGetErrorString(_e));            \
    } while (0)

#define MTP_TRY(call)                  \
    do {                               \
        int _rc = (call);              \
        if (_rc != MTP_OK) return _rc; \
    } while (0)

namespace mtp {

// the state between tents is FP64 for MTP_FP64 and MTP_FP32_SPLIT, FP32 otherwise; the reference
// tables and the tent kernels' arithmetic are FP64 only for MTP_FP64
inline bool state_f64(const Mesh& m) { return m.precision == MTP_FP64 || m.precision == MTP_FP32_SPLIT; }

// device copies that belong to an uploaded mesh (mtp_cuda.cu)
const double* device_geo(const Mesh& m);
const double* const* device_lattice_tables(const Mesh& m);   // V and its inverse
double* device_energy_scratch(const Mesh& m);
// doubles that device_energy_scratch holds (mtp_lattice.cu)
size_t energy_scratch_doubles(const Mesh& m);

}  // namespace mtp
