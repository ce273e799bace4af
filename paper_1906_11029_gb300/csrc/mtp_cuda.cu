// Device-side management of the MTP library: uploads and the evolution drivers.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "mtp_adjoint.cuh"
#include "mtp_apex.cuh"
#include "mtp_apex2.cuh"
#include "mtp_device.h"
#include "mtp_internal.h"
#include "mtp_launch.cuh"

namespace mtp {

struct DeviceMesh {
    int device = -1;
    double* geo = nullptr;
    int32_t* elems = nullptr;
    int64_t* patch_ptr = nullptr;
    int32_t* patch_elem = nullptr;
    int8_t* patch_info = nullptr;
    void* S = nullptr;
    void* Tr = nullptr;
    void* L = nullptr;
    void* Mc = nullptr;           // thread-major copies of M, D^T, Tr, L for the SIMT tent kernels
    void* Dc = nullptr;
    void* Trc = nullptr;
    void* Lc = nullptr;
    double* lattice[2] = {nullptr, nullptr};   // V and its inverse
    void* Mc1 = nullptr;          // the same four tables with one row per thread (shape variant 2)
    void* Dc1 = nullptr;
    void* Trc1 = nullptr;
    void* Lc1 = nullptr;
    float* Sf = nullptr;          // tensor-core fragment tables (TF32 modes)
    float* Lfr = nullptr;
    float* Trf = nullptr;
    float* Sf_lo = nullptr;
    float* Lfr_lo = nullptr;
    float* Trf_lo = nullptr;
    float* Dtc = nullptr;         // tcgen05 A operand (variants 3, 4): D^T in core-matrix layout, hi then lo
    std::mutex apex_lock;         // the three below are made by the first call that runs an apex kernel
    bool apex_ready = false;
    void* ent = nullptr;          // apex tent kernel: patch entry records, change of basis
    void* Rt = nullptr;
    void* apex2 = nullptr;        // tables of the 2D apex tent kernel
    double* partial = nullptr;    // energy reduction scratch: [n_rhs][kEnergyBlocks] partials, then [n_rhs] sums
};

struct DeviceTents {
    int32_t* v = nullptr;
    double* tb = nullptr;
    double* tt = nullptr;
    double* tau = nullptr;
    int* err = nullptr;
    int* err_host = nullptr;      // pinned
    void* host_state = nullptr;   // device buffer for mtp_evolve_host
    cudaStream_t capture = nullptr;
    cudaGraphExec_t exec = nullptr;
    void* graph_state = nullptr;  // state pointer baked into the graph
    // persistent DAG walk
    int32_t* tent_layer = nullptr;
    int64_t* vt_ptr = nullptr;
    int32_t* vt_layer = nullptr;
    int64_t* adj_ptr = nullptr;
    int32_t* adj = nullptr;
    int* cnt = nullptr;
    unsigned long long* next = nullptr;
    // adjoint work buffers (grown on demand)
    void* adj_buf = nullptr;
    size_t adj_bytes = 0;
    double* tau_rev = nullptr;
    int64_t* tent_off = nullptr;   // [n_tents + 1]: patch entries of the tents before each tent
};

static size_t real_size(const Mesh& m) { return state_f64(m) ? sizeof(double) : sizeof(float); }

template <typename T>
static int upload(T** dst, const T* src, size_t n) {
    CUDA_TRY(cudaMalloc((void**)dst, n * sizeof(T) + 16));
    CUDA_TRY(cudaMemcpy(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice));
    return MTP_OK;
}

// rows of `cols` entries -> rows of pad4(cols) entries, zeros in the pad (16-byte vector reads)
static std::vector<double> pad_rows(const std::vector<double>& src, int cols) {
    const int pc = pad4(cols);
    const size_t rows = src.size() / cols;
    std::vector<double> out(rows * pc, 0.0);
    for (size_t r = 0; r < rows; ++r)
        for (int c = 0; c < cols; ++c) out[r * pc + c] = src[r * cols + c];
    return out;
}

// Thread-major layout of `nmat` row-major rows x cols matrices for the SIMT tent kernels.
// With nrg = ceil(rows / ap) row groups, a thread owns rows g, g + nrg, ..., and reads, per
// step, `w` consecutive columns of each of them as one 16-byte vector; consecutive threads
// own consecutive groups.  Entry (r, c) of matrix mt goes to
//   [mt][c / w][r / nrg][r % nrg][c % w]   (columns padded to pad4(cols), rows to ap * nrg)
// so that the vectors that the lanes of a warp read for one (matrix, column block, row of
// the group) are contiguous in memory, and the rows the lanes write are consecutive.
static std::vector<double> thread_major(const std::vector<double>& src, int nmat, int rows, int cols, int w,
                                        int ap) {
    const int nch = pad4(cols) / w, nrg = (rows + ap - 1) / ap;
    const size_t msz = (size_t)nch * ap * nrg * w;
    std::vector<double> out(nmat * msz, 0.0);
    for (int mt = 0; mt < nmat; ++mt)
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c)
                out[mt * msz + (((size_t)(c / w) * ap + r / nrg) * nrg + r % nrg) * w + c % w] =
                    src[((size_t)mt * rows + r) * cols + c];
    return out;
}

static int upload_real(const Mesh& m, void** dst, const std::vector<double>& src) {
    if (m.precision == MTP_FP64) return upload((double**)dst, src.data(), src.size());   // FP32 arithmetic otherwise
    std::vector<float> f(src.begin(), src.end());
    return upload((float**)dst, f.data(), f.size());
}

// A-operand tables in m16n8k8 fragment order: fragment (mt, kt) of a row-major M x K matrix
// A (zero outside rows < rows, cols < cols) is 32 lanes x 4 values: lane (g = lane/4,
// t = lane%4) holds A[16mt+g][8kt+t], A[16mt+g+8][8kt+t], A[16mt+g][8kt+t+4], A[16mt+g+8][8kt+t+4].
// Values are TF32-rounded (round to nearest even at 10 mantissa bits); `lo` receives the
// TF32-rounded remainder for the split mode.
static float tf32_round(float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    if ((u & 0x7f800000u) != 0x7f800000u) u += 0xfffu + ((u >> 13) & 1u);
    u &= 0xffffe000u;
    std::memcpy(&x, &u, 4);
    return x;
}
template <typename Get>
static void append_fragments(std::vector<float>& hi, std::vector<float>& lo, int MT, int KT, Get A) {
    for (int mt = 0; mt < MT; ++mt)
        for (int kt = 0; kt < KT; ++kt)
            for (int lane = 0; lane < 32; ++lane) {
                const int g = lane >> 2, t = lane & 3;
                const double v[4] = {A(16 * mt + g, 8 * kt + t), A(16 * mt + g + 8, 8 * kt + t),
                                     A(16 * mt + g, 8 * kt + t + 4), A(16 * mt + g + 8, 8 * kt + t + 4)};
                for (int q = 0; q < 4; ++q) {
                    const float h = tf32_round((float)v[q]);
                    hi.push_back(h);
                    lo.push_back(tf32_round((float)(v[q] - (double)h)));
                }
            }
}

// Records of the patch entries for the apex tent kernel (layout at kApexRec); one warp per vertex,
// one lane per patch element, FP64 arithmetic, stored in the arithmetic precision.
template <typename Real>
__global__ void apex_record_kernel(int64_t nv, const int64_t* patch_ptr, const int32_t* patch_elem,
                                   const int8_t* patch_info, const double* geo, Real* ent) {
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (v >= nv) return;
    const int64_t pb = patch_ptr[v];
    for (int64_t at = pb + (threadIdx.x & 31); at < patch_ptr[v + 1]; at += 32) {
        const int8_t* info = patch_info + at * 12;
        const double* g = geo + (int64_t)patch_elem[at] * kGeoStride;
        const int j = info[0];
        double gr[3][3], t[3][3];
        for (int w = 0; w < 3; ++w)
            for (int q = 0; q < 3; ++q) gr[w][q] = g[3 * (w < j ? w : w + 1) + q];
        // edges from V: dual to the gradients of the other vertices' barycentric coordinates
        double c[3][3];
        for (int w = 0; w < 3; ++w) {
            const double *x = gr[(w + 1) % 3], *y = gr[(w + 2) % 3];
            c[w][0] = x[1] * y[2] - x[2] * y[1];
            c[w][1] = x[2] * y[0] - x[0] * y[2];
            c[w][2] = x[0] * y[1] - x[1] * y[0];
        }
        const double dg = gr[0][0] * c[0][0] + gr[0][1] * c[0][1] + gr[0][2] * c[0][2];
        const double s = g[28], l = exp2(rint(log2(1.0 / (s * s)) / 3.0));
        for (int w = 0; w < 3; ++w)
            for (int q = 0; q < 3; ++q) {
                t[w][q] = c[w][q] / dg / l;
                gr[w][q] *= l;
            }
        const double det = 1.0 / (dg * l * l * l), ts = l * s, sgn = det > 0 ? 1.0 : -1.0;
        Real* r = ent + at * kApexRec;
        auto dot = [](const double* x, const double* y) { return x[0] * y[0] + x[1] * y[1] + x[2] * y[2]; };
        int n = 0;
        double G[3][3];
        for (int w = 0; w < 3; ++w)
            for (int x = w; x < 3; ++x, ++n) {
                G[w][x] = G[x][w] = dot(t[w], t[x]);
                r[n] = (Real)G[w][x];
                r[6 + n] = (Real)dot(gr[w], gr[x]);
            }
        r[12] = (Real)(1.0 / l);
        r[13] = (Real)g[29];
        r[14] = (Real)g[30];
        r[15] = (Real)det;
        r[16] = (Real)(1.0 / (l * det));
        r[17] = (Real)(ts * l * det);
        r[18] = (Real)(1.0 / (l * det * ts));
        r[19] = (Real)(1.0 / (g[29] * g[30]));
        for (int fi = 0; fi < 3; ++fi) {
            const int X = fi == 0 ? 1 : 0, Y = fi == 2 ? 1 : 2;
            const int s2 = info[4 + (fi < j ? fi : fi + 1)];
            const double zm = g[31], zp = s2 >= 0 ? geo[(int64_t)patch_elem[pb + s2] * kGeoStride + 31] : zm;
            const double area = sqrt(G[X][X] * G[Y][Y] - G[X][Y] * G[X][Y]), q = sgn / (area * (zm + zp));
            Real* o = r + kApexFacet + 6 * fi;
            o[0] = (Real)(zm / (zm + zp));
            o[1] = (Real)(zp / (zm + zp));
            o[2] = (Real)(q * G[Y][Y]);
            o[3] = (Real)(-q * G[X][Y]);
            o[4] = (Real)(q * G[X][X]);
            o[5] = (Real)(zm * zp);
        }
        for (int w = 0; w < 3; ++w)
            for (int q = 0; q < 3; ++q) {
                r[kApexDual + 3 * w + q] = (Real)gr[w][q];
                r[kApexEdge + 3 * w + q] = (Real)t[w][q];
            }
    }
}

template <typename Real>
static int apex_upload_real(const Mesh& m, DeviceMesh& d) {
    std::vector<Real> rt;
    const int nb = m.nb;
    for (int j = 0; j < 4; ++j)
        for (int k = 0, b0 = 0; k <= m.p; b0 += apex_rot_block(k), ++k) {
            const int n = apex_rot_block(k);
            for (int a = 0; a < n; ++a)
                for (int b = 0; b < pad4(n); ++b)
                    rt.push_back(b < n ? (Real)m.ref.Rot[((size_t)j * nb + b0 + a) * nb + b0 + b] : Real(0));
        }
    MTP_TRY(upload((Real**)&d.Rt, rt.data(), rt.size()));
    CUDA_TRY(cudaMalloc(&d.ent, m.patch_elem.size() * kApexRec * sizeof(Real) + 16));
    const int64_t blocks = (m.nv * 32 + 127) / 128;
    apex_record_kernel<Real><<<(unsigned)blocks, 128>>>(m.nv, d.patch_ptr, d.patch_elem, d.patch_info, d.geo, (Real*)d.ent);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaDeviceSynchronize());   // later launches may use any stream
    return MTP_OK;
}

// the same in 2D (layout at kApex2Rec); one thread per patch entry
template <typename Real>
__global__ void apex2_record_kernel(int64_t nv, const int64_t* patch_ptr, const int32_t* patch_elem,
                                    const int8_t* patch_info, const double* geo, Real* ent) {
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    if (v >= nv) return;
    const int64_t pb = patch_ptr[v];
    for (int64_t at = pb + (threadIdx.x & 15); at < patch_ptr[v + 1]; at += 16) {
        const int8_t* info = patch_info + at * 12;
        const double* g = geo + (int64_t)patch_elem[at] * kGeoStride;
        const int j = info[0];
        double gr[2][2], t[2][2];
        for (int w = 0; w < 2; ++w)
            for (int q = 0; q < 2; ++q) gr[w][q] = g[3 * (w < j ? w : w + 1) + q];
        const double dg = gr[0][0] * gr[1][1] - gr[0][1] * gr[1][0];
        const double s = g[28], l = exp2(rint(log2(1.0 / (s * s)) / 2.0));
        t[0][0] = gr[1][1] / dg / l;
        t[0][1] = -gr[1][0] / dg / l;
        t[1][0] = -gr[0][1] / dg / l;
        t[1][1] = gr[0][0] / dg / l;
        for (int w = 0; w < 2; ++w)
            for (int q = 0; q < 2; ++q) gr[w][q] *= l;
        const double det = 1.0 / (dg * l * l), sgn = det > 0 ? 1.0 : -1.0, c1 = 1.0 / (l * det), eps = g[29], mu = g[30];
        Real* r = ent + at * kApex2Rec;
        auto dot = [](const double* x, const double* y) { return x[0] * y[0] + x[1] * y[1]; };
        r[0] = (Real)dot(t[0], t[0]);
        r[1] = (Real)dot(t[0], t[1]);
        r[2] = (Real)dot(t[1], t[1]);
        r[3] = (Real)dot(gr[0], gr[0]);
        r[4] = (Real)dot(gr[0], gr[1]);
        r[5] = (Real)dot(gr[1], gr[1]);
        r[6] = (Real)(1.0 / l);
        r[7] = (Real)eps;
        r[8] = (Real)mu;
        r[9] = (Real)(c1 / (l * s));
        r[10] = (Real)(1.0 / (eps * mu));
        r[11] = (Real)c1;
        r[12] = (Real)(-s / c1);
        r[13] = (Real)(l * s / c1);
        r[14] = (Real)(1.0 / det);
        for (int f = 0; f < 2; ++f) {
            const int s2 = info[4 + (1 - f < j ? 1 - f : 2 - f)];
            const double zm = g[31], zp = s2 >= 0 ? geo[(int64_t)patch_elem[pb + s2] * kGeoStride + 31] : zm;
            const double len = l * sqrt(dot(t[f], t[f]));
            r[15 + 4 * f] = (Real)(zm / (zm + zp));
            r[16 + 4 * f] = (Real)(zp / (zm + zp));
            r[17 + 4 * f] = (Real)(sgn / (len * (zm + zp)));
            r[18 + 4 * f] = (Real)(sgn * zm * zp * len / (zm + zp));
        }
        for (int w = 0; w < 2; ++w)
            for (int q = 0; q < 2; ++q) {
                r[23 + 2 * w + q] = (Real)gr[w][q];
                r[27 + 2 * w + q] = (Real)t[w][q];
            }
        r[31] = (Real)(-c1 / s);
    }
}

template <typename Real>
static int apex2_upload_real(const Mesh& m, DeviceMesh& d) {
    const RefTables& r = m.ref;
    const int nb = m.nb, nfb = m.nfb;
    std::vector<Real> t((size_t)nb * nb, Real(0));
    std::vector<uint8_t> rows(4 * nb + nb * nb + nb, 0);
    auto parity = [](int b) {
        int g = 0;
        while (b >= (g + 1) * (g + 2) / 2) ++g;
        return (b - g * (g + 1) / 2) & 1;
    };
    int n = 0;
    for (int a = 0; a < nb; ++a) {   // compressed rows: equal parity first
        rows[4 * a] = (uint8_t)(n & 255);
        rows[4 * a + 1] = (uint8_t)(n >> 8);
        for (int opp = 0; opp < 2; ++opp)
            for (int b = 0; b < nb; ++b)
                if ((parity(a) != parity(b)) == (opp == 1) && r.C2[(size_t)a * nb + b] != 0.0) {
                    t[n] = (Real)r.C2[(size_t)a * nb + b];
                    rows[4 * nb + n] = (uint8_t)b;
                    rows[4 * a + 2 + opp]++;
                    ++n;
                }
        if (rows[4 * a + 2] + rows[4 * a + 3] > kApex2MaxRow[m.p - 1])
            return set_error(MTP_EINVAL, "2D apex tables: a row is longer than the kernel reads");
        rows[4 * nb + nb * nb + a] = (uint8_t)a;
    }
    std::stable_sort(rows.end() - nb, rows.end(), [&](uint8_t a, uint8_t b) {
        return rows[4 * a + 2] + rows[4 * a + 3] < rows[4 * b + 2] + rows[4 * b + 3];
    });
    for (double v : r.T2) t.push_back((Real)v);
    for (double v : r.L2) t.push_back((Real)v);
    for (int j = 0; j < 3; ++j)
        for (int a = 0, g = 0; a < nb; ++a) {
            while (a >= (g + 1) * (g + 2) / 2) ++g;
            for (int b = 0; b < nfb; ++b)
                t.push_back(b <= g ? (Real)r.Rot[((size_t)j * nb + a) * nb + g * (g + 1) / 2 + b] : Real(0));
        }
    std::vector<uint8_t> buf(t.size() * sizeof(Real) + rows.size());
    std::memcpy(buf.data(), t.data(), t.size() * sizeof(Real));
    std::memcpy(buf.data() + t.size() * sizeof(Real), rows.data(), rows.size());
    MTP_TRY(upload((uint8_t**)&d.apex2, buf.data(), buf.size()));
    CUDA_TRY(cudaMalloc(&d.ent, m.patch_elem.size() * kApex2Rec * sizeof(Real) + 16));
    const int64_t blocks = (m.nv * 16 + 127) / 128;
    apex2_record_kernel<Real><<<(unsigned)blocks, 128>>>(m.nv, d.patch_ptr, d.patch_elem, d.patch_info, d.geo, (Real*)d.ent);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaDeviceSynchronize());
    return MTP_OK;
}

// Records and tables of the apex kernels, made once per mesh by the first evolve, batch or gradient that runs
// one: exchange and energy calls, the other modes and stretched meshes do without them (first exchange on a mesh
// of 32^3 x 6 elements in FP32: 2.5 ms when they came with the mesh, 1.25 ms now).  Tents handles of a mesh may
// come here from several threads.
static int apex_upload(const Mesh& m) {
    DeviceMesh& d = *m.dev;
    std::lock_guard<std::mutex> lock(d.apex_lock);
    if (d.apex_ready) return MTP_OK;
    const bool f64 = m.precision == MTP_FP64;   // the tensor-core modes' adjoint runs in FP32
    const int rc = m.dim == 2 ? (f64 ? apex2_upload_real<double>(m, d) : apex2_upload_real<float>(m, d))
                              : (f64 ? apex_upload_real<double>(m, d) : apex_upload_real<float>(m, d));
    if (rc == MTP_OK) {
        d.apex_ready = true;
        return MTP_OK;
    }
    for (void** p : {&d.ent, &d.Rt, &d.apex2}) {   // the next call tries again
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
    cudaGetLastError();
    return rc;
}

static int mesh_buffers(Mesh& m) {
    DeviceMesh& d = *m.dev;
    MTP_TRY(upload(&d.geo, m.geo.data(), m.geo.size()));
    MTP_TRY(upload(&d.lattice[0], m.ref.V.data(), m.ref.V.size()));
    MTP_TRY(upload(&d.lattice[1], m.ref.Vinv.data(), m.ref.Vinv.size()));
    MTP_TRY(upload(&d.elems, m.elems.data(), m.elems.size()));
    MTP_TRY(upload(&d.patch_ptr, m.patch_ptr.data(), m.patch_ptr.size()));
    MTP_TRY(upload(&d.patch_elem, m.patch_elem.data(), m.patch_elem.size()));
    MTP_TRY(upload(&d.patch_info, m.patch_info.data(), m.patch_info.size()));
    MTP_TRY(upload_real(m, &d.S, pad_rows(m.ref.S, m.nb)));     // [j][l][a][NBP]
    MTP_TRY(upload_real(m, &d.Tr, pad_rows(m.ref.Tr, m.nb)));   // [f][c][NBP]
    MTP_TRY(upload_real(m, &d.L, pad_rows(m.ref.L, m.nfb)));    // [j][f][a][NFBP]
    {
        const int w = m.precision == MTP_FP64 ? 2 : 4, ap = 2, nv = m.dim + 1;
        // factored volume: M[j] (rows c < nbm, columns b) and D[l]^T (rows a, columns c < nbm)
        const int nbm = m.ref.nbm;
        std::vector<double> Dt((size_t)m.dim * m.nb * nbm);
        for (int l = 0; l < m.dim; ++l)
            for (int c = 0; c < nbm; ++c)
                for (int a = 0; a < m.nb; ++a)
                    Dt[((size_t)l * m.nb + a) * nbm + c] = m.ref.D[((size_t)l * nbm + c) * m.nb + a];
        MTP_TRY(upload_real(m, &d.Mc, thread_major(m.ref.M, nv, nbm, m.nb, w, ap)));
        MTP_TRY(upload_real(m, &d.Dc, thread_major(Dt, m.dim, m.nb, nbm, w, ap)));
        MTP_TRY(upload_real(m, &d.Trc, thread_major(m.ref.Tr, nv, m.nfb, m.nb, w, ap)));
        MTP_TRY(upload_real(m, &d.Lc, thread_major(m.ref.L, nv * nv, m.nb, m.nfb, w, ap)));
        if (m.precision == MTP_FP32 && m.dim == 3 && m.p >= 2 && m.p <= 4) {
            // A operand of the tcgen05 volume term: D[a][k], k = l nbm + c, = D_l^T[a][c], rows a
            // padded to tn = 64 (the MMA's M), k to tk = 8, K-major core matrices (8 rows x 4
            // values), 8-row groups tk x 8 floats apart; TF32 hi part, then the TF32 remainder
            const int tk = (3 * nbm + 7) / 8 * 8, tn = 64;
            std::vector<float> bt((size_t)2 * tn * tk, 0.0f);
            for (int a = 0; a < m.nb; ++a)
                for (int l = 0; l < 3; ++l)
                    for (int c = 0; c < nbm; ++c) {
                        const int k = l * nbm + c;
                        const size_t o = (size_t)(a >> 3) * tk * 8 + (k >> 2) * 32 + (a & 7) * 4 + (k & 3);
                        const double v = Dt[((size_t)l * m.nb + a) * nbm + c];
                        const float h = tf32_round((float)v);
                        bt[o] = h;
                        bt[(size_t)tn * tk + o] = tf32_round((float)(v - (double)h));
                    }
            MTP_TRY(upload(&d.Dtc, bt.data(), bt.size()));
        }
        if (m.precision == MTP_FP32 || (m.precision == MTP_FP32_SPLIT && m.dim == 3 && m.p <= 3)) {
            MTP_TRY(upload_real(m, &d.Mc1, thread_major(m.ref.M, nv, nbm, m.nb, w, 1)));
            MTP_TRY(upload_real(m, &d.Dc1, thread_major(Dt, m.dim, m.nb, nbm, w, 1)));
            MTP_TRY(upload_real(m, &d.Trc1, thread_major(m.ref.Tr, nv, m.nfb, m.nb, w, 1)));
            MTP_TRY(upload_real(m, &d.Lc1, thread_major(m.ref.L, nv * nv, m.nb, m.nfb, w, 1)));
        }
    }
    if (m.precision == MTP_TF32 || m.precision == MTP_TF32X3) {
        const RefTables& r = m.ref;
        const int nb = m.nb, nfb = m.nfb, d3 = m.dim, nvx = m.dim + 1;
        const int MT = (nb + 15) / 16, KT = (nb + 7) / 8, KTL = (nfb + 7) / 8;
        std::vector<float> sh, sl, lh, ll, th, tl;
        for (int j = 0; j <= d3; ++j)
            for (int l = 0; l < d3; ++l)
                append_fragments(sh, sl, MT, KT, [&](int a, int b) {
                    return (a < nb && b < nb) ? r.S[(((size_t)j * d3 + l) * nb + a) * nb + b] : 0.0;
                });
        for (int j = 0; j <= d3; ++j)
            for (int f = 0; f < nvx; ++f)
                append_fragments(lh, ll, MT, KTL, [&](int a, int cc) {
                    return (a < nb && cc < nfb) ? r.L[(((size_t)j * nvx + f) * nb + a) * nfb + cc] : 0.0;
                });
        for (int f = 0; f < nvx; ++f)
            append_fragments(th, tl, 1, KT, [&](int cc, int b) {
                return (cc < nfb && b < nb) ? r.Tr[((size_t)f * nfb + cc) * nb + b] : 0.0;
            });
        MTP_TRY(upload(&d.Sf, sh.data(), sh.size()));
        MTP_TRY(upload(&d.Lfr, lh.data(), lh.size()));
        MTP_TRY(upload(&d.Trf, th.data(), th.size()));
        MTP_TRY(upload(&d.Sf_lo, sl.data(), sl.size()));
        MTP_TRY(upload(&d.Lfr_lo, ll.data(), ll.size()));
        MTP_TRY(upload(&d.Trf_lo, tl.data(), tl.size()));
    }
    CUDA_TRY(cudaMalloc((void**)&d.partial, sizeof(double) * energy_scratch_doubles(m)));
    CUDA_TRY(cudaStreamSynchronize(0));   // the copies: the first kernels may run on any stream
    return MTP_OK;
}

// The mesh's device copies, made by the first call, whichever thread it comes from.  Where one of them has no room, all
// are given back and the next call tries again: nothing may run with some of them missing.
int device_mesh_upload(Mesh& m) {
    int dev;
    CUDA_TRY(cudaGetDevice(&dev));
    static std::mutex lock;
    std::lock_guard<std::mutex> guard(lock);
    if (m.dev) {
        if (m.dev->device == dev) return MTP_OK;
        return set_error(MTP_EINVAL, "mesh was uploaded to another device");
    }
    m.dev = new DeviceMesh();
    m.dev->device = dev;
    const int rc = mesh_buffers(m);
    if (rc == MTP_OK) return rc;
    device_mesh_free(m);
    cudaGetLastError();
    return rc;
}

void device_mesh_free(Mesh& m) {
    if (!m.dev) return;
    DeviceMesh& d = *m.dev;
    void* ptrs[] = {d.lattice[0], d.lattice[1], d.geo, d.elems, d.patch_ptr, d.patch_elem, d.patch_info, d.S, d.Tr, d.L, d.Mc, d.Dc, d.Trc, d.Lc, d.Mc1, d.Dc1, d.Trc1, d.Lc1,
                    d.partial,
                    d.Sf, d.Lfr, d.Trf, d.Sf_lo, d.Lfr_lo, d.Trf_lo, d.Dtc, d.ent, d.Rt, d.apex2};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete m.dev;
    m.dev = nullptr;
}

void device_tents_free(Tents& t) {
    if (!t.dev) return;
    DeviceTents& d = *t.dev;
    if (d.exec) cudaGraphExecDestroy(d.exec);
    if (d.capture) cudaStreamDestroy(d.capture);
    void* ptrs[] = {d.v, d.tb, d.tt, d.tau, d.err, d.host_state, d.adj_buf, d.tau_rev, d.tent_off, d.tent_layer, d.vt_ptr,
                    d.vt_layer, d.adj_ptr, d.adj, d.cnt, d.next};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (d.err_host) cudaFreeHost(d.err_host);
    delete t.dev;
    t.dev = nullptr;
}

static int tents_buffers(Tents& t) {
    DeviceTents& d = *t.dev;
    MTP_TRY(upload(&d.v, t.vertex.data(), t.vertex.size()));
    MTP_TRY(upload(&d.tb, t.t_bot.data(), t.t_bot.size()));
    MTP_TRY(upload(&d.tt, t.t_top.data(), t.t_top.size()));
    CUDA_TRY(cudaMalloc((void**)&d.tau, sizeof(double) * t.mesh->nv));
    CUDA_TRY(cudaMalloc((void**)&d.err, sizeof(int)));
    CUDA_TRY(cudaMallocHost((void**)&d.err_host, sizeof(int)));
    CUDA_TRY(cudaStreamCreateWithFlags(&d.capture, cudaStreamNonBlocking));
    // per-vertex tent layers (tents are sorted by layer, so each list is ascending)
    const Mesh& m = *t.mesh;
    std::vector<int64_t> vt_ptr(m.nv + 1, 0);
    for (int32_t v : t.vertex) vt_ptr[v + 1]++;
    for (int64_t v = 0; v < m.nv; ++v) vt_ptr[v + 1] += vt_ptr[v];
    std::vector<int32_t> vt_layer(t.vertex.size());
    {
        std::vector<int64_t> fill(vt_ptr.begin(), vt_ptr.end() - 1);
        for (size_t i = 0; i < t.vertex.size(); ++i) vt_layer[fill[t.vertex[i]]++] = t.layer[i];
    }
    MTP_TRY(upload(&d.tent_layer, t.layer.data(), t.layer.size()));
    MTP_TRY(upload(&d.vt_ptr, vt_ptr.data(), vt_ptr.size()));
    MTP_TRY(upload(&d.vt_layer, vt_layer.data(), vt_layer.size()));
    MTP_TRY(upload(&d.adj_ptr, m.adj_ptr.data(), m.adj_ptr.size()));
    MTP_TRY(upload(&d.adj, m.adj.data(), m.adj.size()));
    CUDA_TRY(cudaMalloc((void**)&d.cnt, sizeof(int) * m.nv));
    CUDA_TRY(cudaMalloc((void**)&d.next, sizeof(unsigned long long)));
    CUDA_TRY(cudaStreamSynchronize(0));
    return MTP_OK;
}

// all or nothing, as device_mesh_upload
static int device_tents_upload(Tents& t) {
    MTP_TRY(device_mesh_upload(*t.mesh));
    if (t.dev) return MTP_OK;
    t.dev = new DeviceTents();
    const int rc = tents_buffers(t);
    if (rc == MTP_OK) return rc;
    device_tents_free(t);
    cudaGetLastError();
    return rc;
}

// item shape of the tents' kernel on the current device
static int item_shape(const Tents& t) {
    int dev = 0, nsm = 0;
    if (t.mesh->precision != MTP_FP32_SPLIT || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return t.variant;
    return walk_shape(t, nsm);
}

// general tent kernels
static const KernelEntry& general_entry(const Mesh& m, int variant) {
    static KernelEntry f64[2][5], f32[2][5], tc[2][5], split[2][5], narrow[3], rk4[2][5], f32v1[2][5], f32v2[2][5], tc5[2][5];
    static std::once_flag once;   // calls come from several threads
    std::call_once(once, [] {
        kernel_table_f32_tc5(tc5);
        kernel_table_f64(f64);
        kernel_table_f32(f32);
        kernel_table_tc(tc);
        kernel_table_split(split);
        kernel_table_split_narrow(narrow);
        kernel_table_rk4(rk4);
        kernel_table_f32_v1(f32v1);
        kernel_table_f32_v2(f32v2);
    });
    if ((variant == 3 || variant == 4) && m.precision == MTP_FP32 && m.dim == 3 && !(m.flags & MTP_FLAG_SUBSTITUTED_RK4))
        return tc5[variant - 3][m.p - 1];   // null entries outside p = 2..4 (refused when the variant is set)
    if (variant == 2 && m.precision == MTP_FP32 && !(m.flags & MTP_FLAG_SUBSTITUTED_RK4))
        return f32v2[m.dim - 2][m.p - 1];
    if (variant == 1 && m.precision == MTP_FP32 && !(m.flags & MTP_FLAG_SUBSTITUTED_RK4))
        return f32v1[m.dim - 2][m.p - 1];
    if (m.flags & MTP_FLAG_SUBSTITUTED_RK4) return rk4[m.dim - 2][m.p - 1];   // FP64 only (checked at creation)
    if (m.precision == MTP_FP32_SPLIT && variant == 2) return narrow[m.p - 1];
    if (m.precision == MTP_FP32_SPLIT) return split[m.dim - 2][m.p - 1];
    if (m.precision == MTP_TF32 || m.precision == MTP_TF32X3)
        return tc[m.precision == MTP_TF32 ? 0 : 1][m.p - 1];
    return (m.precision == MTP_FP64 ? f64 : f32)[m.dim - 2][m.p - 1];
}

// Whether the mesh's tents run in the apex kernels: the plain SAT modes of their degrees, unless the mesh is
// stretched.  A stretched mesh whose patches are too large for the general kernel's shared memory (FP64, 3D,
// p = 4, more than 30 tetrahedra) has no other kernel than the apex one.
static bool apex_runs(const Mesh& m, int variant) {
    if ((m.precision != MTP_FP64 && m.precision != MTP_FP32) || (m.flags & MTP_FLAG_SUBSTITUTED_RK4) || variant > 2 ||
        (m.dim == 3 && m.p > kApexMaxDegree))
        return false;
    size_t bytes = 0;
    return !m.stretched || general_entry(m, variant).prepare(m.max_patch, &bytes) != cudaSuccess;
}

static const KernelEntry& kernel_entry(const Mesh& m, int variant = 0) {
    if (!apex_runs(m, variant)) return general_entry(m, variant);
    static KernelEntry apex[2][2][5];
    static std::once_flag once;   // calls come from several threads
    std::call_once(once, [] {
        for (int p = 1; p <= 5; ++p) {
            apex[0][0][p - 1] = apex2_entry_f64(p);
            apex[1][0][p - 1] = apex2_entry_f32(p);
            if (p > kApexMaxDegree) continue;
            apex[0][1][p - 1] = apex_entry_f64(p);
            apex[1][1][p - 1] = apex_entry_f32(p);
        }
    });
    return apex[m.precision == MTP_FP64 ? 0 : 1][m.dim - 2][m.p - 1];
}

const double* device_geo(const Mesh& m) { return m.dev->geo; }
const double* const* device_lattice_tables(const Mesh& m) { return m.dev->lattice; }
double* device_energy_scratch(const Mesh& m) { return m.dev->partial; }

// ---------------------------------------------------------------------------------
// evolution
// ---------------------------------------------------------------------------------
// `shape`: the item shape of the kernel that reads the arguments, which decides the row grouping of its
// thread-major tables (general batch and adjoint kernels: 0 whatever variant the handle has)
static void fill_args(Tents& t, void* state, KArgs& a, int shape) {
    Mesh& m = *t.mesh;
    DeviceMesh& dm = *m.dev;
    DeviceTents& dt = *t.dev;
    std::memset(&a, 0, sizeof(a));
    a.tent_v = dt.v;
    a.tent_tb = dt.tb;
    a.tent_tt = dt.tt;
    a.patch_ptr = dm.patch_ptr;
    a.patch_elem = dm.patch_elem;
    a.patch_info = dm.patch_info;
    a.elems = dm.elems;
    a.geo = dm.geo;
    a.tau = dt.tau;
    a.S = dm.S;
    a.Tr = dm.Tr;
    a.L = dm.L;
    a.Mc = dm.Mc;
    a.Dc = dm.Dc;
    a.Trc = dm.Trc;
    a.Lc = dm.Lc;
    if (shape == 2 || shape == 4) {   // one row per thread: one row group per matrix row
        a.Mc = dm.Mc1;
        a.Dc = dm.Dc1;
        a.Trc = dm.Trc1;
        a.Lc = dm.Lc1;
    }
    a.Sf = (const float4*)dm.Sf;
    a.Lfr = (const float4*)dm.Lfr;
    a.Trf = (const float4*)dm.Trf;
    a.Sf_lo = (const float4*)dm.Sf_lo;
    a.Lfr_lo = (const float4*)dm.Lfr_lo;
    a.Trf_lo = (const float4*)dm.Trf_lo;
    a.Dtc = dm.Dtc;
    a.ent = dm.ent;
    a.Rt = dm.Rt;
    a.apex2 = dm.apex2;
    a.state = state;
    a.rhs_stride = m.ne * m.nf * m.nb;
    a.err = dt.err;
    a.q = m.q;
    a.m = m.m;
    a.max_patch = m.max_patch;
    double f = 1.0;
    for (int i = 0; i <= kMaxSub; ++i) a.tsub[i] = i <= m.m ? (double)i / (double)m.m : 1.0;
    for (int n = 0; n < kMaxTaylor; ++n) {
        if (n > 0) f = f / (double)m.m / (double)n;
        a.taylor[n] = f;
    }
}

static int enqueue_layers(Tents& t, const KArgs& a, int64_t lb, int64_t le, cudaStream_t st) {
    const KernelEntry& ke = kernel_entry(*t.mesh, item_shape(t));
    for (int64_t l = lb; l < le; ++l) {
        const int64_t t0 = t.layer_ptr[l];
        const int64_t n = t.layer_ptr[l + 1] - t0;
        if (n == 0) continue;
        CUDA_TRY(ke.launch(a, t0, (int)n, t.mesh->n_rhs, st));
    }
    return MTP_OK;
}

static int check_error_word(Tents& t, cudaStream_t st) {
    DeviceTents& d = *t.dev;
    CUDA_TRY(cudaMemcpyAsync(d.err_host, d.err, sizeof(int), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (*d.err_host == 1) return set_error(MTP_ECAUSAL, "a tent violated |grad phi| < sqrt(eps mu)");
    if (*d.err_host == 2) return set_error(MTP_ENUMERIC, "non-finite value in the evolved state");
    if (*d.err_host == 3) return set_error(MTP_ETIMEOUT, "a tent's wait for its predecessors exceeded the limit");
    if (*d.err_host != 0) return set_error(MTP_ECUDA, "unknown device error word");
    return MTP_OK;
}

// front before layer lb (each vertex at the top of its last earlier tent) -> dst (device)
static int set_front(Tents& t, int64_t lb, double* dst, cudaStream_t st) {
    std::vector<double> tau(t.mesh->nv, 0.0);
    for (int64_t i = 0; i < t.layer_ptr[lb]; ++i) tau[t.vertex[i]] = std::fmax(tau[t.vertex[i]], t.t_top[i]);
    CUDA_TRY(cudaMemcpyAsync(dst, tau.data(), sizeof(double) * t.mesh->nv, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaStreamSynchronize(st));   // the host vector goes out of scope
    return MTP_OK;
}

int device_evolve(Tents& t, void* state, int64_t lb, int64_t le, bool use_graph, void* stream) {
    MTP_TRY(device_tents_upload(t));
    Mesh& m = *t.mesh;
    DeviceTents& d = *t.dev;
    cudaStream_t st = (cudaStream_t)stream;
    if (apex_runs(m, item_shape(t))) MTP_TRY(apex_upload(m));
    const KernelEntry& ke = kernel_entry(m, item_shape(t));
    size_t smem = 0;
    const cudaError_t pe = ke.prepare(m.max_patch, &smem);
    int dev, smem_max;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if ((int64_t)smem > smem_max)
        return set_error(MTP_EUNSUPPORTED, "tent kernel needs " + std::to_string(smem) +
                                               " bytes of shared memory per block; the device allows " +
                                               std::to_string(smem_max));
    CUDA_TRY(pe);
    MTP_TRY(set_front(t, lb, d.tau, st));
    CUDA_TRY(cudaMemsetAsync(d.err, 0, sizeof(int), st));
    KArgs a;
    fill_args(t, state, a, item_shape(t));
    const bool full = lb == 0 && le == (int64_t)t.layer_ptr.size() - 1;
    const int launch = (m.flags & MTP_FLAG_LAYER_LAUNCHES) ? 2 : t.launch;
    if (launch != 2 && le > lb) {
        int bpsm = 0, nsm = 0;
        CUDA_TRY(ke.persistent_prepare(m.max_patch, &bpsm));
        CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        const int64_t t0 = t.layer_ptr[lb], nt = t.layer_ptr[le] - t0;
        const int cps = launch == 1 ? 1 : walk_ctas(t, lb, le, nsm, bpsm);
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(nt, (int64_t)cps * nsm));
        if (lb == 0) {
            CUDA_TRY(cudaMemsetAsync(d.cnt, 0, sizeof(int) * m.nv, st));
        } else {   // tents completed before the window, per vertex
            std::vector<int> done(m.nv, 0);
            for (int64_t i = 0; i < t0; ++i) done[t.vertex[i]]++;
            CUDA_TRY(cudaMemcpyAsync(d.cnt, done.data(), sizeof(int) * m.nv, cudaMemcpyHostToDevice, st));
            CUDA_TRY(cudaStreamSynchronize(st));
        }
        CUDA_TRY(cudaMemsetAsync(d.next, 0, sizeof(unsigned long long), st));
        PArgs pa;
        pa.n_tents = nt;
        pa.ticket0 = t0;
        pa.next = d.next;
        pa.cnt = d.cnt;
        pa.vt_ptr = d.vt_ptr;
        pa.vt_layer = d.vt_layer;
        pa.adj_ptr = d.adj_ptr;
        pa.adj = d.adj;
        pa.tent_layer = d.tent_layer;
        pa.timeout_ns = (m.flags & MTP_FLAG_TEST_STALL) ? 200000000LL : 10000000000LL;   // 0.2 s / 10 s per wait
        pa.n_rhs = m.n_rhs;
        pa.withhold_first = (m.flags & MTP_FLAG_TEST_STALL) ? 1 : 0;
        CUDA_TRY(ke.persistent(a, pa, grid, st));
    } else if (use_graph && full) {
        if (!d.exec || d.graph_state != state) {
            if (d.exec) { cudaGraphExecDestroy(d.exec); d.exec = nullptr; }
            cudaGraph_t g;
            CUDA_TRY(cudaStreamBeginCapture(d.capture, cudaStreamCaptureModeThreadLocal));
            int rc = enqueue_layers(t, a, lb, le, d.capture);
            cudaError_t ce = cudaStreamEndCapture(d.capture, &g);
            if (rc != MTP_OK) return rc;
            CUDA_TRY(ce);
            CUDA_TRY(cudaGraphInstantiate(&d.exec, g, 0));
            cudaGraphDestroy(g);
            d.graph_state = state;
        }
        CUDA_TRY(cudaGraphLaunch(d.exec, st));
    } else {
        MTP_TRY(enqueue_layers(t, a, lb, le, st));
    }
    return check_error_word(t, st);
}

int device_evolve_host(Tents& t, const void* in, void* out, void* stream) {
    MTP_TRY(device_tents_upload(t));
    Mesh& m = *t.mesh;
    DeviceTents& d = *t.dev;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = (size_t)m.n_rhs * m.ne * m.nf * m.nb * real_size(m);
    if (!d.host_state) CUDA_TRY(cudaMalloc(&d.host_state, bytes));
    CUDA_TRY(cudaMemcpyAsync(d.host_state, in, bytes, cudaMemcpyHostToDevice, st));
    MTP_TRY(device_evolve(t, d.host_state, 0, (int64_t)t.layer_ptr.size() - 1, true, stream));
    CUDA_TRY(cudaMemcpyAsync(out, d.host_state, bytes, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return MTP_OK;
}

}  // namespace mtp

namespace mtp {

// Patch tape of one layer: the coefficients of the elements of every tent's patch, tents in
// layer order, each patch's elements in patch order; entry e of the tape holds nc = n_fields
// x n_basis values per right-hand side, tape[rhs][e][nc].  One block per (tent, rhs).
template <typename Real, bool GATHER>
__global__ void patch_tape_kernel(Real* state, Real* tape, const int32_t* tent_v, const int64_t* tent_off,
                                  const int64_t* patch_ptr, const int32_t* patch_elem, int64_t t0, int64_t e0,
                                  int nc, int64_t state_rhs_stride, int64_t tape_rhs_stride) {
    const int64_t t = t0 + blockIdx.x;
    const int V = tent_v[t];
    const int64_t pb = patch_ptr[V], ns = patch_ptr[V + 1] - pb;
    Real* st = state + (int64_t)blockIdx.y * state_rhs_stride;
    Real* tp = tape + (int64_t)blockIdx.y * tape_rhs_stride + (tent_off[t] - e0) * nc;
    for (int64_t i = threadIdx.x; i < ns * nc; i += blockDim.x) {
        const int64_t k = i / nc, r = i - k * nc;
        Real* g = st + (int64_t)patch_elem[pb + k] * nc + r;
        if (GATHER) tp[i] = *g; else *g = tp[i];
    }
}

static int patch_tape(Tents& t, void* state, void* tape, int64_t layer, int64_t e0, int64_t tape_entries,
                      bool gather, cudaStream_t st) {
    Mesh& m = *t.mesh;
    const int64_t t0 = t.layer_ptr[layer], n = t.layer_ptr[layer + 1] - t0;
    if (n == 0) return MTP_OK;
    const int nc = m.nf * m.nb;
    dim3 grid((unsigned)n, m.n_rhs);
    const int64_t srs = m.ne * nc, trs = tape_entries * nc;
    DeviceMesh& dm = *m.dev;
    DeviceTents& d = *t.dev;
    if (m.precision == MTP_FP64) {
        if (gather)
            patch_tape_kernel<double, true><<<grid, 128, 0, st>>>((double*)state, (double*)tape, d.v, d.tent_off,
                                                                  dm.patch_ptr, dm.patch_elem, t0, e0, nc, srs, trs);
        else
            patch_tape_kernel<double, false><<<grid, 128, 0, st>>>((double*)state, (double*)tape, d.v, d.tent_off,
                                                                   dm.patch_ptr, dm.patch_elem, t0, e0, nc, srs, trs);
    } else {
        if (gather)
            patch_tape_kernel<float, true><<<grid, 128, 0, st>>>((float*)state, (float*)tape, d.v, d.tent_off,
                                                                 dm.patch_ptr, dm.patch_elem, t0, e0, nc, srs, trs);
        else
            patch_tape_kernel<float, false><<<grid, 128, 0, st>>>((float*)state, (float*)tape, d.v, d.tent_off,
                                                                  dm.patch_ptr, dm.patch_elem, t0, e0, nc, srs, trs);
    }
    CUDA_TRY(cudaGetLastError());
    return MTP_OK;
}

// Reverse sweep with layer checkpointing: the forward pass keeps the state before every
// K-th layer; each segment is recomputed from its checkpoint, saving before each of its
// layers only the patch elements that layer touches (a compact patch tape), and is then
// reversed layer by layer: the layer's patch tape is scattered into a work state and the
// adjoint tent kernel reads its bottom values there.
int device_adjoint(Tents& t, const void* state0, const void* lamT, void* lam0, double* geps, double* gmu,
                   int64_t K, void* stream) {
    MTP_TRY(device_tents_upload(t));
    Mesh& m = *t.mesh;
    DeviceTents& d = *t.dev;
    cudaStream_t st = (cudaStream_t)stream;
    static AdjEntry general[2][2][5], apex[2][5];
    static std::once_flag once;
    std::call_once(once, [] { adjoint_table(general); apex_adjoint_table(apex); });
    if (m.precision == MTP_FP32_SPLIT || (m.flags & MTP_FLAG_SUBSTITUTED_RK4))
        return set_error(MTP_EUNSUPPORTED, "the adjoint runs SAT meshes in FP64, FP32 or a tensor-core mode");
    const int fp = m.precision == MTP_FP64 ? 0 : 1;   // the tensor-core modes' adjoint runs in FP32
    const bool in_apex = m.dim == 3 && apex[fp][m.p - 1].launch && !m.stretched;
    const AdjEntry& ae = in_apex ? apex[fp][m.p - 1] : general[fp][m.dim - 2][m.p - 1];
    const KernelEntry& ke = kernel_entry(m, item_shape(t));
    size_t smem = 0, smem_f = 0;
    const cudaError_t pa_ = ae.prepare(m.max_patch, &smem);
    const cudaError_t pf_ = ke.prepare(m.max_patch, &smem_f);
    int dev, smem_max;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if ((int64_t)std::max(smem, smem_f) > smem_max)
        return set_error(MTP_EUNSUPPORTED, "adjoint tent kernel needs " + std::to_string(smem) +
                                               " bytes of shared memory per block; the device allows " +
                                               std::to_string(smem_max));
    CUDA_TRY(pa_);
    CUDA_TRY(pf_);
    if (in_apex || apex_runs(m, item_shape(t))) MTP_TRY(apex_upload(m));
    const int64_t nl = (int64_t)t.layer_ptr.size() - 1;
    const size_t sbytes = (size_t)m.n_rhs * m.ne * m.nf * m.nb * real_size(m);
    int64_t max_tents = 0;
    for (int64_t l = 0; l < nl; ++l) max_tents = std::max(max_tents, t.layer_ptr[l + 1] - t.layer_ptr[l]);
    // patch entries before each tent; the largest segment's patch tape
    std::vector<int64_t> off(t.vertex.size() + 1, 0);
    for (size_t i = 0; i < t.vertex.size(); ++i)
        off[i + 1] = off[i] + (m.patch_ptr[t.vertex[i] + 1] - m.patch_ptr[t.vertex[i]]);
    if (!d.tent_off) MTP_TRY(upload(&d.tent_off, off.data(), off.size()));
    const int64_t tstride = ae.tape_stride(m.max_patch, m.m, m.q);
    const size_t tape_bytes = (size_t)max_tents * m.n_rhs * tstride * real_size(m);
    auto align = [](size_t x) { return (x + 255) & ~size_t(255); };
    int64_t nck = 0, seg_entries = 0;   // segments of K layers, patch entries of the largest
    size_t ptape_bytes = 0, need = 0;
    auto plan = [&](int64_t layers) {
        K = std::min(layers, nl);
        nck = (nl + K - 1) / K;
        seg_entries = 0;
        for (int64_t c = 0; c < nck; ++c) {
            const int64_t l0 = c * K, l1 = std::min((c + 1) * K, nl);
            seg_entries = std::max(seg_entries, off[t.layer_ptr[l1]] - off[t.layer_ptr[l0]]);
        }
        ptape_bytes = (size_t)seg_entries * m.n_rhs * m.nf * m.nb * real_size(m);
        need = align((size_t)(nck + 2) * sbytes) + align(ptape_bytes) + tape_bytes + 256;
    };
    auto reserve = [&]() {
        if (d.adj_bytes >= need) return cudaSuccess;
        if (d.adj_buf) cudaFree(d.adj_buf);
        d.adj_buf = nullptr;
        d.adj_bytes = 0;
        const cudaError_t e = cudaMalloc(&d.adj_buf, need);
        if (e == cudaSuccess) d.adj_bytes = need;
        else d.adj_buf = nullptr;
        return e;
    };
    bool reserved = false;
    if (K <= 0) {
        // One segment when the patch tape of the whole evolve stays within kAdjointTape and the buffers take
        // at most half of the free memory (the handle keeps them, and the caller has its own tensors): nothing is
        // computed twice (adjoint workload 8^3, p = 2: 98 MB).  About sqrt(layers) otherwise, which
        // balances checkpoints and tape at the price of a second forward pass.
        constexpr size_t kAdjointTape = (size_t)4 << 30;
        plan(nl);
        size_t free_bytes = 0, total = 0;
        if (d.adj_bytes < need) CUDA_TRY(cudaMemGetInfo(&free_bytes, &total));
        if (ptape_bytes <= kAdjointTape && (d.adj_bytes >= need || need <= (free_bytes + d.adj_bytes) / 2)) {
            reserved = reserve() == cudaSuccess;
            if (!reserved) cudaGetLastError();   // no room after all
        }
        if (!reserved) plan(std::max<int64_t>(1, (int64_t)std::ceil(std::sqrt((double)nl))));
    } else {
        plan(K);
    }
    if (!reserved) CUDA_TRY(reserve());
    if (!d.tau_rev) CUDA_TRY(cudaMalloc((void**)&d.tau_rev, sizeof(double) * m.nv));
    char* base = (char*)d.adj_buf;
    auto ckpt = [&](int64_t c) { return (void*)(base + c * sbytes); };
    void* work = (void*)(base + nck * sbytes);          // the recomputed state
    void* ybot = (void*)(base + (nck + 1) * sbytes);    // bottom values of the layer being reversed
    void* ptape = (void*)(base + align((size_t)(nck + 2) * sbytes));
    void* tape = (void*)(base + align((size_t)(nck + 2) * sbytes) + align(ptape_bytes));

    CUDA_TRY(cudaMemsetAsync(d.err, 0, sizeof(int), st));
    // forward pass with checkpoints
    MTP_TRY(set_front(t, 0, d.tau, st));
    CUDA_TRY(cudaMemcpyAsync(work, state0, sbytes, cudaMemcpyDeviceToDevice, st));
    KArgs fa;
    for (int64_t c = 0; c < nck; ++c) {
        CUDA_TRY(cudaMemcpyAsync(ckpt(c), work, sbytes, cudaMemcpyDeviceToDevice, st));
        if (c + 1 == nck) break;   // the last segment's layers run when it is reversed, the last layer of all
                                   // included: it may be the one that a non-finite value first appears in
        fill_args(t, work, fa, item_shape(t));
        MTP_TRY(enqueue_layers(t, fa, c * K, (c + 1) * K, st));
    }
    // reverse sweep
    CUDA_TRY(cudaMemcpyAsync(lam0, lamT, sbytes, cudaMemcpyDeviceToDevice, st));
    CUDA_TRY(cudaMemsetAsync(geps, 0, sizeof(double) * m.ne, st));
    CUDA_TRY(cudaMemsetAsync(gmu, 0, sizeof(double) * m.ne, st));
    {
        std::vector<double> top(m.nv, t.T);
        CUDA_TRY(cudaMemcpyAsync(d.tau_rev, top.data(), sizeof(double) * m.nv, cudaMemcpyHostToDevice, st));
        CUDA_TRY(cudaStreamSynchronize(st));
    }
    AdjArgs aa;
    for (int64_t c = nck - 1; c >= 0; --c) {
        const int64_t l0 = c * K, l1 = std::min((c + 1) * K, nl);
        const int64_t e0 = off[t.layer_ptr[l0]];
        MTP_TRY(set_front(t, l0, d.tau, st));
        CUDA_TRY(cudaMemcpyAsync(work, ckpt(c), sbytes, cudaMemcpyDeviceToDevice, st));
        fill_args(t, work, fa, item_shape(t));
        for (int64_t l = l0; l < l1; ++l) {
            MTP_TRY(patch_tape(t, work, ptape, l, e0, seg_entries, true, st));
            if (l + 1 < l1 || l1 == nl) MTP_TRY(enqueue_layers(t, fa, l, l + 1, st));
        }
        for (int64_t l = l1 - 1; l >= l0; --l) {
            const int64_t t0 = t.layer_ptr[l], n = t.layer_ptr[l + 1] - t0;
            if (n == 0) continue;
            MTP_TRY(patch_tape(t, ybot, ptape, l, e0, seg_entries, false, st));
            fill_args(t, nullptr, aa.k, 0);
            aa.k.tau = d.tau_rev;
            aa.ybot = ybot;
            aa.lam = lam0;
            aa.geps = geps;
            aa.gmu = gmu;
            aa.tape = tape;
            aa.tape_stride = tstride;
            CUDA_TRY(ae.launch(aa, t0, (int)n, m.n_rhs, st));
        }
    }
    return check_error_word(t, st);
}

}  // namespace mtp

namespace mtp {

struct DeviceBatch {
    int32_t* ticket_inst = nullptr;
    int64_t* ticket_tent = nullptr;
    KArgs* kargs = nullptr;
    PArgs* pargs = nullptr;
    int32_t* inst_p = nullptr;
    unsigned long long* next = nullptr;
    int* err = nullptr;
    int* err_host = nullptr;
};

void device_batch_free(Batch& b) {
    if (!b.dev) return;
    DeviceBatch& d = *b.dev;
    void* ptrs[] = {d.ticket_inst, d.ticket_tent, d.kargs, d.pargs, d.inst_p, d.next, d.err};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (d.err_host) cudaFreeHost(d.err_host);
    delete b.dev;
    b.dev = nullptr;
}

static int batch_buffers(Batch& b) {
    DeviceBatch& d = *b.dev;
    const int64_t ni = (int64_t)b.inst.size();
    MTP_TRY(upload(&d.ticket_inst, b.ticket_inst.data(), b.ticket_inst.size()));
    MTP_TRY(upload(&d.ticket_tent, b.ticket_tent.data(), b.ticket_tent.size()));
    std::vector<int32_t> ps(ni);
    for (int64_t i = 0; i < ni; ++i) ps[i] = b.inst[i]->mesh->p;
    MTP_TRY(upload(&d.inst_p, ps.data(), ps.size()));
    CUDA_TRY(cudaMalloc((void**)&d.kargs, sizeof(KArgs) * ni));
    CUDA_TRY(cudaMalloc((void**)&d.pargs, sizeof(PArgs) * ni));
    CUDA_TRY(cudaMalloc((void**)&d.next, sizeof(unsigned long long)));
    CUDA_TRY(cudaMalloc((void**)&d.err, sizeof(int)));
    CUDA_TRY(cudaMallocHost((void**)&d.err_host, sizeof(int)));
    CUDA_TRY(cudaStreamSynchronize(0));
    return MTP_OK;
}

int device_batch_evolve(Batch& b, void* const* states, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t ni = (int64_t)b.inst.size();
    for (Tents* t : b.inst) MTP_TRY(device_tents_upload(*t));
    const Mesh& m0 = *b.inst[0]->mesh;
    static BatchEntry general[2][2];
    static std::once_flag once;
    std::call_once(once, [] { batch_table(general); });
    for (Tents* t : b.inst)
        if (t->mesh->flags & MTP_FLAG_SUBSTITUTED_RK4)
            return set_error(MTP_EUNSUPPORTED, "batches run SAT meshes; MTP_FLAG_SUBSTITUTED_RK4 is per mesh");
    if (m0.precision == MTP_TF32 || m0.precision == MTP_TF32X3 || m0.precision == MTP_FP32_SPLIT)
        return set_error(MTP_EUNSUPPORTED, "batches run FP64 or FP32 SIMT meshes; tensor-core and split modes are per mesh");
    int dev, smem_max;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const bool f64 = m0.precision == MTP_FP64;
    auto smem_of = [&](const BatchEntry& e) {
        size_t n = 0;
        for (Tents* t : b.inst) n = std::max(n, e.smem_bytes(t->mesh->p, t->mesh->max_patch));
        return n;
    };
    int pmax = 0;
    bool stretched = false;
    for (Tents* t : b.inst) {
        pmax = std::max(pmax, t->mesh->p);
        stretched |= t->mesh->stretched;
    }
    BatchEntry be = general[f64 ? 0 : 1][m0.dim - 2];
    if ((m0.dim == 2 || pmax <= kApexMaxDegree) && (!stretched || (int64_t)smem_of(be) > smem_max)) {   // see apex_runs
        for (Tents* t : b.inst) MTP_TRY(apex_upload(*t->mesh));
        be = m0.dim == 2 ? (f64 ? apex2_batch_f64() : apex2_batch_f32()) : (f64 ? apex_batch_f64(pmax) : apex_batch_f32(pmax));
    }
    const size_t smem = smem_of(be);
    if (!b.dev) {
        b.dev = new DeviceBatch();
        const int rc = batch_buffers(b);
        if (rc != MTP_OK) {
            device_batch_free(b);
            cudaGetLastError();
            return rc;
        }
    }
    DeviceBatch& d = *b.dev;
    std::vector<KArgs> ka(ni);
    std::vector<PArgs> pa(ni);
    for (int64_t i = 0; i < ni; ++i) {
        Tents& t = *b.inst[i];
        Mesh& m = *t.mesh;
        fill_args(t, states[i], ka[i], 0);
        ka[i].err = d.err;
        DeviceTents& dt = *t.dev;
        pa[i].n_tents = (int64_t)t.vertex.size();
        pa[i].ticket0 = 0;
        pa[i].next = nullptr;
        pa[i].cnt = dt.cnt;
        pa[i].vt_ptr = dt.vt_ptr;
        pa[i].vt_layer = dt.vt_layer;
        pa[i].adj_ptr = dt.adj_ptr;
        pa[i].adj = dt.adj;
        pa[i].tent_layer = dt.tent_layer;
        pa[i].timeout_ns = 10000000000LL;
        pa[i].n_rhs = m.n_rhs;
        pa[i].withhold_first = 0;
        CUDA_TRY(cudaMemsetAsync(dt.tau, 0, sizeof(double) * m.nv, st));   // flat front t = 0
        CUDA_TRY(cudaMemsetAsync(dt.cnt, 0, sizeof(int) * m.nv, st));
    }
    int bpsm = 0, nsm = 0;
    if ((int64_t)smem > smem_max)
        return set_error(MTP_EUNSUPPORTED, "batch kernel needs " + std::to_string(smem) +
                                               " bytes of shared memory per block; the device allows " +
                                               std::to_string(smem_max));
    CUDA_TRY(be.prepare(smem, &bpsm));
    CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(cudaMemcpyAsync(d.kargs, ka.data(), sizeof(KArgs) * ni, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemcpyAsync(d.pargs, pa.data(), sizeof(PArgs) * ni, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemsetAsync(d.next, 0, sizeof(unsigned long long), st));
    CUDA_TRY(cudaMemsetAsync(d.err, 0, sizeof(int), st));
    BatchArgs ba;
    ba.n_tickets = (int64_t)b.ticket_inst.size();
    ba.next = d.next;
    ba.ticket_inst = d.ticket_inst;
    ba.ticket_tent = d.ticket_tent;
    ba.kargs = d.kargs;
    ba.pargs = d.pargs;
    ba.inst_p = d.inst_p;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ba.n_tickets, (int64_t)std::max(1, bpsm) * nsm));
    CUDA_TRY(be.launch(ba, grid, smem, st));
    CUDA_TRY(cudaMemcpyAsync(d.err_host, d.err, sizeof(int), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));     // also keeps ka / pa alive until copied
    if (*d.err_host == 1) return set_error(MTP_ECAUSAL, "a tent violated |grad phi| < sqrt(eps mu)");
    if (*d.err_host == 2) return set_error(MTP_ENUMERIC, "non-finite value in the evolved state");
    if (*d.err_host == 3) return set_error(MTP_ETIMEOUT, "a tent's wait for its predecessors exceeded the limit");
    if (*d.err_host != 0) return set_error(MTP_ECUDA, "unknown device error word");
    return MTP_OK;
}

}  // namespace mtp

namespace mtp {

// Times the three evolve launch configurations on layers [lb, le) of `state` (overwritten) and
// keeps the fastest in the tents handle.
int device_autotune(Tents& t, void* state, int64_t lb, int64_t le, int* best, double* ms_out, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0, e1;
    CUDA_TRY(cudaEventCreate(&e0));
    CUDA_TRY(cudaEventCreate(&e1));
    double best_ms = 1e300;
    int best_c = 0;
    for (int c = 0; c < 3; ++c) {
        t.launch = c;
        MTP_TRY(device_evolve(t, state, lb, le, false, stream));          // warm-up
        CUDA_TRY(cudaEventRecord(e0, st));
        MTP_TRY(device_evolve(t, state, lb, le, false, stream));
        CUDA_TRY(cudaEventRecord(e1, st));
        CUDA_TRY(cudaEventSynchronize(e1));
        float ms = 0;
        CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
        if (ms_out) ms_out[c] = ms;
        if (ms < best_ms) { best_ms = ms; best_c = c; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    t.launch = best_c;
    if (best) *best = best_c;
    return MTP_OK;
}

}  // namespace mtp
