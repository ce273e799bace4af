// Apex tent kernel: SAT evolution of one 3D tent (FP64 or FP32 arithmetic, p = 1..4) in a frame
// that is adapted to the tent vertex V.
//
// Basis.  Each patch element is re-expressed in the Dubiner basis whose collapsed apex is V, an
// orthogonal change of basis that is block-diagonal in the degree (table Rt, one matrix per local
// index of V).  In it multiplication by lambda_V couples at most three functions, and the
// derivative, trace and lift tables are the same for all elements and mostly zero; ApexOps<P>
// (generated at build time) holds them as straight-line code with literal entries.
//
// Frame.  With t_0, t_1, t_2 the edges from V to the element's other vertices (ascending ids,
// scaled by a power of two l ~ |det|^(1/3)) U is kept in covariant components E . t_X and Y in
// contravariant ones (y = sum_W t_W y^W).  Then the mapped curl needs no geometry,
//   Y_E^W = -k (S_X h_Z - S_Z h_X),  Y_H^W = +k (S_X e_Z - S_Z e_X),  (X, Z, W) cyclic,
// with k = dt / (l det), a facet needs only its two tangential components of E and H, the product
// M' U is (M'U)_f^W = s k (u_Z - u_X) (s = -1 for E, +1 for H, u of the other field), and with the
// coefficients scaled by l / sqrt|det| the traces and lifts carry no factor at all.
// With acc = Y_n / (s k), the stage recursion (Sec. 4, recursion-init) becomes
//   r_n = acc - n (u_Z - u_X),  U_n = K r_n,  delta += taylor_n acc,
// K = (closed-form G^-1 in these frames) x (s k), and a sub-interval starts from r = y0 + delta.
// The increment delta is summed from zero and added once to the state that was read, so the Taylor
// sum rounds at the size of the increment.
//
// Threads.  One CTA of 192 threads per tent: warp (field, component), lane = patch element
// (patches have at most 32 elements), so a shared-memory vector access is conflict-free.  Per
// stage, with a barrier after each: traces of the own column | facet fluxes, once per facet |
// volume term + lift -> r | U = K r, one thread per (element, vector of coefficients).  All six
// warps run one instruction stream: the component only selects columns and signs.  That keeps a
// stage of p = 4 within the 32 KB up to which straight-line code issues at full rate (measured:
// 118 of 128 multiply-adds a clock and SM up to 31 KB, 60 .. 80 beyond 46 KB); a first form with
// its own code for each component was bound by instruction fetches (30 % of the issue slots).
//
// Measured against the general kernel on a GB300, one slab: graded 32^3, p = 4, FP32, 463 -> 137 ms
// (5.2k instead of 17.3k clocks per tent and stage; 52 % of the issue slots, then waits at the
// barriers); 16^3 cavity, p = 3, FP32, 333 -> 87 ms; 8^3 cavity, p = 3, FP64, 560 -> 259 ms (FP64
// issue); 13^3, p = 2, FP32 35.7 -> 9.5 ms.  Error against 64 bits of the first two: 3.8e-7 -> 1.3e-7, 1.9e-6 -> 5.4e-7;
// it grows with the stretch of the elements, and beyond kMaxStretch the general kernel runs.
#pragma once

#include "mtp_apex_ops.h"
#include "mtp_kernels.cuh"

namespace mtp {

// Record of one patch entry (vertex, element) in the state's arithmetic precision, built once per
// mesh by apex_record_kernel in FP64.  [0..5] metric t_X . t_Z (00 01 02 11 12 22), [6..11] its
// inverse, [12] 1 / l, [13] eps, [14] mu, [15] det of the scaled edges, [16] k / dt = 1 / (l det),
// [17] scale of y0 times dt, [18] scale of the increment over dt, [19] 1 / (eps mu), then for the facet
// opposite each other vertex [20 + 6 fi] a, b, q (xx, xy, yy), zz (see phase_fluxes);
// [38..46] dual vectors, [47..55] edges.
constexpr int kApexRec = 56, kApexConst = 38, kApexFacet = 20, kApexDual = 38, kApexEdge = 47;

template <typename Real, int P>
struct ApexShape {
    static constexpr int NB = dim_pk(3, P), NFB = dim_pk(2, P), NM = dim_pk(3, P - 1);
    static constexpr int VW = 16 / (int)sizeof(Real);            // values per 16-byte vector
    static constexpr int GB = (NB + VW - 1) / VW, GF = (NFB + VW - 1) / VW;
    static constexpr int NT = 192;
    static constexpr int SP = (6 * NB) | 1;                      // odd row stride of the staging buffer
    static constexpr int CS = 33;                                // lane stride of the element constants
    static constexpr int COL = 32 * VW;                          // one vector row of all lanes
    static constexpr size_t TR = 0;
    static constexpr size_t U = TR + (size_t)12 * GF * COL * sizeof(Real);
    static constexpr size_t R = U + (size_t)6 * GB * COL * sizeof(Real);
    static constexpr size_t Y0 = R + (size_t)6 * GB * COL * sizeof(Real);
    static constexpr size_t C = Y0 + (size_t)6 * GB * COL * sizeof(Real);
    static constexpr size_t I = C + (size_t)(kApexConst + 3) * CS * sizeof(Real);
    static constexpr size_t T = (I + (32 * 4 + 96 + 4) * sizeof(int) + 15) / 16 * 16;
    static constexpr size_t H = (T + (size_t)(kMaxSub + 1 + kMaxTaylor) * sizeof(Real) + 7) / 8 * 8;   // ApexHead
    static constexpr size_t BYTES = H + 32;
    static constexpr size_t CHECK = R - 6 * 32 * sizeof(double);   // causality partial sums, end of the U buffer
    static_assert((size_t)32 * SP * sizeof(Real) <= CHECK, "the staging buffer shares the trace and U buffers");
    static_assert(BYTES <= 227 * 1024, "one tent per CTA");
    // CTAs per SM that the register budget is shaped for
    static constexpr int MINB = sizeof(Real) == 8 ? 1 : (P >= 3 ? 2 : 3);
    // FP64 issues one instruction in 19 clocks and SM, so there every component has its own code
    // with the fewest operations; FP32 shares one stream (see above)
    static constexpr bool OWN = sizeof(Real) == 8;
};

// Row offsets of the basis-change table: rows of one degree block are padded to 4 entries.
__host__ __device__ constexpr int apex_rot_block(int d) { return (d + 1) * (d + 2) / 2; }
__host__ __device__ constexpr int apex_rot_offset(int d) {
    int o = 0;
    for (int k = 0; k < d; ++k) o += apex_rot_block(k) * pad4(apex_rot_block(k));
    return o;
}

// scalars of the CTA's tent
struct ApexHead {
    double tb, tt;
    const void* ent;
    int ns, nown;
};
static_assert(sizeof(ApexHead) == 32, "shared-memory slot");

__device__ __forceinline__ unsigned char* apex_smem() {
    extern __shared__ __align__(16) unsigned char smem[];
    return smem;
}

template <int N, typename Real>
__device__ __forceinline__ void apex_load(const Real* base, int lane, Real* out) {
    using VT = typename Vec<Real>::T;
    constexpr int W = Vec<Real>::W, G = (N + W - 1) / W;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        Real v[W];
        Vec<Real>::get(*(const VT*)(base + (g * 32 + lane) * W), v);
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (g * W + k < N) out[g * W + k] = v[k];
    }
}
__device__ __forceinline__ float4 apex_pack(const float* v) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ double2 apex_pack(const double* v) { return make_double2(v[0], v[1]); }
template <int N, typename Real>
__device__ __forceinline__ void apex_store(Real* base, int lane, const Real* in) {
    using VT = typename Vec<Real>::T;
    constexpr int W = Vec<Real>::W, G = (N + W - 1) / W;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        Real v[W];
#pragma unroll
        for (int k = 0; k < W; ++k) v[k] = g * W + k < N ? in[g * W + k] : Real(0);
        *(VT*)(base + (g * 32 + lane) * W) = apex_pack(v);
    }
}

template <typename Real, int P>
struct ApexTent {
    using Sh = ApexShape<Real, P>;
    using Op = ApexOps<P>;
    static constexpr int NB = Sh::NB, NFB = Sh::NFB, NM = Sh::NM, COL = Sh::COL, CS = Sh::CS;
    int lane, warp, f, w;   // field (0: E, 1: H) and component of this warp

    __device__ __forceinline__ ApexTent() {
        lane = threadIdx.x & 31;
        warp = threadIdx.x >> 5;
        f = warp / 3;
        w = warp - 3 * f;
    }
    // shared memory at fixed offsets: no base pointers in registers
    static __device__ __forceinline__ Real* sTr() { return (Real*)(apex_smem() + Sh::TR); }
    static __device__ __forceinline__ Real* sU() { return (Real*)(apex_smem() + Sh::U); }
    static __device__ __forceinline__ Real* sR() { return (Real*)(apex_smem() + Sh::R); }
    static __device__ __forceinline__ Real* sY0() { return (Real*)(apex_smem() + Sh::Y0); }
    static __device__ __forceinline__ Real* sC() { return (Real*)(apex_smem() + Sh::C); }
    static __device__ __forceinline__ Real* sG() { return sC() + kApexConst * CS; }
    static __device__ __forceinline__ int* sElem() { return (int*)(apex_smem() + Sh::I); }
    static __device__ __forceinline__ int* sInfo() { return sElem() + 32; }   // three words per element
    static __device__ __forceinline__ int* sOwn() { return sInfo() + 96; }
    static __device__ __forceinline__ Real* sSub() { return (Real*)(apex_smem() + Sh::T); }
    static __device__ __forceinline__ Real* sTay() { return sSub() + kMaxSub + 1; }
    static __device__ __forceinline__ ApexHead* head() { return (ApexHead*)(apex_smem() + Sh::H); }
    __device__ __forceinline__ Real cst(int word, int k) const { return sC()[word * CS + k]; }
    __device__ __forceinline__ Real* tr(int fi, int fs) const { return sTr() + (fi * 4 + fs) * Sh::GF * COL; }
    __device__ __forceinline__ Real* ucol(int c) const { return sU() + c * Sh::GB * COL; }
    __device__ __forceinline__ Real* rcol(int c) const { return sR() + c * Sh::GB * COL; }

    // Facet traces of the own component on the two facets through V that contain its edge.  The
    // facets opposite D and C take the sum and the difference of the even and odd parts: component
    // C lies on the first, D on the second, B on both; C and D also lie on the facet opposite B.
    template <int WT>
    __device__ __forceinline__ void phase_traces() {
        Real u[NB];
        apex_load<NB>(ucol(3 * f + (WT < 0 ? w : WT)), lane, u);
        traces_of<WT, false>(u, sTr());
    }
    // LAM: the traces times lambda_V (used by the adjoint)
    template <int WT, bool LAM>
    __device__ __forceinline__ void traces_of(const Real* u, Real* buf) {
        constexpr int NS = Op::NS;
        const int W = WT < 0 ? w : WT;
        auto put = [&](int fi, int fs, const Real* t) {
            Real* to = buf + (fi * 4 + fs) * Sh::GF * COL;
            if constexpr (LAM) {
                Real g[NFB];
                Op::lam(t, g);
                apex_store<NFB>(to, lane, g);
            } else {
                apex_store<NFB>(to, lane, t);
            }
        };
        {
            Real e[NS], o[NS];
            Op::pair_even(u, e);
            Op::pair_odd(u, o);
            auto facet = [&](int fi) {
                Real s[NS], t[NFB];
#pragma unroll
                for (int q = 0; q < NS; ++q) s[q] = WT < 0 ? e[q] + (fi ? Real(1) : Real(-1)) * o[q] : fi ? e[q] + o[q] : e[q] - o[q];
                Op::pair_trace(s, t);
                put(fi, 2 * f + (W == 2 ? 1 : 0), t);
            };
            if constexpr (WT >= 0) {
                if (W != 0) facet(0);
                if (W != 1) facet(1);
            } else {
                int fi = W == 0 ? 1 : 0;
#pragma unroll 1
                while (true) {
                    facet(fi);
                    if (W != 2 || fi == 1) break;
                    fi = 1;
                }
            }
        }
        if (W != 2) {
            Real t[NFB];
            Op::trace2(u, t);
            put(2, 2 * f + W, t);
        }
    }

    // Upwind flux (impedance form, PEC as mirror state) once per facet on tangential components:
    // with J(x, y) = (y, -x) and Q the facet's adjugate metric / area,
    //   E: r J(a H- + b H+) + q (E- - E+),   H: r J(b E- + a E+) - zz q (H- - H+),
    // a = Z- / (Z- + Z+), b = Z+ / (Z- + Z+), q = sgn Q / (Z- + Z+), zz = Z- Z+; the neighbour
    // takes +- the same values.  One thread per (facet, vector of modes), in place.
    __device__ __forceinline__ void phase_fluxes(int nown, float inv_nown) {
        using VT = typename Vec<Real>::T;
        constexpr int VW = Sh::VW;
        for (int idx = threadIdx.x; idx < nown * Sh::GF; idx += Sh::NT) {
            const int g = (int)(((float)idx + 0.5f) * inv_nown);
            const int pk = sOwn()[idx - g * nown];
            const int k = pk & 31, k2 = (pk >> 5) & 31, fi = (pk >> 10) & 3, fi2 = (pk >> 12) & 3;
            const bool wall = pk & (1 << 14);
            const Real tau = (pk & (1 << 15)) ? Real(-1) : Real(1);
            const Real r = fi == 1 ? Real(1) : Real(-1);
            Real* mine = sTr() + (fi * 4 * Sh::GF + g) * COL + k * VW;
            Real* other = sTr() + (fi2 * 4 * Sh::GF + g) * COL + k2 * VW;
            const int c0 = kApexFacet + 6 * fi;
            const Real a = cst(c0, k), b = cst(c0 + 1, k), qxx = cst(c0 + 2, k), qxy = cst(c0 + 3, k),
                       qyy = cst(c0 + 4, k), zz = cst(c0 + 5, k);
            const Real ra = r * a, rb = r * b;
            Real m[4][VW], o[4][VW];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                Vec<Real>::get(*(const VT*)(mine + s * Sh::GF * COL), m[s]);
                Vec<Real>::get(*(const VT*)(other + s * Sh::GF * COL), o[s]);
            }
            if (wall)
#pragma unroll
                for (int v = 0; v < VW; ++v) {
                    o[0][v] = -m[0][v];
                    o[1][v] = -m[1][v];
                    o[2][v] = m[2][v];
                    o[3][v] = m[3][v];
                }
            Real y[4][VW];
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                const Real ex = m[0][v] - o[0][v], ey = m[1][v] - o[1][v];
                const Real hx = zz * (m[2][v] - o[2][v]), hy = zz * (m[3][v] - o[3][v]);
                y[0][v] = ra * m[3][v] + rb * o[3][v] + (qxx * ex + qxy * ey);
                y[1][v] = -(ra * m[2][v] + rb * o[2][v]) + (qxy * ex + qyy * ey);
                y[2][v] = rb * m[1][v] + ra * o[1][v] - (qxx * hx + qxy * hy);
                y[3][v] = -(rb * m[0][v] + ra * o[0][v]) - (qxy * hx + qyy * hy);
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) *(VT*)(mine + s * Sh::GF * COL) = apex_pack(y[s]);
            if (!wall) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
#pragma unroll
                    for (int v = 0; v < VW; ++v) y[s][v] *= tau;
                    *(VT*)(other + s * Sh::GF * COL) = apex_pack(y[s]);
                }
            }
        }
    }

    // acc = lift of the own component's facet fluxes
    template <int WT>
    __device__ __forceinline__ void phase_lift(Real* acc) {
        constexpr int NS = Op::NS;
        const int W = WT < 0 ? w : WT;
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[b] = Real(0);
        {
            Real e[NS], o[NS];
            auto facet = [&](int fi, Real* s) {
                Real F[NFB], G[NFB];
                apex_load<NFB>(tr(fi, 2 * f + (W == 2 ? 1 : 0)), lane, F);
                Op::lam(F, G);
                Op::pair_lift(G, s);
            };
            if constexpr (WT >= 0) {
                facet(W == 1 ? 0 : 1, e);
                if constexpr (WT == 2) facet(0, o);
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    const Real x = e[q], y = WT == 2 ? o[q] : Real(0);
                    e[q] = WT == 2 ? x + y : x;
                    o[q] = WT == 2 ? x - y : WT == 1 ? -x : x;
                }
            } else {
#pragma unroll
                for (int q = 0; q < NS; ++q) e[q] = o[q] = Real(0);
                int fi = W == 0 ? 1 : 0;
#pragma unroll 1
                while (true) {
                    Real s[NS];
                    facet(fi, s);
                    const Real sg = fi ? Real(1) : Real(-1);
#pragma unroll
                    for (int q = 0; q < NS; ++q) {
                        e[q] += s[q];
                        o[q] += sg * s[q];
                    }
                    if (W != 2 || fi == 1) break;
                    fi = 1;
                }
            }
            Op::pair_even_t(e, acc);
            Op::pair_odd_t(o, acc);
        }
        if (W != 2) {
            Real F[NFB], G[NFB];
            apex_load<NFB>(tr(2, 2 * f + W), lane, F);
            Op::lam(F, G);
            Op::lift2(G, acc);
        }
    }

    // acc += volume term of the own component W, d_X w_Z - d_Z w_X with w = lambda_V u of the other
    // field and (X, Z, W) cyclic, and x = u_Z - u_X (M' U).  The derivatives along two edges from V
    // are rewritten along B - A, B - m and D - C (m the middle of C and D), whose tables are sparse:
    //   W = C:  d_BA (w_B - w_D) - d_Bm w_B + d_DC w_B / 2
    //   W = D:  d_BA (w_C - w_B) + d_Bm w_B + d_DC w_B / 2
    //   W = B:  d_BA (w_D - w_C) - d_Bm (w_D - w_C) - d_DC (w_C + w_D) / 2
    // so the first argument is lambda_V x for all three.
    template <int WT>
    __device__ __forceinline__ void phase_volume(Real* acc, Real* x) {
        const int W = WT < 0 ? w : WT;
        Real p[NM], y[NM], s[NM];
        {
            Real uz[NB], v[NB];
            apex_load<NB>(ucol(3 * (1 - f) + (W == 0 ? 2 : W - 1)), lane, uz);
            apex_load<NB>(ucol(3 * (1 - f) + (W == 2 ? 0 : W + 1)), lane, x);
            const Real cz = W == 1 ? Real(0) : Real(1), cx = W == 0 ? Real(0) : Real(1);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                v[b] = WT < 0 ? cz * uz[b] + cx * x[b] : WT == 0 ? uz[b] : WT == 1 ? x[b] : uz[b] + x[b];
                x[b] = uz[b] - x[b];
            }
            Op::mass(v, y);
        }
        Op::mass(x, p);
        const Real cd = W == 2 ? Real(-0.5) : Real(0.5), my = W == 0 ? Real(-1) : W == 1 ? Real(1) : Real(0),
                   mp = W == 2 ? Real(-1) : Real(0);
#pragma unroll
        for (int c = 0; c < NM; ++c) {
            s[c] = WT < 0 ? my * y[c] + mp * p[c] : WT == 0 ? -y[c] : WT == 1 ? y[c] : -p[c];
            y[c] *= cd;
        }
        Op::vol_cd(y, acc);
        Op::vol_mb(s, acc);
        Op::vol_ab(p, acc);
    }

    // K at t^ = th in the frames: with g the covariant and gu the contravariant components of
    // grad phi, s = k / (eps mu - |g|^2) and M = metric - g g^T / (eps mu) (closed-form G^-1, Sec. 4),
    //   u_E = -s mu M r_E + c (gu x r_H),  u_H = s eps M r_H + c (gu x r_E),  c = -s det.
    struct Mass {
        Real m[6], c[3], dE, dH;
    };
    __device__ __forceinline__ Mass mass_at(Real dt, Real th) const {
        Mass K;
        const Real tl = th * dt * cst(12, lane);
        Real g[3], gu[3], gg = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) g[q] = sG()[q * CS + lane] - tl;
        constexpr int sym[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            gu[q] = cst(6 + sym[q][0], lane) * g[0] + cst(6 + sym[q][1], lane) * g[1] + cst(6 + sym[q][2], lane) * g[2];
            gg += gu[q] * g[q];
        }
        const Real eps = cst(13, lane), mu = cst(14, lane), iem = cst(19, lane);
        const Real s = dt * cst(16, lane) / (eps * mu - gg), c = -s * cst(15, lane);
        K.dE = -s * mu;
        K.dH = s * eps;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            K.c[q] = c * gu[q];
#pragma unroll
            for (int r = q; r < 3; ++r) K.m[sym[q][r]] = cst(sym[q][r], lane) - g[q] * g[r] * iem;
        }
        return K;
    }

    // U = K r for the vectors of coefficients of this warp (TAPE: also into a tape slot)
    template <bool TAPE = false>
    __device__ __forceinline__ void phase_solve(const Mass& K, Real* tape = nullptr) {
        using VT = typename Vec<Real>::T;
        constexpr int VW = Sh::VW;
#pragma unroll 1
        for (int g = warp; g < Sh::GB; g += 6) {
            Real r[6][VW];
#pragma unroll
            for (int c = 0; c < 6; ++c) Vec<Real>::get(*(const VT*)(rcol(c) + (g * 32 + lane) * VW), r[c]);
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                Real e[3], h[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    e[q] = K.dE * r[q][v];
                    h[q] = K.dH * r[3 + q][v];
                }
                const Real e0 = r[0][v], e1 = r[1][v], e2 = r[2][v], h0 = r[3][v], h1 = r[4][v], h2 = r[5][v];
                r[0][v] = K.m[0] * e[0] + K.m[1] * e[1] + K.m[2] * e[2] + (K.c[1] * h2 - K.c[2] * h1);
                r[1][v] = K.m[1] * e[0] + K.m[3] * e[1] + K.m[4] * e[2] + (K.c[2] * h0 - K.c[0] * h2);
                r[2][v] = K.m[2] * e[0] + K.m[4] * e[1] + K.m[5] * e[2] + (K.c[0] * h1 - K.c[1] * h0);
                r[3][v] = K.m[0] * h[0] + K.m[1] * h[1] + K.m[2] * h[2] + (K.c[1] * e2 - K.c[2] * e1);
                r[4][v] = K.m[1] * h[0] + K.m[3] * h[1] + K.m[4] * h[2] + (K.c[2] * e0 - K.c[0] * e2);
                r[5][v] = K.m[2] * h[0] + K.m[4] * h[1] + K.m[5] * h[2] + (K.c[0] * e1 - K.c[1] * e0);
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                *(VT*)(ucol(c) + (g * 32 + lane) * VW) = apex_pack(r[c]);
                if constexpr (TAPE) *(VT*)(tape + (c * Sh::GB + g) * COL + lane * VW) = apex_pack(r[c]);
            }
        }
    }

    // y (library basis) -> rotated basis (ROT) or back; the table row depends on the lane's local
    // index of V, so it is read from the L1-resident table
    template <bool ROT>
    __device__ __forceinline__ void rotate(const Real* Rt, const Real* y, Real* z) {
        using VT = typename Vec<Real>::T;
        constexpr int VW = Sh::VW;
#pragma unroll
        for (int d = 0; d <= P; ++d) {
            const int n = apex_rot_block(d), b0 = dim_pk(3, d - 1), st = pad4(n), off = apex_rot_offset(d);
            if (!ROT)
#pragma unroll
                for (int b = 0; b < n; ++b) z[b0 + b] = Real(0);
#pragma unroll
            for (int r = 0; r < n; ++r) {
                Real acc = 0;
#pragma unroll
                for (int c = 0; c < n; c += VW) {
                    Real t[VW];
                    Vec<Real>::get(__ldg((const VT*)(Rt + off + r * st + c)), t);
#pragma unroll
                    for (int v = 0; v < VW; ++v)
                        if (c + v < n) {
                            if (ROT) acc += t[v] * y[b0 + c + v];
                            else z[b0 + c + v] += t[v] * y[b0 + r];
                        }
                }
                if (ROT) z[b0 + r] = acc;
            }
        }
    }

    template <typename F>
    __device__ __forceinline__ void by_component(F fn) {
        if constexpr (Sh::OWN) {
            if (w == 0) fn(std::integral_constant<int, 0>{});
            else if (w == 1) fn(std::integral_constant<int, 1>{});
            else fn(std::integral_constant<int, 2>{});
        } else {
            fn(std::integral_constant<int, -1>{});
        }
    }

    // What does not depend on the state or the front: may run before the tent's predecessors are
    // done.  Ends without a barrier; run() starts with one.
    __device__ void load_static(const KArgs& a, int64_t tent) {
        const int V = a.tent_v[tent];
        const int64_t pb = a.patch_ptr[V];
        const int ns = (int)(a.patch_ptr[V + 1] - pb);
        const Real* ent = (const Real*)a.ent + pb * kApexRec;
        const int k = lane < ns ? lane : ns - 1;      // idle lanes shadow the last element
        if (threadIdx.x == 0) {
            head()->tb = a.tent_tb[tent];
            head()->tt = a.tent_tt[tent];
            head()->ent = ent;
            head()->ns = ns;
        }
        if (warp == 0) {
            sElem()[lane] = a.patch_elem[pb + k];
            const int* info = (const int*)(a.patch_info + (pb + k) * 12);
#pragma unroll
            for (int q = 0; q < 3; ++q) sInfo()[3 * lane + q] = info[q];
        }
        for (int idx = threadIdx.x; idx < ns * kApexConst; idx += Sh::NT) {
            const int e = idx / kApexConst, r = idx - e * kApexConst;
            sC()[r * CS + e] = __ldg(ent + e * kApexRec + r);
        }
        for (int idx = threadIdx.x; idx <= kMaxSub; idx += Sh::NT) {
            sSub()[idx] = (Real)a.tsub[idx];
            if (idx < kMaxTaylor) sTay()[idx] = (Real)a.taylor[idx];
        }
        __syncthreads();
        if (f == 0) {   // owned facets (boundary facets and the lower slot of interior ones), facet by facet
            const int8_t* inf = (const int8_t*)(sInfo() + 3 * k);
            const int j = inf[0];
            unsigned own[3];
            int mine = 0;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int s2 = inf[4 + (q < j ? q : q + 1)];
                own[q] = __ballot_sync(0xffffffffu, lane < ns && (s2 < 0 || s2 > lane));
                if (q == w) mine = s2;
            }
            const int at = (w > 0 ? __popc(own[0]) : 0) + (w > 1 ? __popc(own[1]) : 0);
            const unsigned ow = w == 0 ? own[0] : w == 1 ? own[1] : own[2];
            if (ow >> lane & 1) {
                const int s2 = mine < 0 ? lane : mine;
                int fi2 = w, neg = 0;
                if (mine >= 0) {
                    const int f2 = inf[8 + (w < j ? w : w + 1)], j2 = *(const int8_t*)(sInfo() + 3 * s2);
                    fi2 = f2 - (f2 > j2 ? 1 : 0);
                    neg = (cst(15, k) > Real(0)) == (cst(15, s2) > Real(0));
                }
                sOwn()[at + __popc(ow & ((1u << lane) - 1))] =
                    lane | s2 << 5 | w << 10 | fi2 << 12 | (mine < 0 ? 1 << 14 : 0) | (neg ? 1 << 15 : 0);
            }
            if (threadIdx.x == 0) head()->nown = __popc(own[0]) + __popc(own[1]) + __popc(own[2]);
        }
    }

    // height of the tent; one of almost no height changes nothing: keep 1 / dt finite
    __device__ __forceinline__ Real height() const {
        return (Real)fmax(head()->tt - head()->tb, sizeof(Real) == 4 ? 1e-30 : 1e-200);
    }

    // patch coefficients (library layout) into the staging buffer
    template <bool CG>
    __device__ __forceinline__ void stage_patch(const Real* state) {
        constexpr int NC = 6 * NB, STEP = 8;   // loads in flight
        const int ns = head()->ns;
        for (int i0 = threadIdx.x; i0 < ns * NC; i0 += STEP * Sh::NT) {
            Real v[STEP];
#pragma unroll
            for (int q = 0; q < STEP; ++q) {
                const int idx = i0 + q * Sh::NT, e = idx / NC, r = idx - e * NC;
                if (idx < ns * NC) {
                    const Real* sp = state + (int64_t)sElem()[e] * NC + r;
                    v[q] = CG ? __ldcg(sp) : *sp;
                }
            }
#pragma unroll
            for (int q = 0; q < STEP; ++q) {
                const int idx = i0 + q * Sh::NT, e = idx / NC, r = idx - e * NC;
                if (idx < ns * NC) sTr()[e * Sh::SP + r] = v[q];
            }
        }
    }
    // own component of the staged patch along the record's vectors at `vec`, in the apex basis
    __device__ __forceinline__ void component_in(const KArgs& a, int vec, Real sc, Real* z) {
        const int ns = head()->ns, k = lane < ns ? lane : ns - 1, j = *(const int8_t*)(sInfo() + 3 * k);
        const Real* rec = (const Real*)head()->ent + k * kApexRec + vec + 3 * w;
        const Real g0 = __ldg(rec), g1 = __ldg(rec + 1), g2 = __ldg(rec + 2);
        const Real* st = sTr() + k * Sh::SP + f * 3 * NB;
        Real y[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) y[b] = g0 * st[b] + g1 * st[NB + b] + g2 * st[2 * NB + b];
        rotate<true>((const Real*)a.Rt + (size_t)j * apex_rot_offset(P + 1), y, z);
#pragma unroll
        for (int b = 0; b < NB; ++b) z[b] *= sc;
    }

    // The tent for one right-hand side: read the patch, evolve bottom to top, write the patch.
    // CG: other CTAs of the same launch write the state and the front (bypass L1).
    template <bool CG>
    __device__ void run(const KArgs& a, Real* state) {
        begin<CG>(a, state);
        Real dl[NB];
        stages<false>(a, dl, nullptr);
        finish<CG>(a, state, dl, kApexEdge, (f ? Real(1) : Real(-1)) * height() * cst(18, lane));
    }

    // read the patch and the front; y0 into its buffer and r
    template <bool CG>
    __device__ __forceinline__ void begin(const KArgs& a, const Real* state) {
        __syncthreads();
        const double tb = head()->tb, dtd = head()->tt - tb;
        const int ns = head()->ns, k = lane < ns ? lane : ns - 1, j = *(const int8_t*)(sInfo() + 3 * k);
        stage_patch<CG>(state);
        double* chk = (double*)((unsigned char*)sTr() + Sh::CHECK);
        const int32_t* verts = a.elems + (int64_t)sElem()[lane] * 4;
        if (f == 0) {   // covariant components of grad phi at the tent bottom
            const double* tp = a.tau + verts[w < j ? w : w + 1];
            sG()[w * CS + lane] = (Real)((CG ? load_cg(tp) : *tp) - tb) * cst(12, k);
        } else {
            // causality in FP64, one component of grad phi per warp: it is affine in t^, so
            // |grad phi| at bottom and top bounds the tent
            const double* gl = a.geo + (int64_t)sElem()[lane] * 32 + w;
            double gp = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double* tp = a.tau + verts[i];
                gp += (i == j ? tb : (CG ? load_cg(tp) : *tp)) * gl[3 * i];
            }
            const double top = gp + dtd * gl[3 * j];
            chk[2 * w * 32 + lane] = gp * gp;
            chk[(2 * w + 1) * 32 + lane] = top * top;
        }
        __syncthreads();
        if (warp == 5 && lane < ns) {
            const double* gl = a.geo + (int64_t)sElem()[lane] * 32;
            const double em = gl[29] * gl[30];
            if (!(chk[lane] + chk[64 + lane] + chk[128 + lane] < em) || !(chk[32 + lane] + chk[96 + lane] + chk[160 + lane] < em))
                atomicCAS(a.err, 0, 1);
        }
        Real z[NB];
        component_in(a, kApexDual, (f ? Real(1) : Real(-1)) * cst(17, k) / height(), z);
        apex_store<NB>(sY0() + (3 * f + w) * Sh::GB * COL, lane, z);
        apex_store<NB>(rcol(3 * f + w), lane, z);
        __syncthreads();
    }

    // all m q stages; dl receives the increment.  TAPE: U_{i,n} of every stage to slot i q + n.
    template <bool TAPE>
    __device__ __forceinline__ void stages(const KArgs& a, Real* dl, Real* tape) {
        constexpr int SLOT = 6 * Sh::GB * COL;
        const int nown = head()->nown;
        const float inv_nown = 1.0f / (float)nown;
        const Real dt = height();
#pragma unroll
        for (int b = 0; b < NB; ++b) dl[b] = Real(0);
        for (int i = 0; i < a.m; ++i) {
            const Mass K = mass_at(dt, sSub()[i]);
            phase_solve<TAPE>(K, tape + (size_t)i * a.q * SLOT);
            __syncthreads();
            for (int n = 1; n <= a.q; ++n) {
                by_component([&](auto W) { phase_traces<decltype(W)::value>(); });
                __syncthreads();
                phase_fluxes(nown, inv_nown);
                __syncthreads();
                const Real cn = sTay()[n], nn = (Real)n;
                const bool last = n == a.q;
                Real acc[NB], x[NB];
                by_component([&](auto W) {
                    phase_lift<decltype(W)::value>(acc);
                    phase_volume<decltype(W)::value>(acc, x);
                });
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    dl[b] += cn * acc[b];
                    acc[b] -= nn * x[b];
                }
                if (last) {
                    if (i + 1 == a.m) break;
                    apex_load<NB>(sY0() + (3 * f + w) * Sh::GB * COL, lane, acc);
#pragma unroll
                    for (int b = 0; b < NB; ++b) acc[b] += dl[b];
                }
                apex_store<NB>(rcol(3 * f + w), lane, acc);
                __syncthreads();
                if (!last) {
                    phase_solve<TAPE>(K, tape + (size_t)(i * a.q + n) * SLOT);
                    __syncthreads();
                }
            }
        }
    }

    // state += the own components dl (apex basis) times sc along the record's vectors at `vec`
    template <bool CG, bool CHECK = true>
    __device__ __forceinline__ void finish(const KArgs& a, Real* state, const Real* dl, int vec, Real sc) {
        constexpr int NC = 6 * NB;
        const int ns = head()->ns, k = lane < ns ? lane : ns - 1;
        const Real* ent = (const Real*)head()->ent;
        {
            const int j = *(const int8_t*)(sInfo() + 3 * k);
            Real z[NB];
            rotate<false>((const Real*)a.Rt + (size_t)j * apex_rot_offset(P + 1), dl, z);
            __syncthreads();   // the staging buffer shares the trace and U buffers (all read)
            Real* st = sTr() + k * Sh::SP + (3 * f + w) * NB;
            if (lane < ns)
#pragma unroll
                for (int b = 0; b < NB; ++b) st[b] = sc * z[b];
        }
        __syncthreads();
        bool bad = false;
        for (int idx = threadIdx.x; idx < ns * NC; idx += Sh::NT) {
            const int e = idx / NC, r = idx - e * NC, c = r / NB, b = r - c * NB, fl = c / 3, x = c - 3 * fl;
            const Real* st = sTr() + e * Sh::SP + fl * 3 * NB + b;
            const Real* t = ent + e * kApexRec + vec + x;
            Real* sp = state + (int64_t)sElem()[e] * NC + r;
            const Real v = (CG ? __ldcg(sp) : *sp) + (__ldg(t) * st[0] + __ldg(t + 3) * st[NB] + __ldg(t + 6) * st[2 * NB]);
            if (CHECK && !isfinite(v)) bad = true;
            *sp = v;
        }
        if (bad) atomicCAS(a.err, 0, 2);
    }
};

// a vertex that no element uses has a tent without elements
__device__ __forceinline__ bool apex_empty(const KArgs& a, int64_t tent) {
    const int V = a.tent_v[tent];
    return a.patch_ptr[V + 1] == a.patch_ptr[V];
}

template <typename Real, int P>
__global__ void __launch_bounds__(192, ApexShape<Real, P>::MINB) apex_layer_kernel(const KArgs a, int64_t t0) {
    ApexTent<Real, P> t;
    const int64_t tent = t0 + blockIdx.x;
    if (!apex_empty(a, tent)) {
        t.load_static(a, tent);
        t.template run<false>(a, (Real*)a.state + (int64_t)blockIdx.y * a.rhs_stride);
    }
    if (threadIdx.x == 0 && blockIdx.y == 0) a.tau[a.tent_v[tent]] = a.tent_tt[tent];
}

// One DAG-walk step (see tent_dag_step): bounded wait, all right-hand sides, publish.
template <typename Real, int P>
__device__ bool apex_dag_step(const KArgs& a, const PArgs& pa, int64_t tent, int* s_abort) {
    ApexTent<Real, P> t;
    const bool empty = apex_empty(a, tent);
    if (!empty) t.load_static(a, tent);
    if (!dag_wait(a, pa, tent, s_abort)) return false;
    for (int r = 0; r < pa.n_rhs && !empty; ++r) {
        t.template run<true>(a, (Real*)a.state + (int64_t)r * a.rhs_stride);
        __threadfence();   // publish this thread's state writes (gpu scope)
        __syncthreads();
    }
    dag_publish(a, pa, tent);
    __syncthreads();
    return true;
}

template <typename Real, int P>
__global__ void __launch_bounds__(192, ApexShape<Real, P>::MINB) apex_persistent_kernel(const KArgs a, const PArgs pa) {
    __shared__ long long s_ticket;
    __shared__ int s_abort;
    while (true) {
        if (threadIdx.x == 0) {
            s_ticket = (long long)atomicAdd(pa.next, 1ull);
            s_abort = 0;
        }
        __syncthreads();
        const long long ticket = s_ticket;
        if (ticket >= pa.n_tents) break;
        if (!apex_dag_step<Real, P>(a, pa, pa.ticket0 + ticket, &s_abort)) break;
    }
}

// Many 3D instances of degrees up to PM (see tent_batch_kernel); an instance's arguments are copied
// to shared memory with its ticket.
template <typename Real, int PM>
__global__ void __launch_bounds__(192, ApexShape<Real, PM>::MINB) apex_batch_kernel(const BatchArgs b) {
    __shared__ long long s_ticket;
    __shared__ int s_abort;
    __shared__ __align__(8) unsigned char s_args[sizeof(KArgs) + sizeof(PArgs)];
    static_assert(sizeof(KArgs) % 8 == 0 && sizeof(PArgs) % 8 == 0, "copied as 8-byte words");
    while (true) {
        if (threadIdx.x == 0) {
            s_ticket = (long long)atomicAdd(b.next, 1ull);
            s_abort = 0;
        }
        __syncthreads();
        const long long t = s_ticket;
        if (t >= b.n_tickets) break;
        const int inst = b.ticket_inst[t];
        const int64_t tent = b.ticket_tent[t];
        const uint64_t *ka = (const uint64_t*)(b.kargs + inst), *pp = (const uint64_t*)(b.pargs + inst);
        uint64_t* dst = (uint64_t*)s_args;
        for (int i = threadIdx.x; i < (int)(sizeof(KArgs) / 8); i += 192) dst[i] = ka[i];
        for (int i = threadIdx.x; i < (int)(sizeof(PArgs) / 8); i += 192) dst[sizeof(KArgs) / 8 + i] = pp[i];
        __syncthreads();
        const KArgs& a = *(const KArgs*)s_args;
        const PArgs& pa = *(const PArgs*)(s_args + sizeof(KArgs));
        bool ok = true;
        const int p = b.inst_p[inst];
        if (p == 1) ok = apex_dag_step<Real, 1>(a, pa, tent, &s_abort);
        else if (p == 2) ok = apex_dag_step<Real, 2>(a, pa, tent, &s_abort);
        if constexpr (PM >= 3)
            if (p == 3) ok = apex_dag_step<Real, 3>(a, pa, tent, &s_abort);
        if constexpr (PM >= 4)
            if (p == 4) ok = apex_dag_step<Real, 4>(a, pa, tent, &s_abort);
        if (!ok) break;
    }
}

}  // namespace mtp
