// Adjoint of the tent map in the apex frame (3D, see mtp_apex.cuh and mtp_adjoint.cuh).
//
// With the forward stages  U_0 = K (y0 + delta), acc_k = A U_{k-1}, delta += c_k acc_k,
// U_k = K (acc_k - k X U_{k-1})  (X: u_Z - u_X of the other field), D the adjoint of delta and
// nu_k = K^T (adjoint of U_k), the reverse of a sub-interval is
//   v_k = c_k D + nu_k (k < q),  adjoint of U_{k-1} = A^T v_k + k X nu_k (X^T = -X),  D += nu_0.
// A^T runs through the phases of A: traces of v, the transposed flux, lambda_V and the
// transposed traces (the lift), and the volume term with its two factors transposed.  K^T is K
// with the sign of the cross products turned.  Material gradients: a solve contributes
// -nu^T (d K^-1) U, which is +- (metric^-1 U) . nu / k for eps and mu; a flux contributes through
// the impedances.  The forward stages are replayed from the tent's bottom state into a tape in
// global memory (apex basis, one slot per stage).
//
// Measured on a GB300, forward and backward of the 8^3 x 6, p = 2, FP64 gradient problem (259 layers):
// 968 -> 321 ms, of which the forward passes fell from about 450 to 110 ms; FP64 issue bounds the rest.
#pragma once

#include "mtp_adjoint.cuh"
#include "mtp_apex.cuh"

namespace mtp {

template <typename Real, int P>
struct ApexAdjoint : ApexTent<Real, P> {
    using Base = ApexTent<Real, P>;
    using Sh = typename Base::Sh;
    using Op = typename Base::Op;
    using Mass = typename Base::Mass;
    using Base::f;
    using Base::lane;
    using Base::w;
    using Base::warp;
    static constexpr int NB = Base::NB, NFB = Base::NFB, NM = Base::NM, COL = Base::COL, CS = Base::CS;
    static constexpr int SLOT = 6 * Sh::GB * COL;
    // traces of U (times lambda_V) and, in FP64, impedances and their gradients per element
    static constexpr size_t TU = (Sh::BYTES + 15) / 16 * 16;
    static constexpr size_t Z = TU + (size_t)12 * Sh::GF * COL * sizeof(Real);
    static constexpr size_t BYTES = Z + 4 * 32 * sizeof(double);

    static __device__ __forceinline__ Real* sTu() { return (Real*)(apex_smem() + TU); }
    static __device__ __forceinline__ double* sZ() { return (double*)(apex_smem() + Z); }       // Z
    static __device__ __forceinline__ double* sGz() { return sZ() + 32; }                       // dJ/dZ
    static __device__ __forceinline__ double* sGe() { return sZ() + 64; }                       // through the solves
    static __device__ __forceinline__ double* sGm() { return sZ() + 96; }
    __device__ __forceinline__ Real* ncol(int c) const { return Base::sY0() + c * Sh::GB * COL; }   // nu

    // transposed flux in place (adjoint traces in, adjoint of the traces out) and dJ/dZ
    __device__ __forceinline__ void flux_adjoint(int nown, float inv_nown) {
        using VT = typename Vec<Real>::T;
        constexpr int VW = Sh::VW;
        for (int idx = threadIdx.x; idx < nown * Sh::GF; idx += Sh::NT) {
            const int g = (int)(((float)idx + 0.5f) * inv_nown);
            const int pk = Base::sOwn()[idx - g * nown];
            const int k = pk & 31, k2 = (pk >> 5) & 31, fi = (pk >> 10) & 3, fi2 = (pk >> 12) & 3;
            const bool wall = pk & (1 << 14);
            const Real tau = wall ? Real(0) : (pk & (1 << 15)) ? Real(-1) : Real(1);
            const Real r = fi == 1 ? Real(1) : Real(-1);
            const int o1 = (fi * 4 * Sh::GF + g) * COL + k * VW, o2 = (fi2 * 4 * Sh::GF + g) * COL + k2 * VW;
            Real *mine = Base::sTr() + o1, *other = Base::sTr() + o2;
            const int c0 = kApexFacet + 6 * fi;
            const Real a = this->cst(c0, k), b = this->cst(c0 + 1, k), qxx = this->cst(c0 + 2, k), qxy = this->cst(c0 + 3, k),
                       qyy = this->cst(c0 + 4, k), zz = this->cst(c0 + 5, k);
            const Real ra = r * a, rb = r * b;
            Real y[4][VW], o[4][VW], um[4][VW], up[4][VW];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                Vec<Real>::get(*(const VT*)(mine + s * Sh::GF * COL), y[s]);
                Vec<Real>::get(*(const VT*)(other + s * Sh::GF * COL), o[s]);
                Vec<Real>::get(*(const VT*)(sTu() + o1 + s * Sh::GF * COL), um[s]);
                Vec<Real>::get(*(const VT*)(sTu() + o2 + s * Sh::GF * COL), up[s]);
            }
            Real p1 = 0, p2 = 0, p3 = 0, p4 = 0;
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                if (g * VW + v >= NFB) {   // padding
#pragma unroll
                    for (int s = 0; s < 4; ++s) y[s][v] = o[s][v] = Real(0);
                    continue;
                }
                const Real ex = y[0][v] + tau * o[0][v], ey = y[1][v] + tau * o[1][v];
                const Real hx = y[2][v] + tau * o[2][v], hy = y[3][v] + tau * o[3][v];
                const Real dex = um[0][v] - (wall ? -um[0][v] : up[0][v]), dey = um[1][v] - (wall ? -um[1][v] : up[1][v]);
                const Real dhx = wall ? Real(0) : um[2][v] - up[2][v], dhy = wall ? Real(0) : um[3][v] - up[3][v];
                p1 += dhy * ex - dhx * ey;
                p2 += (qxx * dex + qxy * dey) * ex + (qxy * dex + qyy * dey) * ey;
                p3 += dey * hx - dex * hy;
                p4 += (qxx * dhx + qxy * dhy) * hx + (qxy * dhx + qyy * dhy) * hy;
                const Real qex = qxx * ex + qxy * ey, qey = qxy * ex + qyy * ey;
                const Real qhx = zz * (qxx * hx + qxy * hy), qhy = zz * (qxy * hx + qyy * hy);
                y[0][v] = qex - rb * hy;
                y[1][v] = qey + rb * hx;
                y[2][v] = -ra * ey - qhx;
                y[3][v] = ra * ex - qhy;
                o[0][v] = -qex - ra * hy;
                o[1][v] = -qey + ra * hx;
                o[2][v] = -rb * ey + qhx;
                o[3][v] = rb * ex + qhy;
                if (wall) {   // E+ = -E-, H+ = H-
                    y[0][v] -= o[0][v];
                    y[1][v] -= o[1][v];
                    y[2][v] += o[2][v];
                    y[3][v] += o[3][v];
                }
            }
            const Real zm = (Real)sZ()[k], zp = (Real)sZ()[k2], is = Real(1) / (zm + zp);
            const Real gm = (b * r * (p1 - p3) - p2) * is - zp * b * p4;
            const Real gp = (a * r * (p3 - p1) - p2) * is - zm * a * p4;
            atomicAdd(&sGz()[k], (double)gm);
            atomicAdd(&sGz()[k2], (double)gp);   // the wall's Z+ is the element's own
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                *(VT*)(mine + s * Sh::GF * COL) = apex_pack(y[s]);
                if (!wall) *(VT*)(other + s * Sh::GF * COL) = apex_pack(o[s]);
            }
        }
    }

    // acc -= transposed volume term of the own component, from v of the other field
    template <int WT>
    __device__ __forceinline__ void volume_adjoint(Real* acc) {
        const int W = WT < 0 ? w : WT, o = 3 * (1 - f);
        Real p[NM];
        {
            Real vz[NB], x[NB], v[NB];
            apex_load<NB>(this->ucol(o + (W == 0 ? 2 : W - 1)), lane, vz);
            apex_load<NB>(this->ucol(o + (W == 2 ? 0 : W + 1)), lane, x);
            const Real cd = W == 2 ? Real(-0.5) : Real(0.5);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                v[b] = W == 0 ? vz[b] : W == 1 ? x[b] : vz[b] + x[b];
                x[b] = vz[b] - x[b];
            }
            Op::volt_ab(x, p);
#pragma unroll
            for (int b = 0; b < NB; ++b) {   // d_Bm of -v_B, v_B or -(v_D - v_C)
                vz[b] = W == 0 ? -v[b] : W == 1 ? v[b] : -x[b];
                v[b] *= cd;
            }
            Op::volt_mb(vz, p);
            Op::volt_cd(v, p);
        }
#pragma unroll
        for (int c = 0; c < NM; ++c) p[c] = -p[c];
        Op::mass_t(p, acc);
    }

    // nu = K^T r, and the solves' material gradients from nu and U of the tape slot
    __device__ __forceinline__ void solve_adjoint(const Mass& K, const Real* tape, double& ge, double& gm) {
        using VT = typename Vec<Real>::T;
        constexpr int VW = Sh::VW;
        Real i0 = this->cst(6, lane), i1 = this->cst(7, lane), i2 = this->cst(8, lane), i3 = this->cst(9, lane),
             i4 = this->cst(10, lane), i5 = this->cst(11, lane);
#pragma unroll 1
        for (int g = warp; g < Sh::GB; g += 6) {
            Real r[6][VW], u[6][VW];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                Vec<Real>::get(*(const VT*)(this->rcol(c) + (g * 32 + lane) * VW), r[c]);
                Vec<Real>::get(*(const VT*)(tape + (c * Sh::GB + g) * COL + lane * VW), u[c]);
            }
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                if (g * VW + v >= NB) continue;
                Real e[3], h[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    e[q] = K.dE * r[q][v];
                    h[q] = K.dH * r[3 + q][v];
                }
                const Real e0 = r[0][v], e1 = r[1][v], e2 = r[2][v], h0 = r[3][v], h1 = r[4][v], h2 = r[5][v];
                r[0][v] = K.m[0] * e[0] + K.m[1] * e[1] + K.m[2] * e[2] - (K.c[1] * h2 - K.c[2] * h1);
                r[1][v] = K.m[1] * e[0] + K.m[3] * e[1] + K.m[4] * e[2] - (K.c[2] * h0 - K.c[0] * h2);
                r[2][v] = K.m[2] * e[0] + K.m[4] * e[1] + K.m[5] * e[2] - (K.c[0] * h1 - K.c[1] * h0);
                r[3][v] = K.m[0] * h[0] + K.m[1] * h[1] + K.m[2] * h[2] - (K.c[1] * e2 - K.c[2] * e1);
                r[4][v] = K.m[1] * h[0] + K.m[3] * h[1] + K.m[4] * h[2] - (K.c[2] * e0 - K.c[0] * e2);
                r[5][v] = K.m[2] * h[0] + K.m[4] * h[1] + K.m[5] * h[2] - (K.c[0] * e1 - K.c[1] * e0);
                ge += (double)(r[0][v] * (i0 * u[0][v] + i1 * u[1][v] + i2 * u[2][v]) +
                               r[1][v] * (i1 * u[0][v] + i3 * u[1][v] + i4 * u[2][v]) +
                               r[2][v] * (i2 * u[0][v] + i4 * u[1][v] + i5 * u[2][v]));
                gm -= (double)(r[3][v] * (i0 * u[3][v] + i1 * u[4][v] + i2 * u[5][v]) +
                               r[4][v] * (i1 * u[3][v] + i3 * u[4][v] + i4 * u[5][v]) +
                               r[5][v] * (i2 * u[3][v] + i4 * u[4][v] + i5 * u[5][v]));
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) *(VT*)(ncol(c) + (g * 32 + lane) * VW) = apex_pack(r[c]);
        }
    }

    __device__ void reverse(const KArgs& a, const Real* ybot, Real* lam, Real* tape, double* geps, double* gmu) {
        const Real sgn = f ? Real(1) : Real(-1);
        this->template begin<false>(a, ybot);
        {
            Real dl[NB];
            this->template stages<true>(a, dl, tape);   // replay
        }
        __syncthreads();
        this->template stage_patch<false>(lam);
        if (warp == 0) {
            sZ()[lane] = a.geo[(int64_t)Base::sElem()[lane] * 32 + 31];
            sGz()[lane] = sGe()[lane] = sGm()[lane] = 0.0;
        }
        __syncthreads();
        const int ns = Base::head()->ns, k = lane < ns ? lane : ns - 1, nown = Base::head()->nown;
        const float inv_nown = 1.0f / (float)nown;
        const Real dt = this->height();
        Real D[NB], y0[NB];
        this->component_in(a, kApexEdge, sgn * dt * this->cst(18, k), D);   // adjoint of the increment
#pragma unroll
        for (int b = 0; b < NB; ++b) y0[b] = Real(0);
        double ge = 0, gm = 0;
        __syncthreads();
        for (int i = a.m - 1; i >= 0; --i) {
            const Mass K = this->mass_at(dt, Base::sSub()[i]);
            for (int n = a.q; n >= 1; --n) {
                const Real* un = tape + (size_t)(i * a.q + n - 1) * SLOT;   // U_{i, n-1}
                const Real cn = Base::sTay()[n];
                this->by_component([&](auto Wc) {
                    constexpr int WT = decltype(Wc)::value;
                    Real v[NB];
                    if (n < a.q) apex_load<NB>(ncol(3 * f + w), lane, v);
#pragma unroll
                    for (int b = 0; b < NB; ++b) v[b] = n < a.q ? v[b] + cn * D[b] : cn * D[b];
                    apex_store<NB>(this->ucol(3 * f + w), lane, v);
                    this->template traces_of<WT, false>(v, Base::sTr());
                    apex_load<NB>(un + (size_t)(3 * f + w) * Sh::GB * COL, lane, v);
                    this->template traces_of<WT, true>(v, sTu());
                });
                __syncthreads();
                flux_adjoint(nown, inv_nown);
                __syncthreads();
                Real acc[NB];
                this->by_component([&](auto Wc) {
                    constexpr int WT = decltype(Wc)::value;
                    this->template phase_lift<WT>(acc);
                    volume_adjoint<WT>(acc);
                });
                if (n < a.q) {
                    Real nz[NB], nx[NB];
                    apex_load<NB>(ncol(3 * (1 - f) + (w == 0 ? 2 : w - 1)), lane, nz);
                    apex_load<NB>(ncol(3 * (1 - f) + (w == 2 ? 0 : w + 1)), lane, nx);
#pragma unroll
                    for (int b = 0; b < NB; ++b) acc[b] += (Real)n * (nz[b] - nx[b]);
                }
                apex_store<NB>(this->rcol(3 * f + w), lane, acc);
                __syncthreads();
                solve_adjoint(K, un, ge, gm);
                __syncthreads();
            }
            Real nu[NB];
            apex_load<NB>(ncol(3 * f + w), lane, nu);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                D[b] += nu[b];
                y0[b] += nu[b];
            }
        }
        if (lane < ns) {
            atomicAdd(&sGe()[lane], ge);
            atomicAdd(&sGm()[lane], gm);
        }
        this->template finish<false, false>(a, lam, y0, kApexDual, sgn * this->cst(17, k) / dt);
        if (warp == 0 && lane < ns) {
            const int e = Base::sElem()[lane];
            const double eps = a.geo[(int64_t)e * 32 + 29], mu = a.geo[(int64_t)e * 32 + 30], z = sZ()[lane];
            const double ik = 1.0 / ((double)dt * (double)this->cst(16, lane));
            atomicAdd(&geps[e], sGe()[lane] * ik - sGz()[lane] * z / (2.0 * eps));
            atomicAdd(&gmu[e], sGm()[lane] * ik + sGz()[lane] * z / (2.0 * mu));
        }
    }
};

template <typename Real, int P>
__global__ void __launch_bounds__(192, 1) apex_adjoint_kernel(const AdjArgs A, int64_t t0) {
    const KArgs& a = A.k;
    const int64_t tent = t0 + blockIdx.x, off = (int64_t)blockIdx.y * a.rhs_stride;
    if (apex_empty(a, tent)) {
        if (threadIdx.x == 0 && blockIdx.y == 0) a.tau[a.tent_v[tent]] = a.tent_tb[tent];
        return;
    }
    ApexAdjoint<Real, P> t;
    t.load_static(a, tent);
    t.reverse(a, (const Real*)A.ybot + off, (Real*)A.lam + off,
              (Real*)A.tape + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * A.tape_stride, A.geps, A.gmu);
    if (threadIdx.x == 0 && blockIdx.y == 0) a.tau[a.tent_v[tent]] = a.tent_tb[tent];
}

}  // namespace mtp
