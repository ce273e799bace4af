// Apex tent kernel in 2D (FP64 or FP32 arithmetic, p = 1..5): the basis and the frame of
// mtp_apex.cuh on triangles, with another split of the work.
//
// A 2D patch has six elements or so and its layers few tents, so an evolve takes layers x latency
// of a tent, and in FP64 that latency is a count of instructions: one costs a warp 64 clocks (19 of
// the SM) however many of its lanes are active (measured).  So lanes are packed: a thread owns one
// (element, row) and reads the coefficients of its row from shared memory.  TE fields:
// e_X = E . t_X (two edges from V), h = H_z; with coefficients scaled by l s (E) and s (H),
// s = 1 / sqrt|det|, traces and lifts carry no factor, and
//   acc_0 = S_1 h,  acc_1 = -S_0 h,  acc_h = S_0 e_1 - S_1 e_0,  r = acc - n (h, -h, e_1 - e_0).
// Exchanging the two edges flips the sign of the odd functions, so S_0 and S_1 are
// sum and difference of a table C of the same parity and one of the opposite parity (each entry of
// C belongs to one of them), so every component is one pass over its row of C, the H component with
// e_1 - e_0 and e_1 + e_0.
//
// Measured against the general kernel on a GB300, one slab of the TE cavity in FP64: 8 x 8, p = 2,
// 14.2 -> 3.3 ms; 32 x 32, p = 4, 134 -> 40 ms (3.3 and 7.7 us a stage and layer; waits at the barriers
// for the warp with the longest FP64 chain, the FP64 pipe is busy 27 % of the time).
#pragma once

#include "mtp_apex.cuh"
#include "mtp_kernels.cuh"

namespace mtp {

// Record of a patch entry: [0..2] metric t_X . t_Z (00 01 11), [3..5] its inverse, [6] 1 / l,
// [7] eps, [8] mu, [10] 1 / (eps mu), [11] k / dt = 1 / (l det), [14] 1 / det of the scaled edges;
// scales of y0 times dt [12] E, [13] H and of the increment over dt [31] E, [9] H; per edge facet f
// [15 + 4 f] a, b, q = sgn / (len (Z- + Z+)), qz = sgn Z- Z+ len / (Z- + Z+); [23..26] dual vectors,
// [27..30] edges.
constexpr int kApex2Rec = 32;
// most entries in a row of C, p = 1..5
constexpr int kApex2MaxRow[5] = {2, 5, 9, 14, 20};

// tables of one degree in the arithmetic precision: C in compressed rows (entries of equal parity
// first), T of the first edge [mode][b], L of the first edge [a][mode], change of basis [j][a][place in
// block]; then bytes: per row its start (two), its entries of equal and of opposite parity, the
// columns, and the rows by ascending length
template <int P>
struct Apex2Tables {
    static constexpr int NB = dim_pk(2, P), NFB = P + 1;
    static constexpr int C = 0, T = C + NB * NB, L = T + NFB * NB, R = L + NB * NFB;
    static constexpr int REALS = R + 3 * NB * NFB;
    static constexpr int COLS = 4 * NB, ORDER = COLS + NB * NB, BYTES = ORDER + NB;
};

template <typename Real, int P>
struct Apex2 {
    using Tab = Apex2Tables<P>;
    static constexpr int NB = Tab::NB, NFB = Tab::NFB, E = 16;
    static constexpr int MAXR = kApex2MaxRow[P - 1];
    static constexpr int KB = 8;                     // sub-intervals whose K is built together
    static constexpr int NT = (3 * 6 * NB + 31) / 32 * 32;   // a six-element patch in one round
    static constexpr int COL = NB * E;
    // shared memory in Reals: u (e_0, e_1, h, e_1 - e_0, -e_1 - e_0), r, y0, delta, traces, fluxes, K,
    // element constants, front, tables
    static constexpr int U = 0, R = U + 5 * COL, Y0 = R + 3 * COL, D = Y0 + 3 * COL, TR = D + 3 * COL,
                         FL = TR + 4 * NFB * E, K = FL + 4 * NFB * E, C = K + KB * 6 * E, G = C + kApex2Rec * E,
                         TB = G + 2 * E, SUB = TB + Tab::R, TAY = SUB + kMaxSub + 1, NUM = TAY + kMaxTaylor,
                         END = NUM + kMaxTaylor;
    static constexpr size_t I = ((size_t)END * sizeof(Real) + 7) / 8 * 8;
    struct Head {
        double tb, tt;
        Real dt, idt;
        int ns, nown;
        int elem[E], info[3 * E], own[2 * E];
        uint8_t row[Tab::BYTES];
    };
    static constexpr size_t BYTES = I + sizeof(Head);

    static __device__ __forceinline__ Real* sm() {
        extern __shared__ __align__(16) unsigned char smem[];
        return (Real*)smem;
    }
    static __device__ __forceinline__ Head* head() { return (Head*)((unsigned char*)sm() + I); }
    static __device__ __forceinline__ Real cst(int word, int e) { return sm()[C + word * E + e]; }
    // (row, element) of item idx when the element runs fastest
    static __device__ __forceinline__ int row_of(int idx, float inv) { return (int)(((float)idx + 0.5f) * inv); }
    static __host__ __device__ constexpr bool odd(int b) {   // parity of the function's collapsed index
        int d = 0;
        while (b >= dim_pk(2, d)) ++d;
        return (b - dim_pk(2, d - 1)) & 1;
    }
    static __device__ __forceinline__ bool is_odd(int b) {
        int d = 0;
#pragma unroll
        for (int k = 0; k < P; ++k) d += b >= dim_pk(2, k);
        return (b - d * (d + 1) / 2) & 1;
    }

    // tables that every tent of the CTA uses
    static __device__ void load_tables(const KArgs& a) {
        const Real* t = (const Real*)a.apex2;
        for (int i = threadIdx.x; i < Tab::R; i += blockDim.x) sm()[TB + i] = t[i];
        const uint8_t* r = (const uint8_t*)(t + Tab::REALS);
        for (int i = threadIdx.x; i < Tab::BYTES; i += blockDim.x) head()->row[i] = r[i];
        for (int i = threadIdx.x; i <= kMaxSub; i += blockDim.x) {
            sm()[SUB + i] = (Real)a.tsub[i];
            if (i < kMaxTaylor) {
                sm()[TAY + i] = (Real)a.taylor[i];
                sm()[NUM + i] = (Real)i;
            }
        }
    }

    static __device__ void load_static(const KArgs& a, int64_t tent) {
        const int V = a.tent_v[tent];
        const int64_t pb = a.patch_ptr[V];
        const int ns = (int)(a.patch_ptr[V + 1] - pb);
        const Real* ent = (const Real*)a.ent + pb * kApex2Rec;
        Head* h = head();
        if (threadIdx.x == 0) {
            h->tb = a.tent_tb[tent];
            h->tt = a.tent_tt[tent];
            // one of almost no height changes nothing: keep 1 / dt finite
            h->dt = (Real)fmax(h->tt - h->tb, sizeof(Real) == 4 ? 1e-30 : 1e-200);
            h->idt = Real(1) / h->dt;
            h->ns = ns;
        }
        for (int i = threadIdx.x; i < ns; i += blockDim.x) h->elem[i] = a.patch_elem[pb + i];
        for (int i = threadIdx.x; i < 3 * ns; i += blockDim.x) h->info[i] = ((const int*)(a.patch_info + pb * 12))[i];
        for (int i = threadIdx.x; i < ns * kApex2Rec; i += blockDim.x) sm()[C + (i % kApex2Rec) * E + i / kApex2Rec] = ent[i];
        __syncthreads();
        if (threadIdx.x < 32) {   // owned facets: boundary ones and the lower slot of interior ones
            const int lane = threadIdx.x, k = lane < ns ? lane : ns - 1;
            const int8_t* inf = (const int8_t*)(h->info + 3 * k);
            const int j = inf[0];
            int s2[2];
            unsigned own[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {   // facet along edge q: opposite the other vertex
                const int lf = 1 - q < j ? 1 - q : 2 - q;
                s2[q] = inf[4 + lf];
                own[q] = __ballot_sync(0xffffffffu, lane < ns && (s2[q] < 0 || s2[q] > lane));
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (own[q] >> lane & 1) {
                    int k2 = lane, q2 = q, neg = 0;
                    if (s2[q] >= 0) {
                        k2 = s2[q];
                        const int lf = 1 - q < j ? 1 - q : 2 - q, f2 = inf[8 + lf], j2 = *(const int8_t*)(h->info + 3 * k2);
                        q2 = 1 - (f2 - (f2 > j2 ? 1 : 0));
                        neg = (cst(14, k) > Real(0)) == (cst(14, k2) > Real(0));
                    }
                    h->own[(q ? __popc(own[0]) : 0) + __popc(own[q] & ((1u << lane) - 1))] =
                        lane | k2 << 4 | q << 8 | q2 << 9 | (s2[q] < 0 ? 1 << 10 : 0) | (neg ? 1 << 11 : 0);
                }
            if (lane == 0) h->nown = __popc(own[0]) + __popc(own[1]);
        }
    }

    // traces of e_0 on edge 0, of e_1 on edge 1 and of h on both (even and odd functions apart)
    static __device__ __forceinline__ void phase_traces(int ns, float inv) {
        const Real* u = sm() + U;
        for (int idx = threadIdx.x; idx < 3 * NFB * ns; idx += blockDim.x) {
            const int q = row_of(idx, inv), e = idx - q * ns, kind = q / NFB, n = q - kind * NFB;
            const Real* T = sm() + TB + Tab::T + n * NB;
            const Real* x = u + kind * COL + e;
            Real ev = 0, od = 0;
#pragma unroll
            for (int d = 0; d <= P; ++d)
                if (d >= n)
#pragma unroll
                    for (int b = dim_pk(2, d - 1); b < dim_pk(2, d); ++b) {
                        if (odd(b)) od += T[b] * x[b * E];
                        else ev += T[b] * x[b * E];
                    }
            Real* t = sm() + TR + n * E + e;
            if (kind == 0) t[0] = ev + od;
            else if (kind == 1) t[2 * NFB * E] = ev - od;
            else {
                t[NFB * E] = ev + od;
                t[3 * NFB * E] = ev - od;
            }
        }
    }

    // upwind flux, once per facet and field (see mtp_apex.cuh):
    //   E: r (a h- + b h+) + q (e- - e+),  H: -r (b e- + a e+) - qz (h- - h+),  r = +-1 on edge 0 / 1
    static __device__ __forceinline__ void phase_fluxes(int nown, float inv) {
        for (int idx = threadIdx.x; idx < 2 * NFB * nown; idx += blockDim.x) {
            const int q = row_of(idx, inv), pk = head()->own[idx - q * nown], fld = q & 1, n = q >> 1;
            const int k = pk & 15, k2 = (pk >> 4) & 15, f1 = (pk >> 8) & 1, f2 = (pk >> 9) & 1;
            const bool wall = pk & (1 << 10);
            const Real* m = sm() + TR + (2 * f1 * NFB + n) * E + k;
            const Real* o = sm() + TR + (2 * f2 * NFB + n) * E + k2;
            const int c = 15 + 4 * f1;
            // one path for both fields: E takes h as the first pair and e as the jump, H the reverse
            const Real x = m[(1 - fld) * NFB * E], z = m[fld * NFB * E];
            const Real xp = wall ? (fld ? -x : x) : o[(1 - fld) * NFB * E];
            const Real zp = wall ? (fld ? z : -z) : o[fld * NFB * E];
            const Real a = cst(c + fld, k), b = cst(c + 1 - fld, k), q2 = cst(c + 2 + fld, k), d = z - zp;
            Real y = a * x + b * xp;
            y = ((f1 != fld) ? -y : y) + (fld ? -q2 : q2) * d;
            sm()[FL + ((2 * f1 + fld) * NFB + n) * E + k] = y;
            if (!wall) sm()[FL + ((2 * f2 + fld) * NFB + n) * E + k2] = (pk & (1 << 11)) ? -y : y;
        }
    }

    // What a thread keeps of its row (component c, row a, element e): the coefficients, with the
    // component's sign, and the places of their operands, so that in the stages nothing waits on an
    // index.  Rows are dealt out by length, and `most` is the longest of the warp: a row of one warp
    // costs what its own length asks for (p = 4: 6.6 entries on average, 14 at most).
    struct Row {
        Real cf[MAXR];
        int at[MAXR];
        int c, a, e, most;
    };
    static __device__ __forceinline__ void load_row(Row& w, int idx, int ns, float inv) {
        const uint8_t* row = head()->row;
        const int q = row_of(idx, inv);
        w.e = idx - q * ns;
        w.c = q / NB;
        w.a = row[Tab::ORDER + q - w.c * NB];
        const uint8_t* col = row + Tab::COLS;
        const int s0 = row[4 * w.a] | row[4 * w.a + 1] << 8, n1 = row[4 * w.a + 2], n = n1 + row[4 * w.a + 3];
#pragma unroll
        for (int i = 0; i < MAXR; ++i) {
            const bool on = i < n;
            const Real v = on ? sm()[TB + Tab::C + s0 + i] : Real(0);
            w.cf[i] = w.c == 1 && i < n1 ? -v : v;
            w.at[i] = (w.c < 2 ? 2 : i < n1 ? 3 : 4) * COL + (on ? col[s0 + i] * E : 0) + w.e;
        }
        w.most = n;
    }

    // volume + lift, delta += cn acc, and r for the next solve: acc - n x, or y0 + delta when the
    // sub-interval ends; one thread per (component, row, element)
    static __device__ __forceinline__ void phase_volume(Row& w, bool one, int ns, float inv, Real cn, Real nn, bool last) {
        for (int idx = threadIdx.x; idx < 3 * NB * ns; idx += blockDim.x) {
            if (!one) load_row(w, idx, ns, inv);
            const int c = w.c;
            Real v[MAXR], fl[2][NFB];
#pragma unroll
            for (int i = 0; i < MAXR; ++i) v[i] = sm()[U + w.at[i]];
            const Real* F = sm() + FL + (c == 2 ? NFB * E : 0) + w.e;
            const Real* L = sm() + TB + Tab::L + w.a * NFB;
            Real l[NFB];
#pragma unroll
            for (int n = 0; n < NFB; ++n) {
                l[n] = L[n];
                fl[0][n] = F[n * E];
                fl[1][n] = F[(2 * NFB + n) * E];
            }
            const int at = c * COL + w.a * E + w.e;
            const Real d0 = sm()[D + at], tail = last ? sm()[Y0 + at] : sm()[U + (c == 2 ? 3 : 2) * COL + w.a * E + w.e];
            Real acc = 0;
#pragma unroll
            for (int i = 0; i < MAXR; ++i)
                if (i < w.most) acc += w.cf[i] * v[i];
            if (c != 1)
#pragma unroll
                for (int n = 0; n < NFB; ++n) acc += l[n] * fl[0][n];
            if (c != 0) {
                const bool odd = is_odd(w.a);
#pragma unroll
                for (int n = 0; n < NFB; ++n) acc += (odd ? -l[n] : l[n]) * fl[1][n];
            }
            const Real d = d0 + cn * acc;
            sm()[D + at] = d;
            sm()[R + at] = last ? tail + d : acc + (c == 1 ? nn : -nn) * tail;
        }
    }

    // K of KB sub-intervals from i0 on: e = [k00 k01; k01 k11] r_e + (k02, k12) r_h,
    // h = -(k02, k12) . r_e + k22 r_h (closed-form G^-1, Sec. 4, between the scaled frames)
    static __device__ void build_k(int ns, float inv, int i0, int m, Real dt) {
        for (int idx = threadIdx.x; idx < KB * ns; idx += blockDim.x) {
            const int q = row_of(idx, inv), e = idx - q * ns;
            if (i0 + q >= m) break;
            const Real tl = sm()[SUB + i0 + q] * dt * cst(6, e);
            const Real g0 = sm()[G + e] - tl, g1 = sm()[G + E + e] - tl;
            const Real p0 = cst(3, e) * g0 + cst(4, e) * g1, p1 = cst(4, e) * g0 + cst(5, e) * g1;
            const Real eps = cst(7, e), mu = cst(8, e), iem = cst(10, e);
            const Real s = dt / (eps * mu - (g0 * p0 + g1 * p1)), d = -s * cst(14, e) * mu, c = s * cst(6, e);
            Real* k = sm() + K + q * 6 * E + e;
            k[0] = d * (cst(0, e) - g0 * g0 * iem);
            k[E] = d * (cst(1, e) - g0 * g1 * iem);
            k[2 * E] = d * (cst(2, e) - g1 * g1 * iem);
            k[3 * E] = -c * p1;
            k[4 * E] = c * p0;
            k[5 * E] = s * eps * cst(11, e) * cst(6, e);
        }
    }
    static __device__ __forceinline__ void phase_solve(int ns, float inv, int i) {
        const Real* kk = sm() + K + (i % KB) * 6 * E;
        for (int idx = threadIdx.x; idx < NB * ns; idx += blockDim.x) {
            const int b = row_of(idx, inv), e = idx - b * ns, at = b * E + e;
            const Real* k = kk + e;
            const Real r0 = sm()[R + at], r1 = sm()[R + COL + at], r2 = sm()[R + 2 * COL + at];
            const Real u0 = k[0] * r0 + k[E] * r1 + k[3 * E] * r2;
            const Real u1 = k[E] * r0 + k[2 * E] * r1 + k[4 * E] * r2;
            Real* u = sm() + U + at;
            u[0] = u0;
            u[COL] = u1;
            u[2 * COL] = k[5 * E] * r2 - (k[3 * E] * r0 + k[4 * E] * r1);
            u[3 * COL] = u1 - u0;
            u[4 * COL] = -u1 - u0;
        }
    }

    // the tent for one right-hand side (see ApexTent::run)
    template <bool CG>
    static __device__ void run(const KArgs& a, Real* state) {
        __syncthreads();
        const Head* h = head();
        const int ns = h->ns, nown = h->nown;
        const double tb = h->tb, dtd = h->tt - tb;
        const float inv = 1.0f / (float)ns, inv_own = 1.0f / (float)nown;
        const Real dt = h->dt, idt = h->idt;
        constexpr int NC = 3 * NB;
        Real* in = sm() + R;   // staged library coefficients [comp][b][e]
        for (int idx = threadIdx.x; idx < ns * NC; idx += blockDim.x) {
            const int e = idx / NC, r = idx - e * NC;
            const Real* sp = state + (int64_t)h->elem[e] * NC + r;
            in[r * E + e] = CG ? __ldcg(sp) : *sp;
        }
        for (int idx = threadIdx.x; idx < 3 * ns; idx += blockDim.x) {
            const int q = row_of(idx, inv), e = idx - q * ns;
            const int32_t* v = a.elems + (int64_t)h->elem[e] * 3;
            const int j = *(const int8_t*)(h->info + 3 * e);
            if (q < 2) {
                const double* tp = a.tau + v[q < j ? q : q + 1];
                sm()[G + q * E + e] = (Real)((CG ? load_cg(tp) : *tp) - tb) * cst(6, e);
            } else {   // causality in FP64 at the bottom and the top of the tent
                const double* gl = a.geo + (int64_t)h->elem[e] * 32;
                double gp[2] = {0, 0}, gb = 0, gt = 0;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const double* tp = a.tau + v[i];
                    const double tv = i == j ? tb : (CG ? load_cg(tp) : *tp);
                    gp[0] += tv * gl[3 * i];
                    gp[1] += tv * gl[3 * i + 1];
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const double top = gp[x] + dtd * gl[3 * j + x];
                    gb += gp[x] * gp[x];
                    gt += top * top;
                }
                const double em = gl[29] * gl[30];
                if (!(gb < em) || !(gt < em)) atomicCAS(a.err, 0, 1);
            }
        }
        __syncthreads();
        // contravariant components, then the apex basis
        const Real* Rt = (const Real*)a.apex2 + Tab::R;
        for (int idx = threadIdx.x; idx < NC * ns; idx += blockDim.x) {
            const int q = row_of(idx, inv), e = idx - q * ns, c = q / NB, r = q - c * NB;
            int d = 0;
#pragma unroll
            for (int k = 0; k < P; ++k) d += r >= dim_pk(2, k);
            const int b0 = d * (d + 1) / 2, j = *(const int8_t*)(h->info + 3 * e);
            const Real* rt = Rt + (j * NB + r) * NFB;
            Real v0 = 0, v1 = 0;
            const Real *x0 = in + (c == 2 ? 2 * NB + b0 : b0) * E + e, *x1 = in + (NB + b0) * E + e;
            for (int b = 0; b <= d; ++b) {
                const Real t = __ldg(rt + b);
                v0 += t * x0[b * E];
                if (c < 2) v1 += t * x1[b * E];
            }
            const Real y = c == 2 ? v0 * (cst(13, e) * idt)
                                  : (cst(23 + 2 * c, e) * v0 + cst(24 + 2 * c, e) * v1) * (cst(12, e) * idt);
            sm()[Y0 + c * COL + r * E + e] = y;
            sm()[D + c * COL + r * E + e] = Real(0);
        }
        build_k(ns, inv, 0, a.m, dt);
        __syncthreads();
        for (int idx = threadIdx.x; idx < NC * ns; idx += blockDim.x) {
            const int q = row_of(idx, inv), at = q * E + idx - q * ns;
            sm()[R + at] = sm()[Y0 + at];
        }
        __syncthreads();
        Row row;
        const bool one = 3 * NB * ns <= (int)blockDim.x;   // every row has a thread of its own
        if (one) {
            load_row(row, min((int)threadIdx.x, 3 * NB * ns - 1), ns, inv);
            row.most = __reduce_max_sync(0xffffffffu, row.most);   // uniform: the loop is skipped by the warp
        }
        for (int i = 0; i < a.m; ++i) {
            phase_solve(ns, inv, i);
            __syncthreads();
            for (int n = 1; n <= a.q; ++n) {
                phase_traces(ns, inv);
                __syncthreads();
                phase_fluxes(nown, inv_own);
                __syncthreads();
                const bool last = n == a.q;
                phase_volume(row, one, ns, inv, sm()[TAY + n], sm()[NUM + n], last);
                if (last && (i + 1) % KB == 0 && i + 1 < a.m) build_k(ns, inv, i + 1, a.m, dt);
                __syncthreads();
                if (!last) {
                    phase_solve(ns, inv, i);
                    __syncthreads();
                }
            }
        }
        // back to the library basis, add the increment
        bool bad = false;
        for (int idx = threadIdx.x; idx < ns * NC; idx += blockDim.x) {
            const int e = idx / NC, q = idx - e * NC, c = q / NB, b = q - c * NB;
            int d = 0;
#pragma unroll
            for (int k = 0; k < P; ++k) d += b >= dim_pk(2, k);
            const int b0 = d * (d + 1) / 2, j = *(const int8_t*)(h->info + 3 * e);
            const Real* rt = Rt + (j * NB + b0) * NFB + (b - b0);
            const Real *x0 = sm() + D + (c == 2 ? 2 * COL : 0) + b0 * E + e, *x1 = sm() + D + COL + b0 * E + e;
            Real v0 = 0, v1 = 0;
            for (int r = 0; r <= d; ++r) {
                const Real t = __ldg(rt + r * NFB);
                v0 += t * x0[r * E];
                if (c < 2) v1 += t * x1[r * E];
            }
            const Real inc = c == 2 ? v0 * (cst(9, e) * dt)
                                    : (cst(27 + c, e) * v0 + cst(29 + c, e) * v1) * (cst(31, e) * dt);
            Real* sp = state + (int64_t)h->elem[e] * NC + q;
            const Real v = (CG ? __ldcg(sp) : *sp) + inc;
            if (!isfinite(v)) bad = true;
            *sp = v;
        }
        if (bad) atomicCAS(a.err, 0, 2);
    }
};

template <typename Real, int P>
__global__ void __launch_bounds__(Apex2<Real, P>::NT, P < 5 ? 2 : 1) apex2_layer_kernel(const KArgs a, int64_t t0) {
    using T = Apex2<Real, P>;
    const int64_t tent = t0 + blockIdx.x;
    if (!apex_empty(a, tent)) {
        T::load_tables(a);
        T::load_static(a, tent);
        T::template run<false>(a, (Real*)a.state + (int64_t)blockIdx.y * a.rhs_stride);
    }
    if (threadIdx.x == 0 && blockIdx.y == 0) a.tau[a.tent_v[tent]] = a.tent_tt[tent];
}

template <typename Real, int P>
__device__ bool apex2_dag_step(const KArgs& a, const PArgs& pa, int64_t tent, int* s_abort) {
    using T = Apex2<Real, P>;
    const bool empty = apex_empty(a, tent);
    if (!empty) T::load_static(a, tent);
    if (!dag_wait(a, pa, tent, s_abort)) return false;
    for (int r = 0; r < pa.n_rhs && !empty; ++r) {
        T::template run<true>(a, (Real*)a.state + (int64_t)r * a.rhs_stride);
        __threadfence();   // publish this thread's state writes (gpu scope)
        __syncthreads();
    }
    dag_publish(a, pa, tent);
    __syncthreads();
    return true;
}

template <typename Real, int P>
__global__ void __launch_bounds__(Apex2<Real, P>::NT, P < 5 ? 2 : 1) apex2_persistent_kernel(const KArgs a, const PArgs pa) {
    __shared__ long long s_ticket;
    __shared__ int s_abort;
    Apex2<Real, P>::load_tables(a);
    while (true) {
        if (threadIdx.x == 0) {
            s_ticket = (long long)atomicAdd(pa.next, 1ull);
            s_abort = 0;
        }
        __syncthreads();
        const long long ticket = s_ticket;
        if (ticket >= pa.n_tents) break;
        if (!apex2_dag_step<Real, P>(a, pa, pa.ticket0 + ticket, &s_abort)) break;
    }
}

// many 2D instances (see apex_batch_kernel); a ticket brings its instance's arguments and tables
template <typename Real>
__global__ void __launch_bounds__(256) apex2_batch_kernel(const BatchArgs b) {
    __shared__ long long s_ticket;
    __shared__ int s_abort;
    __shared__ __align__(8) unsigned char s_args[sizeof(KArgs) + sizeof(PArgs)];
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
        for (int i = threadIdx.x; i < (int)(sizeof(KArgs) / 8); i += blockDim.x) dst[i] = ka[i];
        for (int i = threadIdx.x; i < (int)(sizeof(PArgs) / 8); i += blockDim.x) dst[sizeof(KArgs) / 8 + i] = pp[i];
        __syncthreads();
        const KArgs& a = *(const KArgs*)s_args;
        const PArgs& pa = *(const PArgs*)(s_args + sizeof(KArgs));
        bool ok = true;
        switch (b.inst_p[inst]) {
            case 1: Apex2<Real, 1>::load_tables(a); ok = apex2_dag_step<Real, 1>(a, pa, tent, &s_abort); break;
            case 2: Apex2<Real, 2>::load_tables(a); ok = apex2_dag_step<Real, 2>(a, pa, tent, &s_abort); break;
            case 3: Apex2<Real, 3>::load_tables(a); ok = apex2_dag_step<Real, 3>(a, pa, tent, &s_abort); break;
            case 4: Apex2<Real, 4>::load_tables(a); ok = apex2_dag_step<Real, 4>(a, pa, tent, &s_abort); break;
            default: Apex2<Real, 5>::load_tables(a); ok = apex2_dag_step<Real, 5>(a, pa, tent, &s_abort); break;
        }
        if (!ok) break;
    }
}

}  // namespace mtp
