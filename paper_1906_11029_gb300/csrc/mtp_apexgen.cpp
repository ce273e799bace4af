// Build-time generator: writes mtp_apex_ops.h, the contractions of the apex tent kernel
// (mtp_apex.cuh) as straight-line code with the reference-table entries as literals.
//
// Every tent element is re-expressed in the Dubiner basis whose collapsed apex is the tent vertex
// V (vertex A of the reference tetrahedron, coordinates x = lambda_D, y = lambda_B,
// z = lambda_A = lambda_V; C, D, B are the element's other vertices in ascending id order).
// In that basis the tables no longer depend on V's local index and most of their entries vanish:
// at p = 4 multiplication by lambda_V has 50 non-zeros of 700, the derivatives along three suitable
// directions 108, 112 and 144 of 700, the trace onto a facet through V 105 of 525, or 105 + 105 in
// two factors.  Only the non-zeros are written out, so a thread needs no table loads and no loop.
//
// A second header, mtp_lattice_ops.h, holds the lattice Vandermonde matrix V and its inverse of
// every dimension and degree in the same form.  Exchanging the element's first two vertices maps
// the lattice onto itself and multiplies a basis function by +-1, so values at mirrored points are
// the sum and the difference of an even and an odd part: 653 multiply-adds instead of 1225 at
// p = 4 in 3D.
#include <cstdio>
#include <string>

#include "mtp_tables.cpp"

using namespace mtp;

namespace {

struct Mat {
    int r = 0, c = 0;
    std::vector<double> v;
    Mat(int rows, int cols) : r(rows), c(cols), v((size_t)rows * cols, 0.0) {}
    double& at(int i, int j) { return v[(size_t)i * c + j]; }
    double at(int i, int j) const { return v[(size_t)i * c + j]; }
    // entries at rounding level are exact zeros of the table
    void clean() {
        double mx = 0;
        for (double x : v) mx = std::fmax(mx, std::fabs(x));
        for (double& x : v)
            if (std::fabs(x) < 1e-13 * mx) x = 0.0;
    }
};

std::string term(double c, const std::string& x) {
    if (c == 1.0) return x;
    char b[96];
    std::snprintf(b, sizeof b, "R(%.17g) * %s", c, x.c_str());
    return b;
}

// y[i] (+)= sum_j A[i][j] x[j], one statement per non-zero, inputs outermost
void emit(FILE* f, const char* name, const Mat& A, bool add) {
    std::fprintf(f, "    template <typename R>\n    static __device__ __forceinline__ void %s(const R* x, R* y) {\n", name);
    std::vector<char> set(A.r, add ? 1 : 0);
    for (int j = 0; j < A.c; ++j)
        for (int i = 0; i < A.r; ++i)
            if (A.at(i, j) != 0.0) {
                std::fprintf(f, "        y[%d] %s %s;\n", i, set[i] ? "+=" : "=", term(A.at(i, j), "x[" + std::to_string(j) + "]").c_str());
                set[i] = 1;
            }
    for (int i = 0; i < A.r; ++i)
        if (!set[i]) std::fprintf(f, "        y[%d] = R(0);\n", i);
    std::fprintf(f, "    }\n");
}

Mat transpose(const Mat& A) {
    Mat B(A.c, A.r);
    for (int i = 0; i < A.r; ++i)
        for (int j = 0; j < A.c; ++j) B.at(j, i) = A.at(i, j);
    return B;
}

void emit_degree(FILE* f, int p) {
    std::vector<int> deg;
    auto psi = dubiner(3, p, &deg);
    auto chi = dubiner(2, p);
    const int nb = (int)psi.size(), nfb = (int)chi.size();
    int nm = 0;
    while (nm < nb && deg[nm] < p) ++nm;
    Mat M(nm, nb);
    for (int c = 0; c < nm; ++c) {
        Poly zc = mul(Poly::var(2), psi[c]);
        for (int b = 0; b < nb; ++b) M.at(c, b) = (double)integrate(mul(zc, psi[b]), 3);
    }
    M.clean();
    // D[c][a] = int psi_c (derivative of psi_a along a direction of reference space)
    auto along = [&](double dx, double dy, double dz) {
        Mat A(nm, nb);
        for (int a = 0; a < nb; ++a) {
            Poly g = add(add(scale(deriv(psi[a], 0), dx), scale(deriv(psi[a], 1), dy)), scale(deriv(psi[a], 2), dz));
            for (int c = 0; c < nm; ++c) A.at(c, a) = (double)integrate(mul(psi[c], g), 3);
        }
        A.clean();
        return A;
    };
    // facet traces in the facet basis with apex V and the other two vertices in ascending order
    auto trace = [&](const Poly& X, const Poly& Y) {
        Mat T(nfb, nb);
        for (int a = 0; a < nb; ++a) {
            Poly t = compose(psi[a], X, Y, Poly::var(1));   // s = (s1, s2), s2 = lambda_V
            for (int c = 0; c < nfb; ++c) T.at(c, a) = (double)integrate(mul(chi[c], t), 2);
        }
        T.clean();
        return T;
    };
    const Poly s1 = Poly::var(0), s2 = Poly::var(1), one = Poly::cst(1), zero;
    const Poly rest = add(add(one, s1, -1), s2, -1);
    Mat T0 = trace(rest, s1);   // opposite C: from D to B
    Mat T1 = trace(zero, s1);   // opposite D: from C to B
    Mat T2 = trace(s1, zero);   // opposite B: from C to D
    Mat Lm(nfb, nfb);
    for (int c = 0; c < nfb; ++c) {
        Poly lc = mul(s2, chi[c]);
        for (int e = 0; e < nfb; ++e) Lm.at(c, e) = (double)integrate(mul(lc, chi[e]), 2);
    }
    Lm.clean();
    // The facets opposite C and D mirror each other (T0 = T1 with odd i negated), and on them the
    // basis separates: T1[(m, n)][(i, j, k)] = A[m][(i, j)] B[(m, n)][(l, k)], l = i + j >= m, with
    // A[m][(0, l)] = 1.  Products go through s[(m, l, k)].
    std::vector<int> ti(3 * nb), tm(2 * nfb);   // (i, j, k) of psi, (m, n) of chi
    {
        int q = 0;
        for (int g = 0; g <= p; ++g)
            for (int i = 0; i <= g; ++i)
                for (int j = 0; i + j <= g; ++j, ++q) { ti[3 * q] = i; ti[3 * q + 1] = j; ti[3 * q + 2] = g - i - j; }
        q = 0;
        for (int g = 0; g <= p; ++g)
            for (int i = 0; i <= g; ++i, ++q) { tm[2 * q] = i; tm[2 * q + 1] = g - i; }
    }
    for (int b = 0; b < nb; ++b)
        for (int c = 0; c < nfb; ++c)
            if (std::fabs(T0.at(c, b) - (ti[3 * b] & 1 ? -1 : 1) * T1.at(c, b)) > 1e-12)
                throw std::runtime_error("facet mirror symmetry violated");
    struct S { int m, l, k; };
    std::vector<S> ss;
    for (int l = 0; l <= p; ++l)
        for (int k = 0; k + l <= p; ++k)
            for (int m = 0; m <= l; ++m) ss.push_back({m, l, k});
    const int ns = (int)ss.size();
    Mat Ae(ns, nb), Ao(ns, nb), Bm(nfb, ns);
    auto find_b = [&](int i, int j, int k) {
        for (int b = 0; b < nb; ++b)
            if (ti[3 * b] == i && ti[3 * b + 1] == j && ti[3 * b + 2] == k) return b;
        return -1;
    };
    for (int q = 0; q < ns; ++q) {
        const S& t = ss[q];
        for (int c = 0; c < nfb; ++c)
            if (tm[2 * c] == t.m) Bm.at(c, q) = T1.at(c, find_b(0, t.l, t.k));
        for (int i = 0; i <= t.l; ++i) {
            // A from the largest entry of its (m, l) block over all (n, k)
            double num = 0, den = 0;
            for (int k = 0; k + t.l <= p; ++k)
                for (int c = 0; c < nfb; ++c)
                    if (tm[2 * c] == t.m && std::fabs(T1.at(c, find_b(0, t.l, k))) > std::fabs(den)) {
                        den = T1.at(c, find_b(0, t.l, k));
                        num = T1.at(c, find_b(i, t.l - i, k));
                    }
            (i & 1 ? Ao : Ae).at(q, find_b(i, t.l - i, t.k)) = i == 0 ? 1.0 : num / den;
        }
    }
    for (int c = 0; c < nfb; ++c)
        for (int b = 0; b < nb; ++b) {
            double v = 0;
            for (int q = 0; q < ns; ++q) v += Bm.at(c, q) * (Ae.at(q, b) + Ao.at(q, b));
            if (std::fabs(v - T1.at(c, b)) > 1e-12) throw std::runtime_error("facet traces do not separate");
        }
    std::fprintf(f, "template <>\nstruct ApexOps<%d> {\n    static constexpr int NS = %d;\n", p, ns);
    emit(f, "mass", M, false);
    emit(f, "lam", Lm, false);
    emit(f, "pair_even", Ae, false);
    emit(f, "pair_odd", Ao, false);
    emit(f, "pair_trace", Bm, false);
    emit(f, "pair_lift", transpose(Bm), false);
    emit(f, "pair_even_t", transpose(Ae), true);
    emit(f, "pair_odd_t", transpose(Ao), true);
    emit(f, "trace2", T2, false);
    emit(f, "lift2", transpose(T2), true);
    emit(f, "vol_ab", transpose(along(0, 1, -1)), true);     // along B - A
    emit(f, "vol_mb", transpose(along(-0.5, 1, 0)), true);   // along B - (C + D) / 2
    emit(f, "vol_cd", transpose(along(1, 0, 0)), true);      // along D - C
    // the same for the adjoint: rows c, and lambda_V transposed
    emit(f, "volt_ab", along(0, 1, -1), false);
    emit(f, "volt_mb", along(-0.5, 1, 0), true);
    emit(f, "volt_cd", along(1, 0, 0), true);
    emit(f, "mass_t", transpose(M), true);
    std::fprintf(f, "};\n\n");
}

void emit_lattice(FILE* f, int d, int p) {
    const RefTables t = build_ref_tables(d, p);
    const int nb = t.nb;
    std::vector<int> pt;                       // integer coordinates, lattice order
    for (int c = 0; c <= (d == 3 ? p : 0); ++c)
        for (int b = 0; b + c <= p; ++b)
            for (int a = 0; a + b + c <= p; ++a) pt.insert(pt.end(), {a, b, c});
    std::vector<int> mirror(nb), sg(nb, 0);
    for (int k = 0; k < nb; ++k)
        for (int l = 0; l < nb; ++l)
            if (pt[3 * l] == p - pt[3 * k] - pt[3 * k + 1] - pt[3 * k + 2] && pt[3 * l + 1] == pt[3 * k + 1] &&
                pt[3 * l + 2] == pt[3 * k + 2])
                mirror[k] = l;
    for (int a = 0; a < nb; ++a)
        for (int k = 0; k < nb; ++k) {
            const double x = t.V[(size_t)k * nb + a], y = t.V[(size_t)mirror[k] * nb + a];
            if (std::fabs(x) < 1e-9) continue;
            const int s = x * y > 0 ? 1 : -1;
            if (std::fabs(x - s * y) > 1e-10 || (sg[a] && sg[a] != s)) throw std::runtime_error("lattice mirror symmetry violated");
            sg[a] = s;
        }
    auto lit = [](double v) {
        char b[40];
        std::snprintf(b, sizeof b, "%.17g", v);
        return std::string(b);
    };
    std::fprintf(f, "template <>\nstruct LatticeOps<%d, %d> {\n", d, p);
    std::fprintf(f, "    template <typename Put>\n    static __device__ __forceinline__ void to(const double* x, Put put) {\n        double e, o;\n");
    for (int k = 0; k < nb; ++k) {
        if (mirror[k] < k) continue;
        std::string e, o;
        for (int a = 0; a < nb; ++a) {
            const double v = t.V[(size_t)k * nb + a];
            if (std::fabs(v) < 1e-13) continue;
            std::string& s = sg[a] > 0 ? e : o;
            s = s.empty() ? lit(v) + " * x[" + std::to_string(a) + "]" : "__fma_rn(" + lit(v) + ", x[" + std::to_string(a) + "], " + s + ")";
        }
        if (mirror[k] == k) {
            std::fprintf(f, "        put(%d, %s);\n", k, e.c_str());
        } else {
            std::fprintf(f, "        e = %s;\n        o = %s;\n        put(%d, e + o);\n        put(%d, e - o);\n", e.c_str(), o.c_str(), k, mirror[k]);
        }
    }
    std::fprintf(f, "    }\n    template <typename Put>\n    static __device__ __forceinline__ void from(double* v, Put put) {\n        double t;\n");
    for (int k = 0; k < nb; ++k)               // sums in place of the first, differences of the second
        if (mirror[k] > k)
            std::fprintf(f, "        t = v[%d] - v[%d];\n        v[%d] += v[%d];\n        v[%d] = t;\n", k, mirror[k], k, mirror[k], mirror[k]);
    for (int a = 0; a < nb; ++a) {
        std::string s;
        for (int k = 0; k < nb; ++k) {
            if (mirror[k] < k || (sg[a] < 0 && mirror[k] == k)) continue;
            const double w = t.Vinv[(size_t)a * nb + k], w2 = t.Vinv[(size_t)a * nb + mirror[k]];
            const double c = mirror[k] == k ? w : 0.5 * (w + sg[a] * w2);
            const std::string x = "v[" + std::to_string(sg[a] > 0 ? k : mirror[k]) + "]";
            s = s.empty() ? lit(c) + " * " + x : "__fma_rn(" + lit(c) + ", " + x + ", " + s + ")";
        }
        std::fprintf(f, "        put(%d, %s);\n", a, s.c_str());
    }
    std::fprintf(f, "    }\n};\n\n");
}

}  // namespace

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    FILE* f = std::fopen(argv[1], "w");
    if (!f) return 1;
    std::fprintf(f, "// generated by mtp_apexgen.cpp\n#pragma once\n\nnamespace mtp {\n\ntemplate <int P>\nstruct ApexOps;\n\n");
    for (int p = 1; p <= 4; ++p) emit_degree(f, p);
    std::fprintf(f, "}  // namespace mtp\n");
    if (std::fclose(f)) return 1;
    f = std::fopen(argv[2], "w");
    if (!f) return 1;
    std::fprintf(f, "// generated by mtp_apexgen.cpp\n#pragma once\n\nnamespace mtp {\n\ntemplate <int DIM, int P>\nstruct LatticeOps;\n\n");
    for (int d = 2; d <= 3; ++d)
        for (int p = 1; p <= kMaxDegree; ++p) emit_lattice(f, d, p);
    std::fprintf(f, "}  // namespace mtp\n");
    return std::fclose(f) ? 1 : 0;
}
