// Modal operators of one scalar field on one element, held in a thread's registers: volume
// interpolation, projection on the basis gradients, face traces and face lift of Eq. 11's
// discretisation, with every table entry a compile-time constant (no table is loaded at run time).
//
// The dense operators are factored, so that the FP64 form, which the FP64 pipe bounds (2 lanes a
// clock and SM), executes about half their multiply-adds.  Multiply-adds per field, dense -> here:
//
//                                            P1          P2          P3
//   volume interpolation                   16 -> 13   140 -> 90    480 -> 280
//   projection on the gradients            48 -> 16   420 -> 155  1440 -> 592
//   traces at the 4 faces' points          48 -> 55   240 -> 180   960 -> 513
//   lift of the 4 faces                    48 -> 55   240 -> 180   960 -> 513
//
//   * Swap symmetry.  Exchanging vertices 0 and 1 multiplies mode (i, j, k) by (-1)^i and maps the
//     fully symmetric rules onto themselves: values at a point and at its mirror point are the sum
//     and the difference of the even and the odd modes' parts.
//   * Gradients.  d_k phi_j = sum_m D_k[m][j] phi_m over the modes m of degree <= p - 1, so the flux
//     is projected on those (a half to a quarter of the modes), then D_k^T (sparse) is applied.
//   * Faces.  The restriction of phi_j to face f is sum_m E_f[m][j] psi_m in an orthonormal basis
//     psi of degree <= p on the triangle (the 2D counterpart of the element's basis, with its own
//     swap symmetry); the E_f are sparse, and E_0[m][j] = (-1)^i E_1[m][j] by the swap, so faces 0
//     and 1 share their sums.
//
// Sums over modes start from the highest, so that the mean, the largest term, is added last.
//
// D and E are moments taken with the rules themselves (both integrands have degree <= 2p, which
// the rules integrate exactly); entries that vanish identically are exact zeros and cost nothing.
#pragma once

#include <type_traits>
#include <utility>

#include "dg_device.h"
#include "tc_ops.cuh"

namespace dg {
namespace modal {

constexpr double csqrt(double x) {
    double s = x > 1.0 ? x : 1.0;
    for (int i = 0; i < 64; ++i) s = 0.5 * (s + x / s);
    return s;
}
constexpr double cabs(double x) { return x < 0 ? -x : x; }
constexpr double cpow(double x, int n) {
    double r = 1.0;
    for (int i = 0; i < n; ++i) r *= x;
    return r;
}

// Jacobi P_n^(al,be)(x), three-term recurrence
constexpr double cjacobi(int n, double al, double be, double x) {
    if (n == 0) return 1.0;
    double p0 = 1.0, p1 = 0.5 * ((al + be + 2.0) * x + (al - be));
    for (int k = 2; k <= n; ++k) {
        const double s = 2.0 * k + al + be;
        const double p2 = (((s - 1.0) * (al * al - be * be) + (s - 2.0) * (s - 1.0) * s * x) * p1 -
                           2.0 * (k + al - 1.0) * (k + be - 1.0) * s * p0) / (2.0 * k * (k + al + be) * (s - 2.0));
        p0 = p1;
        p1 = p2;
    }
    return p1;
}
// its derivative for be = 0
constexpr double cjacobi_d(int n, double al, double x) {
    return n == 0 ? 0.0 : 0.5 * (n + al + 1.0) * cjacobi(n - 1, al + 1.0, 1.0, x);
}

// Orbits of the symmetric rules exact to degree 2p (weights sum to 1/6 and 1/2): parameters v, the
// pattern of value indices over the barycentrics, weight.  A rule's points are the distinct
// permutations of each pattern in lexicographic order, the order of the host's tables.
struct Orbit {
    double v[3];
    int pat[4];
    double w;
};
template <int P> struct Rules;
template <> struct Rules<1> {
    static constexpr int NT = 1, NF = 1;
    static constexpr Orbit tet[NT] = {{{0.1381966011250105, 0.5854101966249685, 0}, {0, 0, 0, 1}, 1.0 / 24.0}};
    static constexpr Orbit tri[NF] = {{{1.0 / 6.0, 2.0 / 3.0, 0}, {0, 0, 1, 0}, 1.0 / 6.0}};
};
template <> struct Rules<2> {
    static constexpr int NT = 3, NF = 2;
    static constexpr Orbit tet[NT] = {{{0.09273525031089122, 0.7217942490673264, 0}, {0, 0, 0, 1}, 0.012248840519393659},
                                      {{0.3108859192633006, 0.06734224221009821, 0}, {0, 0, 0, 1}, 0.018781320953002643},
                                      {{0.04550370412564965, 0.45449629587435036, 0}, {0, 0, 1, 1}, 0.007091003462846911}};
    static constexpr Orbit tri[NF] = {{{0.4459484909159649, 0.10810301816807022, 0}, {0, 0, 1, 0}, 0.11169079483900574},
                                      {{0.09157621350977074, 0.8168475729804585, 0}, {0, 0, 1, 0}, 0.054975871827660935}};
};
template <> struct Rules<3> {
    static constexpr int NT = 4, NF = 3;
    static constexpr Orbit tet[NT] = {{{0.214602871259152, 0.356191386222544, 0}, {0, 0, 0, 1}, 0.006653791709694585},
                                      {{0.04067395853461136, 0.877978124396166, 0}, {0, 0, 0, 1}, 0.0016795351758867741},
                                      {{0.32233789014227554, 0.03298632957317338, 0}, {0, 0, 0, 1}, 0.009226196923942453},
                                      {{0.06366100187501753, 0.2696723314583158, 0.6030056647916491}, {0, 0, 1, 2}, 0.008035714285714285}};
    static constexpr Orbit tri[NF] = {{{0.2492867451709104, 0.5014265096581791, 0}, {0, 0, 1, 0}, 0.0583931378631897},
                                      {{0.06308901449150223, 0.8738219710169955, 0}, {0, 0, 1, 0}, 0.02542245318510341},
                                      {{0.05314504984481694, 0.3103524510337844, 0.6365024991213987}, {0, 1, 2, 0}, 0.04142553780918678}};
};

// the distinct permutations of a pattern of n value indices, lexicographically; returns the count
constexpr int permutations(const int* pat, int n, int (*out)[4]) {
    int want[3] = {0, 0, 0}, total = 1, k = 0;
    for (int i = 0; i < n; ++i) {
        ++want[pat[i]];
        total *= 3;
    }
    for (int c = 0; c < total; ++c) {
        int d[4] = {0, 0, 0, 0}, have[3] = {0, 0, 0}, t = c;
        for (int i = n - 1; i >= 0; --i) {
            d[i] = t % 3;
            ++have[d[i]];
            t /= 3;
        }
        if (have[0] != want[0] || have[1] != want[1] || have[2] != want[2]) continue;
        for (int i = 0; i < 4; ++i) out[k][i] = d[i];
        ++k;
    }
    return k;
}

template <int P>
struct Tables {
    static constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P);
    static constexpr int NM = P * (P + 1) * (P + 2) / 6;   // modes of degree <= P - 1 (the first NM)
    static constexpr int NF = (P + 1) * (P + 2) / 2;       // face modes
    double phi[NQ][NB]{};        // basis at the volume points
    double w[NQ]{};
    double D[3][NM][NB]{};       // d_k phi_j = sum_m D[k][m][j] phi_m
    double psi[NQF][NF]{};       // face basis at the face points
    double wf[NQF]{};
    double E[4][NF][NB]{};       // phi_j on face f = sum_m E[f][m][j] psi_m
    bool odd[NB]{};              // parity of the modes under the swap of vertices 0 and 1
    bool fodd[NF]{};             // of the face modes under the swap of the face's first two vertices
    int vmir[NQ]{};              // mirror point of a volume point, of a face point
    int fmir[NQF]{};
    int vpair[NQ]{};             // number of a volume point's mirror pair, counted by its lower point

    static constexpr double chop(double x) { return cabs(x) < 1e-13 ? 0.0 : x; }

    // element basis and reference gradient at barycentrics l
    static constexpr void basis(const double* l, double* f, double* g) {
        const double x = l[1], y = l[2], z = l[3], A = l[0] + l[1], B = 1.0 - z;
        const double a = (x - l[0]) / A, b = 2.0 * y / B - 1.0, c = 2.0 * z - 1.0;
        int n = 0;
        for (int d = 0; d <= P; ++d)
            for (int i = 0; i <= d; ++i)
                for (int j = 0; i + j <= d; ++j, ++n) {
                    const int k = d - i - j;
                    const double q = 2.0 * i + 1.0, r = 2.0 * i + 2.0 * j + 2.0;
                    // unit norm: the Jacobi factors' norms 2^(al+1) / (2n + al + 1)
                    const double s = 8.0 * cpow(2.0, 2 * i + j) *
                                     csqrt((2.0 * i + 1.0) / 2.0 * ((2.0 * j + q + 1.0) / cpow(2.0, 2 * i + 2)) *
                                           ((2.0 * k + r + 1.0) / cpow(2.0, 2 * i + 2 * j + 3)));
                    const double p1 = cjacobi(i, 0.0, 0.0, a), p2 = cjacobi(j, q, 0.0, b), p3 = cjacobi(k, r, 0.0, c);
                    const double d1 = cjacobi_d(i, 0.0, a), d2 = cjacobi_d(j, q, b), d3 = cjacobi_d(k, r, c);
                    const double f1 = p1 * cpow(A, i), f2 = p2 * cpow(B, j);
                    f[n] = s * f1 * f2 * p3;
                    if (!g) continue;
                    const double Ai = i > 0 ? cpow(A, i - 1) : 0.0, Bj = j > 0 ? cpow(B, j - 1) : 0.0;
                    const double f1x = 2.0 * d1 * Ai, f1y = (d1 * (1.0 + a) - i * p1) * Ai;   // f1y: d/dy = d/dz
                    const double f2y = 2.0 * d2 * Bj, f2z = (d2 * (1.0 + b) - j * p2) * Bj;
                    g[3 * n] = s * f1x * f2 * p3;
                    g[3 * n + 1] = s * (f1y * f2 + f1 * f2y) * p3;
                    g[3 * n + 2] = s * ((f1y * f2 + f1 * f2z) * p3 + 2.0 * f1 * f2 * d3);
                }
    }

    constexpr Tables() {
        double bary[NQ][4]{}, fb[NQF][4]{}, grad[NQ][3 * NB]{};
        int q = 0;
        for (int o = 0; o < Rules<P>::NT; ++o) {
            int pm[12][4]{};
            const int n = permutations(Rules<P>::tet[o].pat, 4, pm);
            for (int i = 0; i < n; ++i, ++q) {
                for (int d = 0; d < 4; ++d) bary[q][d] = Rules<P>::tet[o].v[pm[i][d]];
                w[q] = Rules<P>::tet[o].w;
                for (int j = 0; j < n; ++j)
                    if (pm[j][0] == pm[i][1] && pm[j][1] == pm[i][0] && pm[j][2] == pm[i][2] && pm[j][3] == pm[i][3])
                        vmir[q] = q - i + j;
            }
        }
        q = 0;
        for (int o = 0; o < Rules<P>::NF; ++o) {
            int pm[12][4]{};
            const int n = permutations(Rules<P>::tri[o].pat, 3, pm);
            for (int i = 0; i < n; ++i, ++q) {
                for (int d = 0; d < 3; ++d) fb[q][d] = Rules<P>::tri[o].v[pm[i][d]];
                wf[q] = Rules<P>::tri[o].w;
                for (int j = 0; j < n; ++j)
                    if (pm[j][0] == pm[i][1] && pm[j][1] == pm[i][0] && pm[j][2] == pm[i][2]) fmir[q] = q - i + j;
            }
        }
        int n = 0;
        for (int d = 0; d <= P; ++d)
            for (int i = 0; i <= d; ++i)
                for (int j = 0; i + j <= d; ++j) odd[n++] = i % 2 == 1;
        for (q = 0, n = 0; q < NQ; ++q) vpair[q] = vmir[q] < q ? vpair[vmir[q]] : n++;
        for (q = 0; q < NQ; ++q) basis(bary[q], phi[q], grad[q]);
        for (int k = 0; k < 3; ++k)
            for (int m = 0; m < NM; ++m)
                for (int j = 0; j < NB; ++j) {
                    double s = 0.0;
                    for (q = 0; q < NQ; ++q) s += w[q] * phi[q][m] * grad[q][3 * j + k];
                    D[k][m][j] = chop(s);
                }
        n = 0;
        for (int d = 0; d <= P; ++d)
            for (int i = 0; i <= d; ++i, ++n) {
                fodd[n] = i % 2 == 1;
                double nn = 0.0;
                for (q = 0; q < NQF; ++q) {
                    const double A = fb[q][0] + fb[q][1];
                    psi[q][n] = cjacobi(i, 0.0, 0.0, (fb[q][1] - fb[q][0]) / A) * cpow(A, i) *
                                cjacobi(d - i, 2.0 * i + 1.0, 0.0, 2.0 * fb[q][2] - 1.0);
                    nn += wf[q] * psi[q][n] * psi[q][n];
                }
                for (q = 0; q < NQF; ++q) psi[q][n] /= csqrt(nn);
            }
        for (int f = 0; f < 4; ++f) {
            double pf[NQF][NB]{};
            for (q = 0; q < NQF; ++q) {
                double l[4] = {0, 0, 0, 0};
                for (int m = 0; m < 3; ++m) l[m < f ? m : m + 1] = fb[q][m];
                basis(l, pf[q], nullptr);
            }
            for (int m = 0; m < NF; ++m)
                for (int j = 0; j < NB; ++j) {
                    double s = 0.0;
                    for (q = 0; q < NQF; ++q) s += wf[q] * psi[q][m] * pf[q][j];
                    E[f][m][j] = chop(s);
                }
        }
    }
};

template <int P> static __device__ constexpr Tables<P> kT{};

// f(integral_constant First), ..., f(integral_constant Last - 1): a loop whose index stays a constant
// however large the body is (where a nest is too large for the compiler's unrolling, table entries
// would become loads and conversions)
template <int First, typename F, int... I>
__device__ __forceinline__ void unroll_seq(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, First + I>()), ...);
}
template <int First, int Last, typename F>
__device__ __forceinline__ void unroll(F&& f) {
    unroll_seq<First>(f, std::make_integer_sequence<int, Last - First>());
}

// a b + c: in FP64 one rounding by definition, since kernels that must agree bitwise share the expression (in
// FP32 left to the compiler, which needs fewer registers for it)
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float madd(float a, float b, float c) { return a * b + c; }

// r += c x with a compile-time constant; nothing where it is zero
template <typename Real>
__device__ __forceinline__ void axpy(Real& r, double c, Real x) {
    if (c != 0.0) r += (Real)c * x;
}

// values at the volume points Q0 .. Q1 - 1 (a range closed under the mirror) of a field of the first N
// modes, store(q, sum_j c[j] phi_j(x_q)); of PARTS shares of the points, share PART
template <typename Real, int P, int N, int Q0, int Q1, int PART = 0, int PARTS = 1, typename Store>
__device__ __forceinline__ void interpolate(const Real* c, Store store) {
    unroll<Q0, Q1>([&](auto qc) {
        constexpr auto& T = kT<P>;
        constexpr int q = qc.value, m = T.vmir[q];
        if constexpr (m >= q && T.vpair[q] % PARTS == PART) {
            Real e = 0, o = 0;
#pragma unroll
            for (int j = N - 1; j >= 0; --j) {
                if (!T.odd[j]) axpy(e, T.phi[q][j], c[j]);
                else if (m != q) axpy(o, T.phi[q][j], c[j]);
            }
            if constexpr (m == q) {
                store(q, e);
            } else {
                store(q, e + o);
                store(m, e - o);
            }
        }
    });
}

// S[m] += sum over the point q and its mirror point of w phi_m g, for the modes of degree <= p - 1
// (N = NM) or all (N = NB); q is the lower of the two
template <typename Real, int P, int N>
__device__ __forceinline__ void moments(int q, Real g, Real gm, Real* S) {
    constexpr auto& T = kT<P>;
    const bool pair = T.vmir[q] != q;
    const Real s = pair ? g + gm : g, d = g - gm;
#pragma unroll
    for (int m = 0; m < N; ++m) {
        if (!T.odd[m]) axpy(S[m], T.w[q] * T.phi[q][m], s);
        else if (pair) axpy(S[m], T.w[q] * T.phi[q][m], d);
    }
}

// r[j] += sum_m D_k[m][j] S[m]
template <typename Real, int P>
__device__ __forceinline__ void grad_transposed(int k, const Real* S, Real* r) {
    constexpr auto& T = kT<P>;
#pragma unroll
    for (int m = 0; m < T.NM; ++m)
#pragma unroll
        for (int j = 0; j < T.NB; ++j) axpy(r[j], T.D[k][m][j], S[m]);
}

// s[m] = sum_j D_k[m][j] c[j]: the coefficients of d_k of the field
template <typename Real, int P>
__device__ __forceinline__ void grad_modes(int k, const Real* c, Real* s) {
    constexpr auto& T = kT<P>;
#pragma unroll
    for (int m = 0; m < T.NM; ++m) {
        s[m] = 0;
#pragma unroll
        for (int j = 0; j < T.NB; ++j) axpy(s[m], T.D[k][m][j], c[j]);
    }
}

// values at a face's points from its face modes, u[q] = sum_m a[m] psi_m(q)
template <typename Real, int P>
__device__ __forceinline__ void face_values(const Real* a, Real* u) {
    constexpr auto& T = kT<P>;
#pragma unroll
    for (int q = 0; q < T.NQF; ++q) {
        const int n = T.fmir[q];
        if (n < q) continue;
        Real e = 0, o = 0;
#pragma unroll
        for (int m = T.NF - 1; m >= 0; --m) {
            if (!T.fodd[m]) axpy(e, T.psi[q][m], a[m]);
            else if (n != q) axpy(o, T.psi[q][m], a[m]);
        }
        if (n == q) {
            u[q] = e;
        } else {
            u[q] = e + o;
            u[n] = e - o;
        }
    }
}

// b[m] = sum_q wf_q psi_m(q) h[q]
template <typename Real, int P>
__device__ __forceinline__ void face_moments(const Real* h, Real* b) {
    constexpr auto& T = kT<P>;
#pragma unroll
    for (int m = 0; m < T.NF; ++m) b[m] = 0;
#pragma unroll
    for (int q = 0; q < T.NQF; ++q) {
        const int n = T.fmir[q];
        if (n < q) continue;
        const Real s = n != q ? h[q] + h[n] : h[q], d = h[q] - h[n];
#pragma unroll
        for (int m = 0; m < T.NF; ++m) {
            if (!T.fodd[m]) axpy(b[m], T.wf[q] * T.psi[q][m], s);
            else if (n != q) axpy(b[m], T.wf[q] * T.psi[q][m], d);
        }
    }
}

// y[j] = sum_m E_f[m][j] b[m]: face f's lift of its moments
template <typename Real, int P>
__device__ __forceinline__ void face_lift(int f, const Real* b, Real* y) {
    constexpr auto& T = kT<P>;
#pragma unroll
    for (int j = 0; j < T.NB; ++j) y[j] = 0;
#pragma unroll
    for (int m = 0; m < T.NF; ++m)
#pragma unroll
        for (int j = 0; j < T.NB; ++j) axpy(y[j], T.E[f][m][j], b[m]);
}

// traces at the points of the 4 faces; store(f, u) receives each face's NQF values
template <typename Real, int P, typename Store>
__device__ __forceinline__ void traces(const Real* c, Store store) {
    constexpr auto& T = kT<P>;
    Real u[T.NQF];
    {
        Real a[T.NF], b[T.NF];   // faces 1 and 0 share the even and the odd modes' sums
#pragma unroll
        for (int m = 0; m < T.NF; ++m) {
            Real e = 0, o = 0;
#pragma unroll
            for (int j = T.NB - 1; j >= 0; --j) axpy(T.odd[j] ? o : e, T.E[1][m][j], c[j]);
            a[m] = e - o;
            b[m] = e + o;
        }
        face_values<Real, P>(a, u);
        store(0, u);
        face_values<Real, P>(b, u);
        store(1, u);
    }
#pragma unroll
    for (int f = 2; f < 4; ++f) {
        Real a[T.NF];
#pragma unroll
        for (int m = 0; m < T.NF; ++m) {
            a[m] = 0;
#pragma unroll
            for (int j = T.NB - 1; j >= 0; --j) axpy(a[m], T.E[f][m][j], c[j]);
        }
        face_values<Real, P>(a, u);
        store(f, u);
    }
}

// the trace at the points of face F alone, with the sums of traces()
template <typename Real, int P, int F>
__device__ __forceinline__ void face_trace(const Real* c, Real* u) {
    constexpr auto& T = kT<P>;
    Real a[T.NF];
#pragma unroll
    for (int m = 0; m < T.NF; ++m) {
        if constexpr (F < 2) {
            Real e = 0, o = 0;
#pragma unroll
            for (int j = T.NB - 1; j >= 0; --j) axpy(T.odd[j] ? o : e, T.E[1][m][j], c[j]);
            a[m] = F == 0 ? e - o : e + o;
        } else {
            a[m] = 0;
#pragma unroll
            for (int j = T.NB - 1; j >= 0; --j) axpy(a[m], T.E[F][m][j], c[j]);
        }
    }
    face_values<Real, P>(a, u);
}
template <typename Real, int P>
__device__ __forceinline__ void face_trace(int f, const Real* c, Real* u) {
    if (f == 0) face_trace<Real, P, 0>(c, u);
    else if (f == 1) face_trace<Real, P, 1>(c, u);
    else if (f == 2) face_trace<Real, P, 2>(c, u);
    else face_trace<Real, P, 3>(c, u);
}

// r[j] += sum_f sum_q wf_q h_f(q) phi_j on face f; load(f, h) fills a face's NQF values and returns
// a factor of the face, which multiplies its moments
template <typename Real, int P, typename Load>
__device__ __forceinline__ void lift(Load load, Real* r) {
    constexpr auto& T = kT<P>;
    Real h[T.NQF];
    {
        Real a[T.NF], b[T.NF];
        const Real s0 = load(0, h);
        face_moments<Real, P>(h, a);
        const Real s1 = load(1, h);
        face_moments<Real, P>(h, b);
#pragma unroll
        for (int m = 0; m < T.NF; ++m) {
            const Real x = s0 * a[m], e = madd(s1, b[m], x), o = madd(s1, b[m], -x);
#pragma unroll
            for (int j = 0; j < T.NB; ++j) axpy(r[j], T.E[1][m][j], T.odd[j] ? o : e);
        }
    }
#pragma unroll
    for (int f = 2; f < 4; ++f) {
        Real a[T.NF];
        const Real s = load(f, h);
        face_moments<Real, P>(h, a);
#pragma unroll
        for (int m = 0; m < T.NF; ++m) {
            const Real x = s * a[m];
#pragma unroll
            for (int j = 0; j < T.NB; ++j) axpy(r[j], T.E[f][m][j], x);
        }
    }
}

}  // namespace modal

// ---- rows and tiles -------------------------------------------------------------------------------

// The CUDA-core kernels work on tiles of EE consecutive elements, thread per (element, variable) row:
// 32 elements (five full warps), or 6 (30 rows of one warp) on a mesh whose tiles of 32 would not
// give every SM two: 10 SSP-RK3 steps of 1,296 P1 elements in FP64 617 -> 542 us; on 196,608 P3
// elements 6 would cost 4% (17.4 -> 18.1 ms per step).  An element's arithmetic does not depend on EE.
constexpr int rows_of(int ee) { return 5 * ee; }
constexpr int threads_of(int ee) { return (5 * ee + 31) / 32 * 32; }
inline bool small_tiles(int64_t ne) { return ne < 32 * 2 * 152; }

// n bytes of a tile, global -> shared, by all NT threads (asynchronous, 16 bytes each; n rounded up:
// the buffers end in slack)
template <int NT>
__device__ __forceinline__ void copy_tile(void* dst, const void* src, int n) {
    for (int i = threadIdx.x * 16; i < n; i += NT * 16)
        tc::cp_async16(static_cast<char*>(dst) + i, static_cast<const char*>(src) + i);
    tc::cp_async_commit();
}

// the values of one contiguous row, in the widest accesses its alignment allows
template <int N, typename Real>
__device__ __forceinline__ void load_row(const Real* __restrict__ p, Real* x) {
    constexpr int B = N * (int)sizeof(Real);
    if constexpr (B % 16 == 0) {
        constexpr int V = 16 / sizeof(Real);
#pragma unroll
        for (int i = 0; i < N / V; ++i) {
            const float4 t = reinterpret_cast<const float4*>(p)[i];
            const Real* r = reinterpret_cast<const Real*>(&t);
#pragma unroll
            for (int k = 0; k < V; ++k) x[i * V + k] = r[k];
        }
    } else if constexpr (B % 8 == 0) {
        constexpr int V = 8 / sizeof(Real);
#pragma unroll
        for (int i = 0; i < N / V; ++i) {
            const float2 t = reinterpret_cast<const float2*>(p)[i];
            const Real* r = reinterpret_cast<const Real*>(&t);
#pragma unroll
            for (int k = 0; k < V; ++k) x[i * V + k] = r[k];
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] = p[i];
    }
}
template <int N, typename Real>
__device__ __forceinline__ void store_row(Real* p, const Real* x) {
    constexpr int B = N * (int)sizeof(Real);
    if constexpr (B % 16 == 0) {
        constexpr int V = 16 / sizeof(Real);
#pragma unroll
        for (int i = 0; i < N / V; ++i) {
            float4 t;
            Real* r = reinterpret_cast<Real*>(&t);
#pragma unroll
            for (int k = 0; k < V; ++k) r[k] = x[i * V + k];
            reinterpret_cast<float4*>(p)[i] = t;
        }
    } else if constexpr (B % 8 == 0) {
        constexpr int V = 8 / sizeof(Real);
#pragma unroll
        for (int i = 0; i < N / V; ++i) {
            float2 t;
            Real* r = reinterpret_cast<Real*>(&t);
#pragma unroll
            for (int k = 0; k < V; ++k) r[k] = x[i * V + k];
            reinterpret_cast<float2*>(p)[i] = t;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = x[i];
    }
}

}  // namespace dg
