// Navier-Stokes lines of the weak form (Eq. 1 with ivis = 1; Eq. 11's auxiliary-gradient and
// viscous-flux lines in BR1 form, Sec. II-B) on the CUDA cores, in FP64 or FP32 (the mixed forms and
// FP32 without a trace buffer: kernels_ns_mixed.cu).  Three passes after
// the Euler residual, on the traces of U at every face point ([ne][4][5][Nqf], kernels_simt.cu):
//
//   k_ns_grad   the auxiliary gradient Z = grad Q of Eq. 11's first line,
//                 Z_dvj = - sum_k (J^-1)_kd sum_q w_q Q_v(x_q) d_k phi_j
//                         + sum_f n_d s_f sum_q wf_q Qhat_v phi_j,
//               with the orthonormal basis' inverse mass matrix folded into
//               s_f = |grad lambda_f| = 2 |S_f| / |det J|; Qhat = (Q- + Q+) / 2 on interior
//               faces, the no-slip adiabatic wall state Q_b = (rho-, 0, 0, 0, E- - |m-|^2 /
//               (2 rho-)) on walls, Q- on far-field faces.  Integrated by parts (exact: the rules
//               integrate degree 2p): the modes of d_k Q, plus the lift of Qhat - Q-.  Thread per
//               (element, variable) row, the three components at once;
//   k_ns_visc   thread per (element, field) row of the 20 fields U and Z: traces at the face points
//               and values at the volume points, to shared memory; thread per point: F_v . n with
//               the outward normal, to a face buffer HB[ne][4][4][Nqf] (momentum and energy; the
//               mass entry is zero), and the contravariant F_v; thread per (element, equation):
//                 R -= sum_q w_q (J^-1 F_v)_k d_k phi_j;
//   k_ns_lift   the central flux H = (F_v(Q-, Z-) + F_v(Q+, Z+)) . n / 2 from both sides' entries
//               (the neighbour's, at the matching point, has the opposite normal), F_v(Q_b, Z-) . n
//               with a zero energy entry on walls (adiabatic, the wall at rest does no work),
//               F_v(Q-, Z-) . n on far-field faces:
//                 R += sum_f s_f sum_q wf_q H phi_j.
// Each face's viscous flux is evaluated once per side and no element reads a neighbour's
// gradient coefficients.  The result is independent of the launch configuration (fixed
// per-element summation order, no atomics).
//
// FP64 is bound by its pipe (12k operations per P2 element in these passes, 23k with dense tables and
// the weak form of the gradient: 8.0 ms per residual of 196,608 elements); the FP32 form was bound by
// shared-memory loads of tables and coefficients (P3, 96,000 elements: 0.83 ms).
//
// F_v (Eq. 1 restated in 3D), for direction d: (0, tau_1d, tau_2d, tau_3d,
// sum_i u_i tau_id + kappa dT/dx_d), Stokes' hypothesis tau = mu (grad u + grad u^T -
// 2/3 div u I), T = p / rho (gas constant 1), kappa = mu gamma / ((gamma - 1) Pr).  The velocity
// and temperature gradients follow from the conserved gradient Z by the chain rule.
#include <algorithm>

#include "dg_internal.h"
#include "face_flux.cuh"
#include "modal_ops.cuh"

namespace dg {

namespace {

template <typename Real>
struct NSArgs {
    const Real* U;        // [ne][5][Nb] internal order
    const Real* T;        // traces of U [ne][4][5][Nqf]
    Real* Z;              // [ne][3][5][Nb]
    Real* R;              // [ne][5][Nb] Euler residual, the viscous terms are added
    Real* HB;             // [ne][4][4][Nqf] own F_v . n (twice it on boundary faces)
    const int32_t* nbr;     // [ne][4] (boundary faces: -1 - bc type)
    const uint8_t* fcode;   // [ne][4]
    const Real* jinv;     // [ne][9]
    const int8_t* fperm;    // [6][Nqf]
    int64_t ne;
    Real mu, kappa, gamma;
};

// s_f n_f = -grad lambda_f from the row-major J^-1
template <typename Real>
__device__ __forceinline__ void scaled_normal(const Real* I, int f, Real* g) {
#pragma unroll
    for (int d = 0; d < 3; ++d) g[d] = f == 0 ? I[d] + I[3 + d] + I[6 + d] : -I[3 * (f - 1) + d];
}

// TR: the traces come from the buffer T; without it (small P1 meshes) each row evaluates its own and its
// neighbours', 55 multiply-adds a face at most, and the launch that fills the buffer is saved
template <typename Real, int P, int EE, bool TR>
__global__ void __launch_bounds__(threads_of(EE)) k_ns_grad(NSArgs<Real> a) {
    constexpr int NB = nb_of(P), NQF = nqf_of(P), NM = modal::Tables<P>::NM, NF = modal::Tables<P>::NF, NT = threads_of(EE);
    __shared__ Real sJ[EE * 9];
    __shared__ int snbr[EE * 4];
    __shared__ uint8_t sfc[EE * 4];
    __shared__ int8_t sperm[6 * NQF];
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (a.ne - e0) < (int64_t)EE ? (int)(a.ne - e0) : EE;
    for (int i = t; i < nel * 9; i += NT) sJ[i] = a.jinv[e0 * 9 + i];
    for (int i = t; i < nel * 4; i += NT) {
        snbr[i] = a.nbr[e0 * 4 + i];
        sfc[i] = a.fcode[e0 * 4 + i];
    }
    for (int i = t; i < 6 * NQF; i += NT) sperm[i] = a.fperm[i];
    __syncthreads();
    if (t >= 5 * nel) return;
    const int e = t / 5, v = t - 5 * e;
    const Real* I = sJ + 9 * e;
    Real z[3][NB], c[NB];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < NB; ++j) z[d][j] = 0;
    load_row<NB>(a.U + (e0 * 5 + t) * NB, c);
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Real s[NM];
            modal::grad_modes<Real, P>(k, c, s);
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
                for (int m = 0; m < NM; ++m) z[d][m] += I[3 * k + d] * s[m];
        }
    }
    const Real* own = TR ? a.T + (e0 + e) * 20 * NQF : nullptr;
    modal::unroll<0, 4>([&](auto fc) {
        constexpr int f = fc.value;
        // Qhat - Q- at the face's points
        const int n = snbr[4 * e + f];
        Real x[NQF], b[NF], y[NB], g[3];
        if constexpr (TR) load_row<NQF>(own + (f * 5 + v) * NQF, x);
        else modal::face_trace<Real, P, f>(c, x);
        if (n >= 0) {
            const int code = sfc[4 * e + f];
            const int8_t* pm = sperm + (code >> 2) * NQF;
            Real u[TR ? 1 : NQF];
            const Real* o;
            if constexpr (TR) {
                o = a.T + (((int64_t)n * 4 + (code & 3)) * 5 + v) * NQF;
            } else {
                Real cn[NB];
                load_row<NB>(a.U + ((int64_t)n * 5 + v) * NB, cn);
                modal::face_trace<Real, P>(code & 3, cn, u);
                o = u;
            }
#pragma unroll
            for (int q = 0; q < NQF; ++q) x[q] = Real(0.5) * (o[pm[q]] - x[q]);
        } else if (n == -1 - DG_BC_WALL) {
            Real wt[TR ? 1 : 4 * NQF];
            const Real* w;
            if constexpr (TR) {
                w = own + f * 5 * NQF;
            } else {
                if (v == 4)   // density and momenta of the element
                    for (int k = 0; k < 4; ++k) {
                        Real ck[NB];
                        load_row<NB>(a.U + ((e0 + e) * 5 + k) * NB, ck);
                        modal::face_trace<Real, P, f>(ck, wt + k * NQF);
                    }
                else
                    for (int k = 0; k < 4 * NQF; ++k) wt[k] = Real(1);   // unused
                w = wt;
            }
#pragma unroll
            for (int q = 0; q < NQF; ++q) {
                const Real m0 = w[NQF + q], m1 = w[2 * NQF + q], m2 = w[3 * NQF + q];
                x[q] = v == 0 ? Real(0) : v < 4 ? -x[q] : Real(-0.5) * (m0 * m0 + m1 * m1 + m2 * m2) / w[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < NQF; ++q) x[q] = 0;
        }
        modal::face_moments<Real, P>(x, b);
        modal::face_lift<Real, P>(f, b, y);
        scaled_normal(I, f, g);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int j = 0; j < NB; ++j) z[d][j] += g[d] * y[j];
    });
#pragma unroll
    for (int d = 0; d < 3; ++d) store_row<NB>(a.Z + (((e0 + e) * 3 + d) * 5 + v) * NB, z[d]);
}

// F_v . n (momentum, energy) at a point: state U, gradient Z (d-major rows of 5), stride between fields
template <typename Real>
__device__ __forceinline__ void viscous_normal(const Real* U, const Real* Z, const Real* n, Real mu, Real kappa, Real g1, Real* F) {
    const Real ri = recip(U[0]);
    const Real u[3] = {U[1] * ri, U[2] * ri, U[3] * ri}, eh = U[4] * ri;
    Real du[3][3];   // du[i][d] = d u_i / d x_d
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int i = 0; i < 3; ++i) du[i][d] = (Z[5 * d + 1 + i] - u[i] * Z[5 * d]) * ri;
    const Real div = Real(2.0 / 3.0) * (du[0][0] + du[1][1] + du[2][2]);
    const Real r = Z[0] * n[0] + Z[5] * n[1] + Z[10] * n[2], en = Z[4] * n[0] + Z[9] * n[1] + Z[14] * n[2];
    Real w = 0, k = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const Real dn = du[i][0] * n[0] + du[i][1] * n[1] + du[i][2] * n[2];   // d u_i / d n
        const Real tn = du[0][i] * n[0] + du[1][i] * n[1] + du[2][i] * n[2];   // d u_n / d x_i
        F[i] = mu * (dn + tn - div * n[i]);
        w += u[i] * F[i];
        k += u[i] * dn;
    }
    // T = (gamma - 1) (E / rho - |u|^2 / 2)
    F[3] = w + kappa * (g1 * ((en - eh * r) * ri - k));
}

// (J^-1 F_v)_k (momentum, energy) at a point
template <typename Real>
__device__ __forceinline__ void viscous_contravariant(const Real* U, const Real* Z, const Real* I, Real mu, Real kappa, Real g1,
                                                      Real G[3][4]) {
    const Real ri = recip(U[0]);
    const Real u[3] = {U[1] * ri, U[2] * ri, U[3] * ri}, eh = U[4] * ri;
    Real du[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int i = 0; i < 3; ++i) du[i][d] = (Z[5 * d + 1 + i] - u[i] * Z[5 * d]) * ri;
    const Real div = Real(2.0 / 3.0) * (du[0][0] + du[1][1] + du[2][2]);
    Real F[3][4];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int i = 0; i <= d; ++i) F[d][i] = F[i][d] = mu * (i == d ? du[i][d] + du[i][d] - div : du[i][d] + du[d][i]);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const Real dT = g1 * ((Z[5 * d + 4] - eh * Z[5 * d]) * ri - (u[0] * du[0][d] + u[1] * du[1][d] + u[2] * du[2][d]));
        F[d][3] = u[0] * F[d][0] + u[1] * F[d][1] + u[2] * F[d][2] + kappa * dT;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v) G[k][v] = I[3 * k] * F[0][v] + I[3 * k + 1] * F[1][v] + I[3 * k + 2] * F[2][v];
}

constexpr int EV = 8;           // elements per tile of k_ns_visc
constexpr int VT = 20 * EV;     // rows (element, field) = threads

template <typename Real, int P>
struct ViscPlan {
    static constexpr int NQ = nq_of(P), NPF = 4 * nqf_of(P);
    // shared memory (Reals): fields at the face points, then at the volume points [VT][odd stride];
    // contravariant viscous flux [EV][4][NQ][3]; J^-1; unit normals [EV][4][3]
    static constexpr int SF = NPF | 1, SV = NQ | 1;
    static constexpr int G = VT * (SF > SV ? SF : SV), J = G + EV * 12 * NQ, N = J + EV * 9, REALS = N + EV * 12;
    static constexpr size_t BYTES = REALS * sizeof(Real);
};

template <typename Real, int P, bool TR>
__global__ void __launch_bounds__(VT) k_ns_visc(NSArgs<Real> a) {
    using S = ViscPlan<Real, P>;
    constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), NPF = S::NPF, NM = modal::Tables<P>::NM;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* sP = reinterpret_cast<Real*>(smem);
    Real* sG = sP + S::G;
    Real* sJ = sP + S::J;
    Real* sN = sP + S::N;
    __shared__ int snbr[EV * 4];
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EV;
    const int nel = (a.ne - e0) < (int64_t)EV ? (int)(a.ne - e0) : EV;
    const Real mu = a.mu, kappa = a.kappa, g1 = a.gamma - Real(1);
    for (int i = t; i < nel * 9; i += VT) sJ[i] = a.jinv[e0 * 9 + i];
    if (t < nel * 4) snbr[t] = a.nbr[e0 * 4 + t];
    const int e = t / 20, r = t - 20 * e;   // row r: U (5), then Z (15, direction-major)
    const bool live = e < nel;
    Real c[NB];
    if (live) {
        Real* o = sP + t * S::SF;
        if (!TR) {
            load_row<NB>(r < 5 ? a.U + ((e0 + e) * 5 + r) * NB : a.Z + ((e0 + e) * 15 + r - 5) * NB, c);
            modal::traces<Real, P>(c, [&](int f, const Real* u) {
#pragma unroll
                for (int q = 0; q < NQF; ++q) o[f * NQF + q] = u[q];
            });
        } else if (r < 5) {
            load_row<NB>(a.U + ((e0 + e) * 5 + r) * NB, c);
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                Real x[NQF];
                load_row<NQF>(a.T + (((e0 + e) * 4 + f) * 5 + r) * NQF, x);
#pragma unroll
                for (int q = 0; q < NQF; ++q) o[f * NQF + q] = x[q];
            }
        } else {
            load_row<NB>(a.Z + ((e0 + e) * 15 + r - 5) * NB, c);
            modal::traces<Real, P>(c, [&](int f, const Real* u) {
#pragma unroll
                for (int q = 0; q < NQF; ++q) o[f * NQF + q] = u[q];
            });
        }
    }
    __syncthreads();
    if (t < nel * 4) {
        Real g[3];
        scaled_normal(sJ + (t >> 2) * 9, t & 3, g);
        const Real inv = Real(1) / EulerOps<Real>::sqrt_(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
#pragma unroll
        for (int d = 0; d < 3; ++d) sN[3 * t + d] = g[d] * inv;
    }
    __syncthreads();
    // faces: the own viscous flux at every (element, face, point)
    for (int i = t; i < nel * NPF; i += VT) {
        const int el = i / NPF, fq = i - el * NPF, f = fq / NQF, q = fq - f * NQF;
        const Real* x = sP + el * 20 * S::SF + fq;
        Real W[20], F[4];
#pragma unroll
        for (int k = 0; k < 20; ++k) W[k] = x[k * S::SF];
        const int n = snbr[4 * el + f];
        if (n == -1 - DG_BC_WALL) {   // the wall state: interior density and internal energy, at rest
            W[4] -= Real(0.5) * (W[1] * W[1] + W[2] * W[2] + W[3] * W[3]) / W[0];
            W[1] = W[2] = W[3] = 0;
        }
        viscous_normal(W, W + 5, sN + 3 * (4 * el + f), mu, kappa, g1, F);
        if (n < 0) {
            F[3] = n == -1 - DG_BC_WALL ? Real(0) : F[3];
#pragma unroll
            for (int v = 0; v < 4; ++v) F[v] *= Real(2);
        }
        Real* hb = a.HB + ((e0 + el) * 4 + f) * 4 * NQF + q;
#pragma unroll
        for (int v = 0; v < 4; ++v) hb[v * NQF] = F[v];
    }
    __syncthreads();
    // volume: contravariant viscous flux at every (element, point)
    if (live) modal::interpolate<Real, P, NB, 0, NQ>(c, [&](int q, Real u) { sP[t * S::SV + q] = u; });
    __syncthreads();
    for (int i = t; i < nel * NQ; i += VT) {
        const int el = i / NQ, q = i - el * NQ;
        const Real* x = sP + el * 20 * S::SV + q;
        Real W[20], G[3][4];
#pragma unroll
        for (int k = 0; k < 20; ++k) W[k] = x[k * S::SV];
        viscous_contravariant(W, W + 5, sJ + 9 * el, mu, kappa, g1, G);
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int k = 0; k < 3; ++k) sG[((el * 4 + v) * NQ + q) * 3 + k] = G[k][v];
    }
    __syncthreads();
    // projection of the momentum and energy rows: thread per (element, equation)
    if (t >= nel * 4) return;
    Real M[3][NM];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int m = 0; m < NM; ++m) M[k][m] = 0;
    const Real* g = sG + t * NQ * 3;
    modal::unroll<0, NQ>([&](auto qc) {
        constexpr int q = qc.value, m = modal::kT<P>.vmir[q];
        if constexpr (m >= q) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
                modal::moments<Real, P, NM>(q, g[3 * q + k], m != q ? g[3 * m + k] : Real(0), M[k]);
        }
    });
    Real x[NB], y[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) y[j] = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) modal::grad_transposed<Real, P>(k, M[k], y);
    Real* R = a.R + ((e0 + t / 4) * 5 + 1 + (t & 3)) * NB;
    load_row<NB>(R, x);
#pragma unroll
    for (int j = 0; j < NB; ++j) x[j] -= y[j];
    store_row<NB>(R, x);
}

template <typename Real, int P, int EL>
__global__ void __launch_bounds__(4 * EL) k_ns_lift(NSArgs<Real> a) {
    constexpr int NB = nb_of(P), NQF = nqf_of(P), NT = 4 * EL;
    __shared__ int snbr[EL * 4];
    __shared__ uint8_t sfc[EL * 4];
    __shared__ int8_t sperm[6 * NQF];
    __shared__ Real sS[EL * 4];   // s_f / 2
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EL;
    const int nel = (a.ne - e0) < (int64_t)EL ? (int)(a.ne - e0) : EL;
    if (t < 4 * nel) {
        Real g[3];
        scaled_normal(a.jinv + (e0 + (t >> 2)) * 9, t & 3, g);
        sS[t] = Real(0.5) * EulerOps<Real>::sqrt_(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
        snbr[t] = a.nbr[e0 * 4 + t];
        sfc[t] = a.fcode[e0 * 4 + t];
    }
    for (int i = t; i < 6 * NQF; i += NT) sperm[i] = a.fperm[i];
    __syncthreads();
    if (t >= 4 * nel) return;
    const int e = t >> 2, v = t & 3;
    Real* R = a.R + ((e0 + e) * 5 + 1 + v) * NB;
    Real x[NB];
    load_row<NB>(R, x);
    const Real* own = a.HB + ((e0 + e) * 16 + v) * NQF;
    modal::lift<Real, P>(
        [&](int f, Real* h) {
            load_row<NQF>(own + f * 4 * NQF, h);
            const int n = snbr[4 * e + f];
            if (n >= 0) {
                const int code = sfc[4 * e + f];
                const Real* o = a.HB + (((int64_t)n * 4 + (code & 3)) * 4 + v) * NQF;
                const int8_t* pm = sperm + (code >> 2) * NQF;
#pragma unroll
                for (int q = 0; q < NQF; ++q) h[q] -= o[pm[q]];
            }
            return sS[4 * e + f];
        },
        x);
    store_row<NB>(R, x);
}

template <typename Real, int P, bool TR>
cudaError_t ns_launch(const NSArgs<Real>& a, cudaStream_t s) {
    constexpr size_t bytes = ViscPlan<Real, P>::BYTES;
    auto visc = k_ns_visc<Real, P, TR>;
    static bool init = false;
    if (!init) {
        cudaError_t e = cudaFuncSetAttribute(visc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        init = true;
    }
    // one warp per tile: a row holds three gradients' modes in registers
    k_ns_grad<Real, P, 6, TR><<<(unsigned)((a.ne + 5) / 6), threads_of(6), 0, s>>>(a);
    visc<<<(unsigned)((a.ne + EV - 1) / EV), VT, bytes, s>>>(a);
    if (small_tiles(a.ne)) k_ns_lift<Real, P, 8><<<(unsigned)((a.ne + 7) / 8), 32, 0, s>>>(a);
    else k_ns_lift<Real, P, 32><<<(unsigned)((a.ne + 31) / 32), 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

size_t ns_face_buffer_values(int p, int64_t ne) { return (size_t)ne * 4 * nqf_of(p) * 4; }

namespace {
// SSP-RK3 stage update from a stored residual: out = a U0 + b (U + dt R) (a = 0: U0 unread)
template <typename Real>
__global__ void __launch_bounds__(256) k_rk_axpy(const Real* __restrict__ U, const Real* __restrict__ U0,
                                                 const Real* __restrict__ R, Real* out, int64_t n, Real dt, Real a,
                                                 Real b) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        Real r = b * (U[i] + dt * R[i]);
        if (a != Real(0)) r += a * U0[i];
        out[i] = r;
    }
}

// the same update of a float-float state (hi plane, then lo plane) from an FP32 residual, as the
// mixed stage kernel's epilogue forms it: the increment a (U0 - U) + b dt R in FP32, added to
// (hi, lo) with an error-free sum
__global__ void __launch_bounds__(256) k_rk_axpy_ff(const float* __restrict__ U, const float* __restrict__ U0,
                                                    const float* __restrict__ R, float* out, int64_t n, float bdt,
                                                    float a) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float uh = U[i], ul = U[n + i];
        const float dlt = a != 0.f ? fmaf(a, (U0[i] - uh) + (U0[n + i] - ul), bdt * R[i]) : bdt * R[i];
        const float sm = uh + dlt;
        const float bb = sm - uh;
        const float err = ((uh - (sm - bb)) + (dlt - bb)) + ul;
        const float oh = sm + err;
        out[i] = oh;
        out[n + i] = err - (oh - sm);
    }
}

template <typename Real>
cudaError_t ns_dispatch(dg_mesh* m, const void* U, void* T, void* Z, void* HB, void* R, double mu, double prandtl,
                        cudaStream_t s) {
    // FP32 P1 below 6,000 elements: us per residual without | with the launch of the traces, 1,296 elements
    // 40 | 42, 4,374 with boundary faces 40 | 44, 6,000 44 | 44
    const bool rows_only = sizeof(Real) == 4 && m->p == 1 && m->host.ne < 6000;
    cudaError_t e = rows_only ? cudaSuccess : launch_traces2(m, U, T, nullptr, nullptr, s);
    if (e != cudaSuccess) return e;
    NSArgs<Real> a;
    a.U = static_cast<const Real*>(U);
    a.T = static_cast<const Real*>(T);
    a.Z = static_cast<Real*>(Z);
    a.R = static_cast<Real*>(R);
    a.HB = static_cast<Real*>(HB);
    a.nbr = m->d_nbr;
    a.fcode = m->d_fcode;
    a.jinv = static_cast<const Real*>(m->d_jinv);
    a.fperm = m->d_fperm;
    a.ne = m->host.ne;
    a.mu = (Real)mu;
    a.gamma = (Real)m->gamma;
    a.kappa = (Real)(mu * m->gamma / ((m->gamma - 1.0) * prandtl));
    if constexpr (sizeof(Real) == 4)
        if (rows_only) return ns_launch<Real, 1, false>(a, s);
    switch (m->p) {
        case 1: return ns_launch<Real, 1, true>(a, s);
        case 2: return ns_launch<Real, 2, true>(a, s);
        default: return ns_launch<Real, 3, true>(a, s);
    }
}
}  // namespace

cudaError_t launch_rk_axpy(dg_mesh* m, const void* U, const void* U0, const void* R, void* out, double dt, double a,
                           double b, cudaStream_t s) {
    const int64_t n = m->host.ne * 5 * m->nb;
    const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16);
    if (m->precision == DG_FP64)
        k_rk_axpy<double><<<blocks, 256, 0, s>>>(static_cast<const double*>(U), static_cast<const double*>(U0),
                                                 static_cast<const double*>(R), static_cast<double*>(out), n, dt, a, b);
    else if (m->precision == DG_FP32)
        k_rk_axpy<float><<<blocks, 256, 0, s>>>(static_cast<const float*>(U), static_cast<const float*>(U0),
                                                static_cast<const float*>(R), static_cast<float*>(out), n, (float)dt,
                                                (float)a, (float)b);
    else
        k_rk_axpy_ff<<<blocks, 256, 0, s>>>(static_cast<const float*>(U), static_cast<const float*>(U0),
                                            static_cast<const float*>(R), static_cast<float*>(out), n,
                                            (float)(b * dt), (float)a);
    return cudaGetLastError();
}

cudaError_t launch_ns_viscous(dg_mesh* m, const void* U, void* T, void* Z, void* HB, void* R, double mu, double prandtl,
                              cudaStream_t s) {
    if (m->precision == DG_FP64) return ns_dispatch<double>(m, U, T, Z, HB, R, mu, prandtl, s);
    if (m->precision == DG_FP32 && T) return ns_dispatch<float>(m, U, T, Z, HB, R, mu, prandtl, s);
    return launch_ns_viscous_mixed(m, static_cast<const float*>(U), static_cast<float*>(Z), static_cast<float*>(HB),
                                   static_cast<float*>(R), mu, prandtl, s);
}

}  // namespace dg
