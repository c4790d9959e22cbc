// Adjoint of the residual: out = (dR/dU)^T lambda (FP64 / FP32, CUDA cores).
// The paper has no adjoint; this is the reverse of the forward kernels' steps, in the same three
// launches with every face once:
//   k_traces       (kernels_simt.cu) the traces of U and of lambda at the points of every face, to
//                  two face buffers;
//   k_faces_vjp    thread per (interior face, point): the flux H(U_owner, U_other, n_owner) enters the
//                  owner's residual with -s wf and the other's with +s' wf, so its cotangent is
//                  s' lambda_other - s lambda_owner (wf is applied by the lift below); one reverse
//                  sweep gives both states' adjoints, written over the traces of U.  At a kink, where
//                  the two residuals take different branches, a sweep for each;
//   k_bfaces_vjp   the same on boundary faces, through the ghost state (dual numbers: few faces); on small FP32
//                  meshes both in one launch, k_allfaces_vjp;
//   k_element_vjp  tiles of 32 elements, thread per (element, variable) row: U and the three
//                  derivatives of lambda at the volume points; thread per (element, point): the
//                  reverse of the contravariant Euler flux; rows again: the transposed interpolation,
//                  the lift of the face adjoints, and the epilogue
//                  out = c0 X + c1 Y + c2 Z + c3 (dR/dU)^T lambda.
// FP64 is bound by the FP64 pipe.  Before, each side of each face differentiated two fluxes in forward
// mode (5 tangents each) between dense contractions: one P2 Rusanov VJP of 196,608 elements took
// 13.4 ms.
#include <algorithm>
#include <type_traits>

#include "dg_internal.h"
#include "dual.cuh"
#include "face_flux.cuh"
#include "modal_ops.cuh"

namespace dg {

namespace {

constexpr int NT = 256;

// ---- FP32 without face buffers: each element differentiates its faces from both sides in forward
// mode; used only where there is no room for the face buffers

template <int P> struct VTile;
template <> struct VTile<1> { static constexpr int EPB = 16; };
template <> struct VTile<2> { static constexpr int EPB = 8; };
template <> struct VTile<3> { static constexpr int EPB = 4; };

template <typename Real, int P>
struct VPlan {
    static constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), EPB = VTile<P>::EPB;
    static constexpr int PHIQ = 0, DPHIW = NB * NQ, PHIF = DPHIW + 3 * NQ * NB, PHIFW = PHIF + 4 * NB * NQF,
                         WQ = PHIFW + 4 * NQF * NB, TAB = WQ + NQ;
    static constexpr int COWN = EPB * 5 * NB;          // U_e, lambda_e each
    static constexpr int CNBR = EPB * 4 * 5 * NB;      // U_n, lambda_n each
    static constexpr int UBV = EPB * 5 * NQ;           // volume point adjoints
    static constexpr int UBF = EPB * 4 * 5 * NQF;      // face point adjoints (own point order)
    static constexpr int GEO = EPB * 4 * 8;            // own n(3), s; neighbour n(3), s
    static constexpr int JI = EPB * 9;
    static constexpr int REALS = TAB + 2 * COWN + 2 * CNBR + UBV + UBF + GEO + JI;
    static constexpr size_t BYTES = REALS * sizeof(Real) + EPB * 4 * sizeof(int) + EPB * 4 + 6 * NQF + 16;
};

template <typename Real>
struct VjpArgs {
    const Real* U;
    const Real* lam;
    const Real *X, *Y, *Z;   // epilogue vectors (nullable)
    Real c0, c1, c2, c3;
    Real* out;
    const int32_t* nbr;
    const uint8_t* fcode;
    const Real* jinv;
    const Real* tab;
    const int8_t* fperm;
    int64_t ne;
    Real gamma, roe_eps;
    Real finf[5];
};

template <typename Real>
__device__ __forceinline__ void face_grad(const Real* I, int f, Real& g0, Real& g1, Real& g2) {
    if (f == 0) {
        g0 = -(I[0] + I[3] + I[6]);
        g1 = -(I[1] + I[4] + I[7]);
        g2 = -(I[2] + I[5] + I[8]);
    } else {
        g0 = I[3 * (f - 1)];
        g1 = I[3 * (f - 1) + 1];
        g2 = I[3 * (f - 1) + 2];
    }
}

// H(UL, UR, n) with the Riemann solver of the instantiation.
template <int FLUX, typename T>
__device__ __forceinline__ void riemann(const T UL[5], const T UR[5], const T n[3], T gamma, T eps, T H[5]) {
    if (FLUX == DG_ROE) roe_flux(UL, UR, n, gamma, eps, H);
    else rusanov_flux(UL, UR, n, gamma, H);
}

template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(NT) k_residual_vjp(VjpArgs<Real> a) {
    using S = VPlan<Real, P>;
    using D5 = Dual<Real, 5>;
    constexpr int NB = S::NB, NQ = S::NQ, NQF = S::NQF, EPB = S::EPB;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* tab = reinterpret_cast<Real*>(smem);
    Real* uo = tab + S::TAB;
    Real* lo = uo + S::COWN;
    Real* un = lo + S::COWN;
    Real* ln = un + S::CNBR;
    Real* ubv = ln + S::CNBR;
    Real* ubf = ubv + S::UBV;
    Real* geo = ubf + S::UBF;
    Real* ji = geo + S::GEO;
    int* snbr = reinterpret_cast<int*>(ji + S::JI);
    uint8_t* sfc = reinterpret_cast<uint8_t*>(snbr + EPB * 4);
    int8_t* sperm = reinterpret_cast<int8_t*>(sfc + EPB * 4);
    const int tid = threadIdx.x;
    const Real gamma = a.gamma;

    for (int i = tid; i < S::TAB; i += NT) tab[i] = a.tab[i];
    for (int i = tid; i < 6 * NQF; i += NT) sperm[i] = a.fperm[i];

    const int64_t ntiles = (a.ne + EPB - 1) / EPB;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t e0 = tile * EPB;
        const int nel = (a.ne - e0) < (int64_t)EPB ? (int)(a.ne - e0) : EPB;
        __syncthreads();
        for (int i = tid; i < nel * 5 * NB; i += NT) {
            uo[i] = a.U[e0 * 5 * NB + i];
            lo[i] = a.lam[e0 * 5 * NB + i];
        }
        for (int i = tid; i < nel * 4; i += NT) {
            snbr[i] = a.nbr[e0 * 4 + i];
            sfc[i] = a.fcode[e0 * 4 + i];
        }
        for (int i = tid; i < nel * 9; i += NT) ji[i] = a.jinv[e0 * 9 + i];
        __syncthreads();
        for (int i = tid; i < nel * 4 * 5 * NB; i += NT) {
            const int ef = i / (5 * NB), k = i - ef * 5 * NB;
            const int n = snbr[ef];
            un[i] = n >= 0 ? a.U[(int64_t)n * 5 * NB + k] : Real(0);
            ln[i] = n >= 0 ? a.lam[(int64_t)n * 5 * NB + k] : Real(0);
        }
        for (int i = tid; i < nel * 4; i += NT) {
            const int el = i >> 2, f = i & 3;
            Real g0, g1, g2;
            face_grad(ji + el * 9, f, g0, g1, g2);
            Real s = EulerOps<Real>::sqrt_(g0 * g0 + g1 * g1 + g2 * g2);
            Real inv = Real(-1) / s;
            Real* G = geo + 8 * i;
            G[0] = g0 * inv;
            G[1] = g1 * inv;
            G[2] = g2 * inv;
            G[3] = s;
            const int n = snbr[i];
            if (n >= 0) {   // the neighbour's outward normal and scale on the shared face
                const int fn = sfc[i] & 3;
                face_grad(a.jinv + (int64_t)n * 9, fn, g0, g1, g2);
                s = EulerOps<Real>::sqrt_(g0 * g0 + g1 * g1 + g2 * g2);
                inv = Real(-1) / s;
                G[4] = g0 * inv;
                G[5] = g1 * inv;
                G[6] = g2 * inv;
                G[7] = s;
            }
        }
        __syncthreads();
        // faces
        for (int i = tid; i < nel * 4 * NQF; i += NT) {
            const int ef = i / NQF, q = i - ef * NQF;
            const int el = ef >> 2, f = ef & 3;
            const Real* G = geo + 8 * ef;
            const Real* co = uo + el * 5 * NB;
            const Real* lc = lo + el * 5 * NB;
            const Real* phif = tab + S::PHIF + f * NB * NQF;
            const Real* phifw = tab + S::PHIFW + f * NQF * NB;
            Real Um[5], Up[5], Hb[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                Real s = 0, h = 0;
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    s += co[v * NB + j] * phif[j * NQF + q];
                    h += lc[v * NB + j] * phifw[q * NB + j];
                }
                Um[v] = s;
                Hb[v] = -G[3] * h;
            }
            D5 Dm[5], Dn[3], Dg = D5(gamma), De = D5(a.roe_eps);
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                Dm[v] = D5(Um[v]);
                Dm[v].d[v] = Real(1);
            }
            Dn[0] = D5(G[0]);
            Dn[1] = D5(G[1]);
            Dn[2] = D5(G[2]);
            Real ub[5] = {0, 0, 0, 0, 0};
            const int n = snbr[ef];
            D5 H[5];
            if (n >= 0) {
                const int code = sfc[ef];
                const int fn = code & 3, qn = sperm[(code >> 2) * NQF + q];
                const Real* cn = un + ef * 5 * NB;
                const Real* lcn = ln + ef * 5 * NB;
                const Real* phin = tab + S::PHIF + fn * NB * NQF;
                const Real* phinw = tab + S::PHIFW + fn * NQF * NB;
                Real Hbn[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    Real s = 0, h = 0;
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        s += cn[v * NB + j] * phin[j * NQF + qn];
                        h += lcn[v * NB + j] * phinw[qn * NB + j];
                    }
                    Up[v] = s;
                    Hbn[v] = -G[7] * h;
                }
                D5 Dp[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) Dp[v] = D5(Up[v]);
                riemann<FLUX>(Dm, Dp, Dn, Dg, De, H);          // own residual: d/dU-
#pragma unroll
                for (int k = 0; k < 5; ++k)
#pragma unroll
                    for (int v = 0; v < 5; ++v) ub[k] += H[v].d[k] * Hb[v];
                D5 Dnn[3] = {D5(G[4]), D5(G[5]), D5(G[6])};
                riemann<FLUX>(Dp, Dm, Dnn, Dg, De, H);         // neighbour's residual: d/d(second argument)
#pragma unroll
                for (int k = 0; k < 5; ++k)
#pragma unroll
                    for (int v = 0; v < 5; ++v) ub[k] += H[v].d[k] * Hbn[v];
            } else {
                D5 Gh[5], Fi[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) Fi[v] = D5(a.finf[v]);
                if (n == -1 - DG_BC_WALL) wall_ghost(Dm, Dn, Gh);
                else farfield_ghost(Dm, Dn, Fi, Dg, Gh);
                riemann<FLUX>(Dm, Gh, Dn, Dg, De, H);
#pragma unroll
                for (int k = 0; k < 5; ++k)
#pragma unroll
                    for (int v = 0; v < 5; ++v) ub[k] += H[v].d[k] * Hb[v];
            }
#pragma unroll
            for (int v = 0; v < 5; ++v) ubf[(ef * 5 + v) * NQF + q] = ub[v];
        }
        // volume
        for (int i = tid; i < nel * NQ; i += NT) {
            const int el = i / NQ, q = i - el * NQ;
            const Real* co = uo + el * 5 * NB;
            const Real* lc = lo + el * 5 * NB;
            const Real* I = ji + el * 9;
            D5 U[5];
            Real Gb[3][5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                Real s = 0, g0 = 0, g1 = 0, g2 = 0;
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const Real c = co[v * NB + j], l = lc[v * NB + j];
                    s += c * tab[S::PHIQ + j * NQ + q];
                    g0 += l * tab[S::DPHIW + (0 * NQ + q) * NB + j];
                    g1 += l * tab[S::DPHIW + (1 * NQ + q) * NB + j];
                    g2 += l * tab[S::DPHIW + (2 * NQ + q) * NB + j];
                }
                U[v] = D5(s);
                U[v].d[v] = Real(1);
                Gb[0][v] = g0;
                Gb[1][v] = g1;
                Gb[2][v] = g2;
            }
            // G_k = sum_d Jinv_kd F_d  =>  Fbar_d = sum_k Jinv_kd Gbar_k
            const D5 ri = D5(Real(1)) / U[0];
            const D5 u[3] = {U[1] * ri, U[2] * ri, U[3] * ri};
            const D5 p = D5(gamma - Real(1)) * (U[4] - D5(Real(0.5)) * (U[1] * u[0] + U[2] * u[1] + U[3] * u[2]));
            Real ub[5] = {0, 0, 0, 0, 0};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                D5 F[5];
                F[0] = U[1 + d];
                F[1] = U[1] * u[d];
                F[2] = U[2] * u[d];
                F[3] = U[3] * u[d];
                F[1 + d] = F[1 + d] + p;
                F[4] = (U[4] + p) * u[d];
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    const Real fb = I[d] * Gb[0][v] + I[3 + d] * Gb[1][v] + I[6 + d] * Gb[2][v];
#pragma unroll
                    for (int k = 0; k < 5; ++k) ub[k] += F[v].d[k] * fb;
                }
            }
#pragma unroll
            for (int v = 0; v < 5; ++v) ubv[(el * 5 + v) * NQ + q] = ub[v];
        }
        __syncthreads();
        for (int i = tid; i < nel * 5 * NB; i += NT) {
            const int ev = i / NB, j = i - ev * NB;
            const int el = ev / 5, v = ev - el * 5;
            Real r = 0;
            const Real* bv = ubv + (el * 5 + v) * NQ;
#pragma unroll
            for (int q = 0; q < NQ; ++q) r += bv[q] * tab[S::PHIQ + j * NQ + q];
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const Real* bf = ubf + ((el * 4 + f) * 5 + v) * NQF;
#pragma unroll
                for (int q = 0; q < NQF; ++q) r += bf[q] * tab[S::PHIF + (f * NB + j) * NQF + q];
            }
            const int64_t gi = e0 * 5 * NB + i;
            Real res = a.c3 * r;
            if (a.X) res += a.c0 * a.X[gi];
            if (a.Y) res += a.c1 * a.Y[gi];
            if (a.Z) res += a.c2 * a.Z[gi];
            a.out[gi] = res;
        }
    }
}

template <typename Real, int P, int FLUX>
cudaError_t vlaunch(const VjpArgs<Real>& args, cudaStream_t s, int nsm) {
    using S = VPlan<Real, P>;
    auto kern = k_residual_vjp<Real, P, FLUX>;
    static int occ = -1;
    if (occ < 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::BYTES);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, S::BYTES);
        if (e != cudaSuccess) return e;
        if (occ < 1) occ = 1;
    }
    const int64_t ntiles = (args.ne + S::EPB - 1) / S::EPB;
    const int grid = (int)std::min<int64_t>(ntiles, (int64_t)nsm * occ);
    kern<<<grid, NT, S::BYTES, s>>>(args);
    return cudaGetLastError();
}

// ---- face-once form -------------------------------------------------------------------------------

constexpr int VF = 128;   // threads of the face kernels; 32 where that would leave SMs without a block
inline unsigned vface_block(int64_t n) { return n < (int64_t)VF * 4 * 152 ? 32 : VF; }

template <typename Real>
struct FaceVjpArgs {
    Real* T;                // traces of U in, face adjoints out [ne][4][5][Nqf]
    const Real* TL;         // traces of lambda
    const FaceRec* rec;
    const Real* normal;     // [faces][3]
    const Real* scale;      // [faces][2] |grad lambda_f| of the slot and of the matching one
    const int8_t* fperm;
    int64_t n;              // faces x Nqf
    Real gamma, roe_eps;
    Real finf[5];
};

// the i-th (interior face, point)
template <typename Real, int P, int FLUX>
__device__ __forceinline__ void face_vjp(const FaceVjpArgs<Real>& a, int64_t i) {
    constexpr int NQF = nqf_of(P);
    if (i >= a.n) return;
    const int64_t li = i / NQF;
    const int q = (int)(i - li * NQF);
    const int4 f = *reinterpret_cast<const int4*>(a.rec + li);   // slot (the owner's), other, code
    const Real n[3] = {a.normal[3 * li], a.normal[3 * li + 1], a.normal[3 * li + 2]};
    const Real so = a.scale[2 * li], sn = a.scale[2 * li + 1];
    const int64_t oe = (int64_t)f.x * 5 * NQF + q, on = (int64_t)f.y * 5 * NQF + a.fperm[(f.z & 7) * NQF + q];
    Real L[5], R[5], Ho[5], Hn[5], Hb[5], Lb[5], Rb[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        L[v] = a.T[oe + v * NQF];
        R[v] = a.T[on + v * NQF];
        Ho[v] = -so * a.TL[oe + v * NQF];
        Hn[v] = sn * a.TL[on + v * NQF];
        Hb[v] = Ho[v] + Hn[v];
    }
    if (face_reverse<Real, FLUX>(L, R, n, a.gamma, a.roe_eps, Hb, Real(1), Lb, Rb)) {
        Real x[5], y[5];
        face_reverse<Real, FLUX>(L, R, n, a.gamma, a.roe_eps, Ho, Real(1), Lb, Rb);
        face_reverse<Real, FLUX>(L, R, n, a.gamma, a.roe_eps, Hn, Real(-1), x, y);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            Lb[v] += x[v];
            Rb[v] += y[v];
        }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        a.T[oe + v * NQF] = Lb[v];
        a.T[on + v * NQF] = Rb[v];
    }
}

// the i-th (boundary face, point)
template <typename Real, int P, int FLUX>
__device__ __forceinline__ void bface_vjp(const FaceVjpArgs<Real>& a, int64_t i) {
    using D5 = Dual<Real, 5>;
    constexpr int NQF = nqf_of(P);
    if (i >= a.n) return;
    const int64_t li = i / NQF;
    const int q = (int)(i - li * NQF);
    const int4 f = *reinterpret_cast<const int4*>(a.rec + li);
    const Real s = a.scale[2 * li];
    const int64_t oe = (int64_t)f.x * 5 * NQF + q;
    D5 U[5], G[5], n[3], Fi[5], H[5];
    const D5 g = D5(a.gamma), eps = D5(a.roe_eps);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        U[v] = D5(a.T[oe + v * NQF]);
        U[v].d[v] = Real(1);
        Fi[v] = D5(a.finf[v]);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) n[d] = D5(a.normal[3 * li + d]);
    if (f.y == -1 - DG_BC_WALL) wall_ghost(U, n, G);
    else farfield_ghost(U, n, Fi, g, G);
    riemann<FLUX>(U, G, n, g, eps, H);
    Real ub[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        const Real hb = -s * a.TL[oe + v * NQF];
#pragma unroll
        for (int k = 0; k < 5; ++k) ub[k] += H[v].d[k] * hb;
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) a.T[oe + v * NQF] = ub[v];
}

template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(VF) k_faces_vjp(FaceVjpArgs<Real> a) {
    face_vjp<Real, P, FLUX>(a, blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
}
template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(VF) k_bfaces_vjp(FaceVjpArgs<Real> a) {
    bface_vjp<Real, P, FLUX>(a, blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
}

// Both in one launch of one-warp blocks, side by side: on a small mesh the boundary faces' long chain (dual
// numbers) and its launch were a quarter of a VJP (FP32 P2 Rusanov with boundary faces, 750 elements, with the
// two gathers in one launch 33.8 -> 25.4 us; the single kernel 25.5).  The registers of the longer part allow 10 warps an SM, so larger meshes keep two launches.
constexpr int64_t BOTH_MAX_WARPS = 8 * 152;
template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(32) k_allfaces_vjp(FaceVjpArgs<Real> a, FaceVjpArgs<Real> b, unsigned interior) {
    if (blockIdx.x < interior) face_vjp<Real, P, FLUX>(a, blockIdx.x * (int64_t)32 + threadIdx.x);
    else bface_vjp<Real, P, FLUX>(b, (blockIdx.x - interior) * (int64_t)32 + threadIdx.x);
}

template <typename Real, int P, int EE>
struct VElemPlan {
    static constexpr int ER = rows_of(EE);
    // the volume points go in NC chunks of consecutive points, closed under the mirror, so that
    // several tiles fit an SM
    static constexpr int NQ = nq_of(P), NC = P == 1 ? 1 : 2;
    static constexpr int first(int c) { return c == 0 ? 0 : c == NC ? NQ : P == 2 ? 8 : 12; }
    static constexpr int MAXQ = P == 1 ? 4 : P == 2 ? 8 : 12;
    // shared memory (Reals): point states, then their adjoints [MAXQ][ER]; d_k lambda [MAXQ][3][ER];
    // J^-1 [EE][9]
    static constexpr int D = MAXQ * ER, J = D + 3 * MAXQ * ER, REALS = J + EE * 9;
    static constexpr size_t BYTES = REALS * sizeof(Real);
};

template <typename Real, int P, int EE>
__global__ void __launch_bounds__(threads_of(EE)) k_element_vjp(VjpArgs<Real> a, const Real* __restrict__ UB) {
    using S = VElemPlan<Real, P, EE>;
    constexpr int ER = S::ER, NT = threads_of(EE);
    constexpr int NB = nb_of(P), NQF = nqf_of(P), NM = modal::Tables<P>::NM;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* sU = reinterpret_cast<Real*>(smem);
    Real* sD = sU + S::D;
    Real* sJ = sU + S::J;
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (a.ne - e0) < (int64_t)EE ? (int)(a.ne - e0) : EE;
    const bool live = t < 5 * nel;
    const int64_t row = e0 * 5 + t;
    const Real g1 = a.gamma - Real(1);
    for (int i = t; i < nel * 9; i += NT) sJ[i] = a.jinv[e0 * 9 + i];
    Real r[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) r[j] = 0;
    // one chunk of points; its bounds are compile-time constants, as the operators' loops need
    auto chunk = [&](auto ch) {
        constexpr int q0 = S::first(ch.value), q1 = S::first(ch.value + 1);
        if (live) {
            Real c[NB];
            load_row<NB>(a.U + row * NB, c);
            modal::interpolate<Real, P, NB, q0, q1>(c, [&](int q, Real u) { sU[(q - q0) * ER + t] = u; });
            load_row<NB>(a.lam + row * NB, c);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                Real d[NM];
                modal::grad_modes<Real, P>(k, c, d);
                modal::interpolate<Real, P, NM, q0, q1>(d, [&](int q, Real x) { sD[((q - q0) * 3 + k) * ER + t] = x; });
            }
        }
        __syncthreads();
        // reverse of G_k = W_k (m_.. , E + p) + p J^-1_k, W = J^-1 u, against the derivatives of lambda
        for (int i = t; i < (q1 - q0) * EE; i += NT) {
            const int e = i % EE, q = i / EE;
            if (e >= nel) continue;
            Real* u = sU + q * ER + 5 * e;
            const Real* g = sD + q * 3 * ER + 5 * e;
            const Real* I = sJ + e * 9;
            const Real ri = recip(u[0]);
            const Real x[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
            const Real k2 = Real(0.5) * (x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
            const Real p = g1 * (u[4] - u[0] * k2), ep = u[4] + p;
            Real ub[5] = {0, 0, 0, 0, 0}, vb[3] = {0, 0, 0}, pb = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Real* gk = g + k * ER;
                const Real W = I[3 * k] * x[0] + I[3 * k + 1] * x[1] + I[3 * k + 2] * x[2];
                const Real Wb = gk[0] * u[0] + gk[1] * u[1] + gk[2] * u[2] + gk[3] * u[3] + gk[4] * ep;
#pragma unroll
                for (int v = 0; v < 5; ++v) ub[v] += gk[v] * W;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    vb[d] += I[3 * k + d] * Wb;
                    pb += I[3 * k + d] * gk[1 + d];
                }
            }
            pb = g1 * (pb + ub[4]);
            ub[0] += pb * k2 - ri * (vb[0] * x[0] + vb[1] * x[1] + vb[2] * x[2]);
#pragma unroll
            for (int d = 0; d < 3; ++d) ub[1 + d] += vb[d] * ri - pb * x[d];
            ub[4] += pb;
#pragma unroll
            for (int v = 0; v < 5; ++v) u[v] = ub[v];
        }
        __syncthreads();
        if (live) {
            modal::unroll<q0, q1>([&](auto qc) {
                constexpr int q = qc.value, m = modal::kT<P>.vmir[q];
                if constexpr (m >= q)
                    modal::moments<Real, P, NB>(q, sU[(q - q0) * ER + t], m != q ? sU[(m - q0) * ER + t] : Real(0), r);
            });
        }
    };
    chunk(std::integral_constant<int, 0>());
    if constexpr (S::NC > 1) {
        __syncthreads();
        chunk(std::integral_constant<int, 1>());
    }
    if (!live) return;
    const int e = t / 5, v = t - 5 * e;
    const Real* h = UB + ((e0 + e) * 20 + v) * NQF;
    modal::lift<Real, P>(
        [&](int f, Real* x) {
            load_row<NQF>(h + f * 5 * NQF, x);
            return Real(1);
        },
        r);
#pragma unroll
    for (int j = 0; j < NB; ++j) r[j] *= a.c3;
    auto add = [&](const Real* X, Real c) {
        if (!X) return;
        Real x[NB];
        load_row<NB>(X + row * NB, x);
#pragma unroll
        for (int j = 0; j < NB; ++j) r[j] += c * x[j];
    };
    add(a.X, a.c0);
    add(a.Y, a.c1);
    add(a.Z, a.c2);
    store_row<NB>(a.out + row * NB, r);
}

template <typename Real, int P, int EE>
cudaError_t vlaunch_tiles(const VjpArgs<Real>& r, const Real* UB, cudaStream_t s) {
    auto kern = k_element_vjp<Real, P, EE>;
    constexpr size_t bytes = VElemPlan<Real, P, EE>::BYTES;
    static bool init = false;
    if (!init) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        init = true;
    }
    kern<<<(unsigned)((r.ne + EE - 1) / EE), threads_of(EE), bytes, s>>>(r, UB);
    return cudaGetLastError();
}

template <typename Real, int P, int FLUX>
cudaError_t vlaunch_faces(dg_mesh* m, const VjpArgs<Real>& r, cudaStream_t s) {
    constexpr int NQF = nqf_of(P);
    cudaError_t e = launch_traces2(m, r.U, m->d_TA, r.lam, m->d_TL, s);
    if (e != cudaSuccess) return e;
    FaceVjpArgs<Real> f;
    f.T = static_cast<Real*>(m->d_TA);
    f.TL = static_cast<const Real*>(m->d_TL);
    f.rec = m->d_frec;
    f.normal = static_cast<const Real*>(m->d_fnorm);
    f.scale = static_cast<const Real*>(m->d_fscale);
    f.fperm = m->d_fperm;
    f.n = m->n_interior * NQF;
    f.gamma = r.gamma;
    f.roe_eps = r.roe_eps;
    for (int v = 0; v < 5; ++v) f.finf[v] = r.finf[v];
    FaceVjpArgs<Real> b = f;   // the boundary faces
    b.rec += m->n_interior;
    b.normal += 3 * m->n_interior;
    b.scale += 2 * m->n_interior;
    b.n = (m->n_flist - m->n_interior) * NQF;
    const int64_t wi = (f.n + 31) / 32, wb = (b.n + 31) / 32;
    bool both = false;
    if constexpr (sizeof(Real) == 4) both = wi > 0 && wb > 0 && wi + wb <= BOTH_MAX_WARPS;
    if (both) {
        if constexpr (sizeof(Real) == 4) k_allfaces_vjp<Real, P, FLUX><<<(unsigned)(wi + wb), 32, 0, s>>>(f, b, (unsigned)wi);
    } else {
        unsigned nt = vface_block(f.n);
        if (f.n > 0) k_faces_vjp<Real, P, FLUX><<<(unsigned)((f.n + nt - 1) / nt), nt, 0, s>>>(f);
        nt = vface_block(b.n);
        if (b.n > 0) k_bfaces_vjp<Real, P, FLUX><<<(unsigned)((b.n + nt - 1) / nt), nt, 0, s>>>(b);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return small_tiles(r.ne) ? vlaunch_tiles<Real, P, 6>(r, f.T, s) : vlaunch_tiles<Real, P, 32>(r, f.T, s);
}

template <typename Real>
cudaError_t vdispatch(dg_mesh* m, const void* U, const void* lam, const void* X, const void* Y, const void* Z,
                      const double c[4], void* out, cudaStream_t s) {
    VjpArgs<Real> r;
    r.U = static_cast<const Real*>(U);
    r.lam = static_cast<const Real*>(lam);
    r.X = static_cast<const Real*>(X);
    r.Y = static_cast<const Real*>(Y);
    r.Z = static_cast<const Real*>(Z);
    r.c0 = (Real)c[0];
    r.c1 = (Real)c[1];
    r.c2 = (Real)c[2];
    r.c3 = (Real)c[3];
    r.out = static_cast<Real*>(out);
    r.nbr = m->d_nbr;
    r.fcode = m->d_fcode;
    r.jinv = static_cast<const Real*>(m->d_jinv);
    r.tab = static_cast<const Real*>(m->d_tab);
    r.fperm = m->d_fperm;
    r.ne = m->host.ne;
    r.gamma = (Real)m->gamma;
    r.roe_eps = (Real)m->roe_eps;
    for (int v = 0; v < 5; ++v) r.finf[v] = (Real)m->finf[v];
    const bool roe = m->flux == DG_ROE;
    if (m->face_once && m->d_TA && m->d_TL) {
        switch (m->p) {
            case 1: return roe ? vlaunch_faces<Real, 1, DG_ROE>(m, r, s) : vlaunch_faces<Real, 1, DG_RUSANOV>(m, r, s);
            case 2: return roe ? vlaunch_faces<Real, 2, DG_ROE>(m, r, s) : vlaunch_faces<Real, 2, DG_RUSANOV>(m, r, s);
            default: return roe ? vlaunch_faces<Real, 3, DG_ROE>(m, r, s) : vlaunch_faces<Real, 3, DG_RUSANOV>(m, r, s);
        }
    }
    if constexpr (sizeof(Real) == 8) {
        return cudaErrorInvalidValue;   // FP64 has no other form
    } else {
        int nsm = 0;
        cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
        if (e != cudaSuccess) return e;
        switch (m->p) {
            case 1: return roe ? vlaunch<Real, 1, DG_ROE>(r, s, nsm) : vlaunch<Real, 1, DG_RUSANOV>(r, s, nsm);
            case 2: return roe ? vlaunch<Real, 2, DG_ROE>(r, s, nsm) : vlaunch<Real, 2, DG_RUSANOV>(r, s, nsm);
            default: return roe ? vlaunch<Real, 3, DG_ROE>(r, s, nsm) : vlaunch<Real, 3, DG_RUSANOV>(r, s, nsm);
        }
    }
}

}  // namespace

cudaError_t launch_residual_vjp(dg_mesh* m, const void* U, const void* lam, const void* X, const void* Y,
                                const void* Z, const double c[4], void* out, cudaStream_t s) {
    if (m->precision == DG_FP64) return vdispatch<double>(m, U, lam, X, Y, Z, c, out, s);
    return vdispatch<float>(m, U, lam, X, Y, Z, c, out, s);
}

}  // namespace dg
