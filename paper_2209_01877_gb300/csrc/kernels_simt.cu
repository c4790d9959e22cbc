// Residual and SSP-RK3 stage on the CUDA cores: FP64, and the FP32 stages of larger meshes, with every
// face's traces and numerical flux evaluated once (FP32 residual calls, the stages of smaller
// meshes and of meshes with boundary faces: the single kernel k_residual below; capi.cpp has
// the rules).  Three launches per residual or stage:
//   k_traces  thread per (element, variable): the element's own trace at the points of its 4 faces,
//             to a face buffer T[e][f][v][q];
//   k_faces   thread per (listed face, point): the flux in the owner's orientation,
//             H(U_owner, U_other, n_owner) with the owner's normal (owner: the element with the
//             smaller caller index; boundary faces: the element), written over the two traces it was
//             evaluated from: +H in the owner's slot, -H in the other's at the matching point;
//   k_element tiles of 32 elements, thread per (element, variable) row: volume interpolation (Eq. 11
//             volume line), thread per (element, point) for the contravariant velocity and the
//             pressure, then the projection of G_k = W_k U + p (J^-1)_k on the basis gradients, the
//             lift of the stored fluxes, and either R or the RK stage out = a U0 + b (U + dt R).
// Every input of a face's flux (both traces, the normal, the argument order) is independent of the
// internal element order, and an element's sums run in a fixed order: the residual is bitwise the
// same in every element order and through partitions, without atomics.
//
// What bounds them: FP64 the FP64 pipe (2 lanes a clock and SM), so the operators are factored
// (modal_ops.cuh) and their constants are operands of the instructions; FP32 the traffic of the face
// buffer (written and read twice per stage, 4 Nqf 5 values per element) and of the states.
// Measured, one SSP-RK3 step between set and get of the state, dense operators and one thread per
// point before -> factored operators: FP64 P3 Roe, 196,608 elements 27.7 -> 17.1 ms; FP64 P1 Rusanov,
// 1,296 elements 85 -> 62 us; FP32 P2 Rusanov, 663,552 elements, per stage 980 us (one kernel, each face
// from both sides) -> 65 + 153 + 147 us.
#include <algorithm>
#include <type_traits>

#include "dg_internal.h"
#include "euler_device.cuh"
#include "face_flux.cuh"
#include "modal_ops.cuh"
#include "tc_ops.cuh"

namespace dg {

namespace {

constexpr int NT = 256;

// ---- FP32 without a face buffer ------------------------------------------------------------------
// One persistent kernel per residual that evaluates every face from both sides: the calls that return
// an FP32 residual (their values stay those of this order of summation), the RK stages of meshes on which
// it is the faster form, of meshes with boundary faces, and of meshes without room for the face
// buffer (80 Nqf bytes per element; on large meshes a P2 stage takes two and a half times the time of
// the face-once form below).

template <int P> struct Tile;
template <> struct Tile<1> { static constexpr int EPB = 32; };
template <> struct Tile<2> { static constexpr int EPB = 16; };
template <> struct Tile<3> { static constexpr int EPB = 8; };

template <typename Real, int P>
struct Plan {
    static constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), EPB = Tile<P>::EPB;
    static constexpr int PHIQ = 0, DPHIW = NB * NQ, PHIF = DPHIW + 3 * NQ * NB, PHIFW = PHIF + 4 * NB * NQF,
                         WQ = PHIFW + 4 * NQF * NB, TAB = WQ + NQ;
    static constexpr int COWN = EPB * 5 * NB;
    static constexpr int CNBR = EPB * 4 * 5 * NB;
    static constexpr int GV = EPB * 3 * 5 * NQ;
    static constexpr int BIG = CNBR > GV ? CNBR : GV;
    static constexpr int HW = EPB * 4 * 5 * NQF;
    static constexpr int GEO = EPB * 4 * 4;
    static constexpr int JI = EPB * 9;
    static constexpr int REALS = TAB + COWN + BIG + HW + GEO + JI;
    static constexpr size_t BYTES = REALS * sizeof(Real) + EPB * 4 * sizeof(int) + EPB * 4 + 6 * NQF + 16;
};

template <typename Real>
__device__ __forceinline__ void flag(unsigned int* status, unsigned int bit) {
    atomicOr(status, bit);
}

template <typename Real, int P, int FLUX, bool RK>
__global__ void __launch_bounds__(NT) k_residual(ResArgs<Real> a) {
    using S = Plan<Real, P>;
    constexpr int NB = S::NB, NQ = S::NQ, NQF = S::NQF, EPB = S::EPB;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* tab = reinterpret_cast<Real*>(smem);
    Real* cown = tab + S::TAB;
    Real* big = cown + S::COWN;
    Real* hw = big + S::BIG;
    Real* geo = hw + S::HW;
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
        {
            const Real* Ut = a.U + e0 * 5 * NB;
            for (int i = tid; i < nel * 5 * NB; i += NT) cown[i] = Ut[i];
            for (int i = tid; i < nel * 4; i += NT) {
                snbr[i] = a.nbr[e0 * 4 + i];
                sfc[i] = a.fcode[e0 * 4 + i];
            }
            for (int i = tid; i < nel * 9; i += NT) ji[i] = a.jinv[e0 * 9 + i];
        }
        __syncthreads();
        // neighbour coefficient blocks and per-face normals / scale factors
        for (int i = tid; i < nel * 4 * 5 * NB; i += NT) {
            const int ef = i / (5 * NB), k = i - ef * 5 * NB;
            const int n = snbr[ef];
            big[i] = n >= 0 ? a.U[(int64_t)n * 5 * NB + k] : Real(0);
        }
        for (int i = tid; i < nel * 4; i += NT) {
            const int el = i >> 2, f = i & 3;
            const Real* I = ji + el * 9;
            Real g0, g1, g2;   // grad_x lambda_f (row f-1 of J^-1; lambda_0 = 1 - sum)
            if (f == 0) {
                g0 = -(I[0] + I[3] + I[6]);
                g1 = -(I[1] + I[4] + I[7]);
                g2 = -(I[2] + I[5] + I[8]);
            } else {
                g0 = I[3 * (f - 1)];
                g1 = I[3 * (f - 1) + 1];
                g2 = I[3 * (f - 1) + 2];
            }
            const Real s = EulerOps<Real>::sqrt_(g0 * g0 + g1 * g1 + g2 * g2);
            const Real inv = Real(-1) / s;   // outward normal is -grad lambda_f / |grad lambda_f|
            geo[4 * i + 0] = g0 * inv;
            geo[4 * i + 1] = g1 * inv;
            geo[4 * i + 2] = g2 * inv;
            geo[4 * i + 3] = s;
        }
        __syncthreads();
        // faces: numerical flux at every (element, face, point)
        for (int i = tid; i < nel * 4 * NQF; i += NT) {
            const int ef = i / NQF, q = i - ef * NQF;
            const int el = ef >> 2, f = ef & 3;
            const Real* co = cown + el * 5 * NB;
            const Real* phif = tab + S::PHIF + f * NB * NQF;
            Real Um[5], Up[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                Real s = 0;
#pragma unroll
                for (int j = 0; j < NB; ++j) s += co[v * NB + j] * phif[j * NQF + q];
                Um[v] = s;
            }
            const Real* nr = geo + 4 * ef;
            const Real nv[3] = {nr[0], nr[1], nr[2]};
            const int n = snbr[ef];
            if (n >= 0) {
                const int code = sfc[ef];
                const int fn = code & 3, qn = sperm[(code >> 2) * NQF + q];
                const Real* cn = big + ef * 5 * NB;
                const Real* phin = tab + S::PHIF + fn * NB * NQF;
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    Real s = 0;
#pragma unroll
                    for (int j = 0; j < NB; ++j) s += cn[v * NB + j] * phin[j * NQF + qn];
                    Up[v] = s;
                }
            } else if (n == -1 - DG_BC_WALL) {
                wall_ghost(Um, nv, Up);
            } else {
                farfield_ghost(Um, nv, a.finf, gamma, Up);
            }
            if (!physical(Um, gamma)) flag<Real>(a.status, 1u);
            Real H[5];
            if (FLUX == DG_ROE) roe_flux(Um, Up, nv, gamma, a.roe_eps, H);
            else rusanov_flux(Um, Up, nv, gamma, H);
            const Real sc = -nr[3];
#pragma unroll
            for (int v = 0; v < 5; ++v) hw[(ef * 5 + v) * NQF + q] = sc * H[v];
        }
        __syncthreads();
        // volume: contravariant flux at every (element, point); overwrites the neighbour blocks
        for (int i = tid; i < nel * NQ; i += NT) {
            const int el = i / NQ, q = i - el * NQ;
            const Real* co = cown + el * 5 * NB;
            Real U[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                Real s = 0;
#pragma unroll
                for (int j = 0; j < NB; ++j) s += co[v * NB + j] * tab[S::PHIQ + j * NQ + q];
                U[v] = s;
            }
            if (!physical(U, gamma)) flag<Real>(a.status, 1u);
            const Real ri = Real(1) / U[0];
            const Real u[3] = {U[1] * ri, U[2] * ri, U[3] * ri};
            const Real p = (gamma - Real(1)) * (U[4] - Real(0.5) * (U[1] * u[0] + U[2] * u[1] + U[3] * u[2]));
            Real F[3][5];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                F[d][0] = U[1 + d];
                F[d][1] = U[1] * u[d];
                F[d][2] = U[2] * u[d];
                F[d][3] = U[3] * u[d];
                F[d][1 + d] += p;
                F[d][4] = (U[4] + p) * u[d];
            }
            const Real* I = ji + el * 9;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int v = 0; v < 5; ++v)
                    big[((el * 3 + k) * 5 + v) * NQ + q] = I[3 * k] * F[0][v] + I[3 * k + 1] * F[1][v] + I[3 * k + 2] * F[2][v];
        }
        __syncthreads();
        // projection onto the basis gradients, face lift, epilogue
        for (int i = tid; i < nel * 5 * NB; i += NT) {
            const int ev = i / NB, j = i - ev * NB;
            const int el = ev / 5, v = ev - el * 5;
            Real r = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Real* g = big + ((el * 3 + k) * 5 + v) * NQ;
#pragma unroll
                for (int q = 0; q < NQ; ++q) r += g[q] * tab[S::DPHIW + (k * NQ + q) * NB + j];
            }
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const Real* h = hw + ((el * 4 + f) * 5 + v) * NQF;
#pragma unroll
                for (int q = 0; q < NQF; ++q) r += h[q] * tab[S::PHIFW + (f * NQF + q) * NB + j];
            }
            const int64_t gi = e0 * 5 * NB + i;
            if (RK) {
                Real res = a.b * (cown[i] + a.dt * r);
                if (a.a != Real(0)) res += a.a * a.U0[gi];
                a.out[gi] = res;
            } else {
                a.out[gi] = r;
            }
        }
    }
}

template <typename Real, int P, int FLUX, bool RK>
cudaError_t launch_one(const ResArgs<Real>& args, cudaStream_t s, int nsm) {
    using S = Plan<Real, P>;
    auto kern = k_residual<Real, P, FLUX, RK>;
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

template <typename Real, int P>
cudaError_t dispatch_flux(const ResArgs<Real>& args, int flux, bool rk, cudaStream_t s, int nsm) {
    if (flux == DG_ROE) return rk ? launch_one<Real, P, DG_ROE, true>(args, s, nsm) : launch_one<Real, P, DG_ROE, false>(args, s, nsm);
    return rk ? launch_one<Real, P, DG_RUSANOV, true>(args, s, nsm) : launch_one<Real, P, DG_RUSANOV, false>(args, s, nsm);
}

// ---- face-once form -----------------------------------------------------------------------------

constexpr int FT = 128;       // threads of k_faces; 32 where that would leave SMs without a block
inline unsigned face_block(int64_t n) { return n < (int64_t)FT * 4 * 152 ? 32 : FT; }

// |grad lambda_f| = 2 |S_f| / |det J| from the row-major J^-1
__device__ __forceinline__ double face_scale(const double* I, int f) {
    double g[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) g[d] = f == 0 ? -(I[d] + I[3 + d] + I[6 + d]) : I[3 * (f - 1) + d];
    return sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
}

// The trace of every (element, face, point) of one or (gridDim.y = 2) two states: thread per (element,
// variable) row.  In FP32 the tile's
// coefficients and traces pass through shared memory, so that the global accesses are whole lines:
// rows written directly (24 to 48 bytes each) kept the load-store unit busy (P2, 663,552 elements:
// 127 us at 39 % of the DRAM rate).  FP64 is bound by its pipe and writes its rows directly.
template <typename Real, int P, int EE>
__global__ void __launch_bounds__(threads_of(EE), EE == 32 ? (sizeof(Real) == 8 ? (P == 3 ? 3 : P == 2 ? 6 : 10) : (P == 3 ? 5 : 10)) : 14)
    k_traces(const Real* U0, Real* T0, const Real* U1, Real* T1, int64_t ne) {
    constexpr int NB = nb_of(P), NQF = nqf_of(P), NT = threads_of(EE);
    const Real* __restrict__ U = blockIdx.y == 0 ? U0 : U1;
    Real* __restrict__ T = blockIdx.y == 0 ? T0 : T1;
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (ne - e0) < (int64_t)EE ? (int)(ne - e0) : EE;
    const int e = t / 5, v = t - 5 * e;
    if constexpr (sizeof(Real) == 8) {
        if (t >= 5 * nel) return;
        Real c[NB];
        load_row<NB>(U + (e0 * 5 + t) * NB, c);
        Real* o = T + ((e0 + e) * 20 + v) * NQF;
        modal::traces<Real, P>(c, [&](int f, const Real* u) { store_row<NQF>(o + f * 5 * NQF, u); });
    } else {
        __shared__ __align__(16) Real sU[rows_of(EE) * NB + 4], sT[EE * 20 * NQF];
        copy_tile<NT>(sU, U + e0 * 5 * NB, nel * 5 * NB * (int)sizeof(Real));
        tc::cp_async_wait_all();
        __syncthreads();
        if (t < 5 * nel) {
            Real c[NB];
            load_row<NB>(sU + t * NB, c);
            Real* o = sT + (e * 20 + v) * NQF;
            modal::traces<Real, P>(c, [&](int f, const Real* u) { store_row<NQF>(o + f * 5 * NQF, u); });
        }
        __syncthreads();
        float4* g = reinterpret_cast<float4*>(T + e0 * 20 * NQF);
        for (int i = t; i < nel * 5 * NQF; i += NT) g[i] = reinterpret_cast<const float4*>(sT)[i];
    }
}

template <typename Real, int P>
cudaError_t traces(const void* U, void* T, const void* U1, void* T1, int64_t ne, cudaStream_t s) {
    const Real *u = static_cast<const Real*>(U), *u1 = static_cast<const Real*>(U1);
    Real *t = static_cast<Real*>(T), *t1 = static_cast<Real*>(T1);
    if (small_tiles(ne))
        k_traces<Real, P, 6><<<dim3((unsigned)((ne + 5) / 6), U1 ? 2 : 1), threads_of(6), 0, s>>>(u, t, u1, t1, ne);
    else
        k_traces<Real, P, 32><<<dim3((unsigned)((ne + 31) / 32), U1 ? 2 : 1), threads_of(32), 0, s>>>(u, t, u1, t1, ne);
    return cudaGetLastError();
}

template <typename Real>
struct FaceArgs {
    Real* T;                // face buffer [n_trace][4][5][Nqf]: traces in, fluxes out
    const FaceRec* rec;
    const Real* normal;     // [faces][3] the owner's outward normal
    const int8_t* fperm;
    int64_t n;              // listed faces x Nqf
    Real gamma, roe_eps;
    Real finf[5];
    unsigned int* status;
};

// the flux of every listed face at every point, in the owner's orientation, to both slots (in
// place: each thread writes the entries it read)
template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(FT) k_faces(FaceArgs<Real> a) {
    constexpr int NQF = nqf_of(P);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const int64_t li = i / NQF;
    const int q = (int)(i - li * NQF);
    const int4 f = *reinterpret_cast<const int4*>(a.rec + li);   // slot, other, code
    const Real* nc = a.normal + li * 3;
    const Real nv[3] = {nc[0], nc[1], nc[2]};
    const int64_t slot = f.x;
    Real* te = a.T + slot * 5 * NQF + q;
    Real Ue[5], Un[5], H[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) Ue[v] = te[v * NQF];
    bool okL, okR;
    if (f.y < 0) {
        if (f.y == -1 - DG_BC_WALL) wall_ghost(Ue, nv, Un);
        else farfield_ghost(Ue, nv, a.finf, a.gamma, Un);
        face_flux<Real, FLUX>(Ue, Un, nv, a.gamma, a.roe_eps, H, okL, okR);
        if (!okL) atomicOr(a.status, 1u);
#pragma unroll
        for (int v = 0; v < 5; ++v) te[v * NQF] = H[v];
        return;
    }
    const int qn = a.fperm[(f.z & 7) * NQF + q];
    Real* tn = a.T + (int64_t)f.y * 5 * NQF + qn;
#pragma unroll
    for (int v = 0; v < 5; ++v) Un[v] = tn[v * NQF];
    const bool own = (f.z & 8) != 0;   // false only for a face shared with a halo element that owns it
    Real sg = Real(1);
    if (!own) {
        sg = Real(-1);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            const Real t = Ue[v];
            Ue[v] = Un[v];
            Un[v] = t;
        }
    }
    face_flux<Real, FLUX>(Ue, Un, nv, a.gamma, a.roe_eps, H, okL, okR);
    // FP64 reports the listed slot's trace (the volume points cover every element), FP32 both
    if (sizeof(Real) == 4 ? !(okL && okR) : !(own ? okL : okR)) atomicOr(a.status, 1u);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        te[v * NQF] = sg * H[v];
        tn[v * NQF] = -sg * H[v];
    }
}

// contravariant velocity W_k = sum_d (J^-1)_kd u_d and pressure of the i-th (point, element) of a tile
// (points from NQ on are no quadrature points: their states are not reported)
template <typename Real, int EE, int ER>
__device__ __forceinline__ void contravariant_point(const ResArgs<Real>& a, int nel, int i, int NQ, const Real* sU, Real* sW,
                                                    const Real* sJ) {
    const int e = i % EE, q = i / EE;
    if (e >= nel) return;
    const Real* u = sU + q * ER + 5 * e;
    const Real rho = u[0], ri = recip(rho);
    const Real x = u[1] * ri, y = u[2] * ri, z = u[3] * ri;
    const Real p = (a.gamma - Real(1)) * (u[4] - Real(0.5) * (u[1] * x + u[2] * y + u[3] * z));
    if (q < NQ && !(positive(rho) && positive(p))) atomicOr(a.status, 1u);
    const Real* I = sJ + e * 9;
    Real o[4] = {I[0] * x + I[1] * y + I[2] * z, I[3] * x + I[4] * y + I[5] * z, I[6] * x + I[7] * y + I[8] * z, p};
    store_row<4>(sW + (q * EE + e) * 4, o);
}

template <typename Real, int P, int EE>
struct ElemPlan {
    // FP32 projects the deviation from the flux of the element's mean state, which is point NQ, and
    // passes its rows through shared memory
    static constexpr bool F32 = sizeof(Real) == 4;
    static constexpr int ER = rows_of(EE);
    static constexpr int NB = nb_of(P), NQ = nq_of(P), NP = NQ + (F32 ? 1 : 0);
    // shared memory (Reals): point states [NP][ER], (W_0, W_1, W_2, p) [NP][EE][4], then J^-1 [EE][9],
    // |grad lambda_f| [EE][4]; FP32: the tile's coefficients [ER][NB] (the new ones at the end) and
    // its face fluxes, which take the place of the point values once those are projected (P3: 5
    // tiles per SM instead of 2)
    static constexpr int r4(int n) { return (n + 3) / 4 * 4; }   // regions start on 16-byte boundaries
    static constexpr int W = r4(NP * ER), POINTS = W + NP * EE * 4, FACES = F32 ? EE * 20 * nqf_of(P) : 0;
    static constexpr int J = POINTS > FACES ? POINTS : FACES;
    static constexpr int G = J + EE * 9, C = r4(G + EE * 4), REALS = C + (F32 ? ER * NB + 4 : 0);
    static constexpr size_t BYTES = REALS * sizeof(Real);
};

template <typename Real, int P, bool RK, int EE>
__global__ void __launch_bounds__(threads_of(EE)) k_element(ResArgs<Real> a) {
    using S = ElemPlan<Real, P, EE>;
    constexpr int ER = S::ER, NT = threads_of(EE);
    constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), NM = modal::Tables<P>::NM;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* sU = reinterpret_cast<Real*>(smem);
    Real* sW = sU + S::W;
    Real* sJ = sU + S::J;
    Real* sG = sU + S::G;
    Real* sC = sU + S::C;
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (a.ne - e0) < (int64_t)EE ? (int)(a.ne - e0) : EE;
    const bool live = t < 5 * nel;
    const int64_t row = e0 * 5 + t;
    if (S::F32) {
        copy_tile<NT>(sC, a.U + e0 * 5 * NB, nel * 5 * NB * (int)sizeof(Real));
    }
    for (int i = t; i < nel * 9; i += NT) sJ[i] = a.jinv[e0 * 9 + i];
    if (S::F32) {
        tc::cp_async_wait_all();
        __syncthreads();
    }
    if (live) {
        Real c[NB];
        load_row<NB>(S::F32 ? sC + t * NB : a.U + row * NB, c);
        modal::interpolate<Real, P, NB, 0, NQ>(c, [&](int q, Real u) { sU[q * ER + t] = u; });
        if (S::F32) sU[NQ * ER + t] = Real(2.449489742783178) * c[0];
    }
    __syncthreads();
    if (t < nel * 4) {   // |grad lambda_f| = 2 |S_f| / |det J|
        const Real* I = sJ + (t >> 2) * 9;
        const int f = t & 3;
        Real g[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) g[d] = f == 0 ? -(I[d] + I[3 + d] + I[6 + d]) : I[3 * (f - 1) + d];
        sG[t] = EulerOps<Real>::sqrt_(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    }
    for (int i = t; i < S::NP * EE; i += NT) contravariant_point<Real, EE, ER>(a, nel, i, NQ, sU, sW, sJ);
    __syncthreads();
    const int e = t / 5, v = t - 5 * e;
    // G_k of variable v: W_k b + p J_k, b = U_v (+ p for the energy), J_k = (J^-1)_k,v-1 for a momentum
    const Real s4 = v == 4 ? Real(1) : Real(0);
    Real Jk[3], M[3][NM], G0[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Jk[k] = live && v >= 1 && v <= 3 ? sJ[e * 9 + 3 * k + v - 1] : Real(0);
#pragma unroll
        for (int m = 0; m < NM; ++m) M[k][m] = 0;
    }
    auto flux = [&](int q, Real* g) {
        Real w[4];
        load_row<4>(sW + (q * EE + e) * 4, w);
        const Real b = modal::madd(s4, w[3], sU[q * ER + t]);
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] = modal::madd(w[k], b, modal::madd(w[3], Jk[k], -G0[k]));
    };
    if (live) {
        if (S::F32) flux(NQ, G0);
        modal::unroll<0, NQ>([&](auto qc) {
            constexpr int q = qc.value, m = modal::kT<P>.vmir[q];
            if constexpr (m >= q) {
                Real g[3], gm[3] = {0, 0, 0};
                flux(q, g);
                if (m != q) flux(m, gm);
#pragma unroll
                for (int k = 0; k < 3; ++k) modal::moments<Real, P, NM>(q, g[k], gm[k], M[k]);
            }
        });
    }
    if (S::F32) {
        __syncthreads();
        copy_tile<NT>(sU, a.Hs + e0 * 20 * NQF, nel * 20 * NQF * (int)sizeof(Real));
        tc::cp_async_wait_all();
        __syncthreads();
    }
    if (live) {
        Real r[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) r[j] = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) modal::grad_transposed<Real, P>(k, M[k], r);
        // the lift of -s_f H; a constant flux F has s_f F.n_f = -grad lambda_f . F = -G_f-1 (f = 0:
        // the sum of the three), so its part cancels that of the volume term
        const Real* h = (S::F32 ? sU + e * 20 * NQF : a.Hs + (e0 + e) * 20 * NQF) + v * NQF;
        modal::lift<Real, P>(
            [&](int f, Real* x) {
                load_row<NQF>(h + f * 5 * NQF, x);
                const Real s = -sG[4 * e + f];
                if (!S::F32) return s;
                const Real g = f == 0 ? G0[0] + G0[1] + G0[2] : -G0[f - 1];
#pragma unroll
                for (int q = 0; q < NQF; ++q) x[q] = s * x[q] + g;
                return Real(1);
            },
            r);
        if (RK) {
            Real c[NB];
            load_row<NB>(S::F32 ? sC + t * NB : a.U + row * NB, c);
#pragma unroll
            for (int j = 0; j < NB; ++j) r[j] = a.b * (c[j] + a.dt * r[j]);
            if (!S::F32 && a.a != Real(0)) {
                load_row<NB>(a.U0 + row * NB, c);
#pragma unroll
                for (int j = 0; j < NB; ++j) r[j] += a.a * c[j];
            }
        }
        store_row<NB>(S::F32 ? sC + t * NB : a.out + row * NB, r);
    }
    if constexpr (S::F32) {   // whole lines: out = the tile (+ a U0)
        __syncthreads();
        const int n = nel * 5 * NB;
        for (int i = 4 * t; i < n; i += 4 * NT) {
            float4 x = *reinterpret_cast<const float4*>(sC + i);
            const int64_t g = e0 * 5 * NB + i;
            if (i + 4 <= n) {
                if (RK && a.a != 0.f) {
                    const float4 y = *reinterpret_cast<const float4*>(a.U0 + g);
                    x = make_float4(x.x + a.a * y.x, x.y + a.a * y.y, x.z + a.a * y.z, x.w + a.a * y.w);
                }
                *reinterpret_cast<float4*>(a.out + g) = x;
            } else {   // P2: an odd number of elements leaves two values
                for (int k = 0; i + k < n; ++k) a.out[g + k] = sC[i + k] + (RK && a.a != 0.f ? a.a * a.U0[g + k] : 0.f);
            }
        }
    }
}

template <typename Real, int P, bool RK, int EE>
cudaError_t launch_tiles(const ResArgs<Real>& r, cudaStream_t s) {
    constexpr size_t bytes = ElemPlan<Real, P, EE>::BYTES;
    auto kern = k_element<Real, P, RK, EE>;
    static bool init = false;
    if (!init) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        init = true;
    }
    kern<<<(unsigned)((r.ne + EE - 1) / EE), threads_of(EE), bytes, s>>>(r);
    return cudaGetLastError();
}

// Four warps share the rows of a tile of 6 elements (FP64).  A scheduler's FP64 pipe takes a warp's
// instruction every 64 clocks however many of its lanes are active, so on a mesh of few tiles the time
// is the instruction count of one warp: each of the four interpolates to a quarter of the volume points;
// three take one component of the flux's moments each and the fourth the face moments; each
// sums a quarter of the modes.  Every sum runs in the order of k_element, with the same fused operations,
// so the results are bitwise its own (a partition may take this kernel where the whole mesh does not).
// P3 (one warp per tile before), 162 elements: 72 -> 31 us, an SSP-RK3 step 282 -> 176 us; 1,296: 298 -> 232; 2,058:
// 316 -> 300; 3,072: 372 -> 391, so the line lies between, at two and a half tiles per SM.
constexpr int WIDE = 4;
constexpr int64_t WIDE_MAX_NE = 16 * 152;

// f(integral_constant w) for a warp's number w < WIDE
template <typename F>
__device__ __forceinline__ void by_warp(int w, F&& f) {
    if (w == 0) f(std::integral_constant<int, 0>());
    else if (w == 1) f(std::integral_constant<int, 1>());
    else if (w == 2) f(std::integral_constant<int, 2>());
    else f(std::integral_constant<int, 3>());
}

template <int P, bool RK>
__global__ void __launch_bounds__(32 * WIDE) k_element_wide(ResArgs<double> a) {
    using Real = double;
    constexpr int EE = 6, ER = rows_of(EE), NT = 32 * WIDE;
    constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), NM = modal::Tables<P>::NM, NF = modal::Tables<P>::NF;
    __shared__ __align__(16) Real sW[NQ * EE * 4];           // (W_0, W_1, W_2, p) at the points
    __shared__ Real sU[NQ * ER], sM[3 * NM * ER], sA[4 * NF * ER], sJ[EE * 9], sG[EE * 4];
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (a.ne - e0) < (int64_t)EE ? (int)(a.ne - e0) : EE;
    const bool live = l < 5 * nel;
    const int64_t row = e0 * 5 + l;
    const int e = l / 5, v = l - 5 * e;
    for (int i = t; i < nel * 9; i += NT) sJ[i] = a.jinv[e0 * 9 + i];
    if (live) {
        Real c[NB];
        load_row<NB>(a.U + row * NB, c);
        by_warp(w, [&](auto wc) {
            modal::interpolate<Real, P, NB, 0, NQ, wc.value, WIDE>(c, [&](int q, Real u) { sU[q * ER + l] = u; });
        });
    }
    __syncthreads();
    if (t < nel * 4) sG[t] = face_scale(sJ + (t >> 2) * 9, t & 3);
    for (int i = t; i < NQ * EE; i += NT) contravariant_point<Real, EE, ER>(a, nel, i, NQ, sU, sW, sJ);
    __syncthreads();
    if (live && w < 3) {
        const Real s4 = v == 4 ? Real(1) : Real(0), Jk = v >= 1 && v <= 3 ? sJ[e * 9 + 3 * w + v - 1] : Real(0), G0 = 0;
        Real M[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) M[m] = 0;
        auto flux = [&](int q) {
            const Real wk = sW[(q * EE + e) * 4 + w], p = sW[(q * EE + e) * 4 + 3];
            return modal::madd(wk, modal::madd(s4, p, sU[q * ER + l]), modal::madd(p, Jk, -G0));
        };
        modal::unroll<0, NQ>([&](auto qc) {
            constexpr int q = qc.value, m = modal::kT<P>.vmir[q];
            if constexpr (m >= q) {
                const Real g = flux(q), gm = m != q ? flux(m) : Real(0);
                modal::moments<Real, P, NM>(q, g, gm, M);
            }
        });
#pragma unroll
        for (int m = 0; m < NM; ++m) sM[(w * NM + m) * ER + l] = M[m];
    } else if (live) {
        const Real* h = a.Hs + (e0 + e) * 20 * NQF + v * NQF;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            Real x[NQF], b[NF];
            load_row<NQF>(h + f * 5 * NQF, x);
            modal::face_moments<Real, P>(x, b);
#pragma unroll
            for (int m = 0; m < NF; ++m) sA[(f * NF + m) * ER + l] = b[m];
        }
    }
    __syncthreads();
    if (!live) return;
    by_warp(w, [&](auto wc) {
        constexpr auto& T = modal::kT<P>;
        constexpr int J0 = NB * wc.value / WIDE, J1 = NB * (wc.value + 1) / WIDE;
        Real r[J1 - J0];
#pragma unroll
        for (int j = J0; j < J1; ++j) r[j - J0] = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                const Real s = sM[(k * NM + m) * ER + l];
#pragma unroll
                for (int j = J0; j < J1; ++j) modal::axpy(r[j - J0], T.D[k][m][j], s);
            }
        // modal::lift of the moments, the faces' scales as its factors
        const Real s0 = -sG[4 * e], s1 = -sG[4 * e + 1];
#pragma unroll
        for (int m = 0; m < NF; ++m) {
            const Real x = s0 * sA[m * ER + l], b = sA[(NF + m) * ER + l], ev = modal::madd(s1, b, x), od = modal::madd(s1, b, -x);
#pragma unroll
            for (int j = J0; j < J1; ++j) modal::axpy(r[j - J0], T.E[1][m][j], T.odd[j] ? od : ev);
        }
#pragma unroll
        for (int f = 2; f < 4; ++f) {
            const Real s = -sG[4 * e + f];
#pragma unroll
            for (int m = 0; m < NF; ++m) {
                const Real x = s * sA[(f * NF + m) * ER + l];
#pragma unroll
                for (int j = J0; j < J1; ++j) modal::axpy(r[j - J0], T.E[f][m][j], x);
            }
        }
        const int64_t g = row * NB;
#pragma unroll
        for (int j = J0; j < J1; ++j) {
            Real x = r[j - J0];
            if (RK) {
                x = a.b * (a.U[g + j] + a.dt * x);
                if (a.a != Real(0)) x += a.a * a.U0[g + j];
            }
            a.out[g + j] = x;
        }
    });
}

template <typename Real, int P, bool RK>
cudaError_t launch_element(const ResArgs<Real>& r, cudaStream_t s) {
    if constexpr (sizeof(Real) == 8 && P == 3) {
        if (r.ne <= WIDE_MAX_NE) {
            k_element_wide<P, RK><<<(unsigned)((r.ne + 5) / 6), 32 * WIDE, 0, s>>>(r);
            return cudaGetLastError();
        }
    }
    return small_tiles(r.ne) ? launch_tiles<Real, P, RK, 6>(r, s) : launch_tiles<Real, P, RK, 32>(r, s);
}

template <typename Real, int P>
cudaError_t launch_face_once(dg_mesh* m, ResArgs<Real>& r, bool rk, void* T, cudaStream_t s) {
    FaceArgs<Real> f;
    f.T = static_cast<Real*>(T);
    f.rec = m->d_frec;
    f.normal = static_cast<const Real*>(m->d_fnorm);
    f.fperm = m->d_fperm;
    f.n = m->n_flist * nqf_of(P);
    f.gamma = r.gamma;
    f.roe_eps = r.roe_eps;
    for (int v = 0; v < 5; ++v) f.finf[v] = r.finf[v];
    f.status = m->d_status;
    cudaError_t e = traces<Real, P>(r.U, f.T, nullptr, nullptr, m->n_trace, s);
    if (e != cudaSuccess) return e;
    if (f.n > 0) {
        const unsigned nt = face_block(f.n), grid = (unsigned)((f.n + nt - 1) / nt);
        if (m->flux == DG_ROE) k_faces<Real, P, DG_ROE><<<grid, nt, 0, s>>>(f);
        else k_faces<Real, P, DG_RUSANOV><<<grid, nt, 0, s>>>(f);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    r.Hs = f.T;
    return rk ? launch_element<Real, P, true>(r, s) : launch_element<Real, P, false>(r, s);
}

template <typename Real>
cudaError_t dispatch(dg_mesh* m, const void* U, const void* U0, void* out, int mode, double dt, double ca,
                     double cb, void* T, cudaStream_t s) {
    ResArgs<Real> r;
    r.U = static_cast<const Real*>(U);
    r.U0 = static_cast<const Real*>(U0);
    r.out = static_cast<Real*>(out);
    r.nbr = m->d_nbr;
    r.fcode = m->d_fcode;
    r.jinv = static_cast<const Real*>(m->d_jinv);
    r.tab = static_cast<const Real*>(m->d_tab);
    r.fperm = m->d_fperm;
    r.ne = m->host.ne;
    r.dt = (Real)dt;
    r.a = (Real)ca;
    r.b = (Real)cb;
    r.gamma = (Real)m->gamma;
    r.roe_eps = (Real)m->roe_eps;
    for (int v = 0; v < 5; ++v) r.finf[v] = (Real)m->finf[v];
    r.status = m->d_status;
    r.Hs = nullptr;
    const bool rk = mode != 0;
    if (T) {
        switch (m->p) {
            case 1: return launch_face_once<Real, 1>(m, r, rk, T, s);
            case 2: return launch_face_once<Real, 2>(m, r, rk, T, s);
            default: return launch_face_once<Real, 3>(m, r, rk, T, s);
        }
    }
    if constexpr (sizeof(Real) == 8) {
        return cudaErrorInvalidValue;   // FP64 has no other form
    } else {
        int nsm = 0;
        cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
        if (e != cudaSuccess) return e;
        switch (m->p) {
            case 1: return dispatch_flux<Real, 1>(r, m->flux, rk, s, nsm);
            case 2: return dispatch_flux<Real, 2>(r, m->flux, rk, s, nsm);
            default: return dispatch_flux<Real, 3>(r, m->flux, rk, s, nsm);
        }
    }
}

}  // namespace

namespace {
// ---- the face list, from the connectivity on the device (on the host, with a branch per slot that is taken every
// other time, it took 19 of the 240 ms of a 384,000-element creation, and its upload more) ----------

struct ListArgs {
    const int32_t* nbr;     // of the listing mesh, local numbers
    const uint8_t* fcode;
    const int32_t* wnbr;    // the whole mesh's neighbours and caller indices
    const int32_t* perm;
    int64_t ne, first;      // own elements; the first one's number in the whole mesh
};

// whether slot's face is listed from it, among the boundary faces (BND) or the interior ones, and its record
template <bool BND>
__device__ __forceinline__ bool listed(const ListArgs& a, int64_t slot, FaceRec& r) {
    if (slot >= 4 * a.ne) return false;
    const int32_t n = a.nbr[slot], ws = (int32_t)(4 * a.first + slot);
    if (BND) {
        r = {(int32_t)slot, n, 8, ws};
        return n < 0;
    }
    if (n < 0) return false;
    const int c = a.fcode[slot], fn = c & 3;
    const int32_t wn = a.wnbr[ws];
    const bool own = a.perm[wn] > a.perm[ws >> 2];
    r = {(int32_t)slot, 4 * n + fn, (c >> 2) | (own ? 8 : 0), own ? ws : 4 * wn + fn};
    return own || n >= a.ne;   // else listed on the owner's side
}

constexpr int LT = 256;

template <bool BND>
__global__ void __launch_bounds__(LT) k_list_count(ListArgs a, int32_t* counts) {
    FaceRec r;
    const int n = __syncthreads_count(listed<BND>(a, blockIdx.x * (int64_t)LT + threadIdx.x, r));
    if (threadIdx.x == 0) counts[blockIdx.x] = n;
}

// exclusive sums, in place: one block, a piece of 1,024 after the other
__global__ void __launch_bounds__(1024) k_list_scan(int32_t* counts, int64_t n) {
    __shared__ int32_t s[1024];
    __shared__ int32_t carry;
    const int t = threadIdx.x;
    if (t == 0) carry = 0;
    for (int64_t base = 0; base < n; base += 1024) {
        const int32_t x = base + t < n ? counts[base + t] : 0;
        s[t] = x;
        __syncthreads();
        for (int d = 1; d < 1024; d *= 2) {
            const int32_t y = t >= d ? s[t - d] : 0;
            __syncthreads();
            s[t] += y;
            __syncthreads();
        }
        const int32_t c = carry, total = s[1023];
        if (base + t < n) counts[base + t] = c + s[t] - x;
        __syncthreads();
        if (t == 0) carry = c + total;
        __syncthreads();
    }
}

template <bool BND>
__global__ void __launch_bounds__(LT) k_list_write(ListArgs a, const int32_t* counts, FaceRec* out, int64_t n) {
    __shared__ int32_t warp_n[LT / 32];
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    FaceRec r;
    const bool on = listed<BND>(a, blockIdx.x * (int64_t)LT + t, r);
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (l == 0) warp_n[w] = __popc(m);
    __syncthreads();
    int64_t at = counts[blockIdx.x] + __popc(m & ((1u << l) - 1u));
    for (int k = 0; k < w; ++k) at += warp_n[k];
    if (on && at < n) out[at] = r;
}

template <bool BND>
cudaError_t list_faces(const ListArgs& a, int32_t* counts, FaceRec* out, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const unsigned nblk = (unsigned)((4 * a.ne + LT - 1) / LT);
    k_list_count<BND><<<nblk, LT, 0, s>>>(a, counts);
    k_list_scan<<<1, 1024, 0, s>>>(counts, nblk);
    k_list_write<BND><<<nblk, LT, 0, s>>>(a, counts, out, n);
    return cudaGetLastError();
}

// per listed face the owner's outward unit normal -grad lambda_f / |grad lambda_f| and, with scales, the
// |grad lambda| of the slot's element and of the matching one
template <typename Real>
__global__ void k_face_geometry(const double* __restrict__ jinv, const FaceRec* __restrict__ rec, int64_t n, Real* normal,
                                Real* scale) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    auto gradient = [&](int32_t slot, double* g) {
        const double* I = jinv + (int64_t)(slot >> 2) * 9;
        const int f = slot & 3;
        for (int d = 0; d < 3; ++d) g[d] = f == 0 ? -(I[d] + I[3 + d] + I[6 + d]) : I[3 * (f - 1) + d];
        return sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    };
    const FaceRec r = rec[i];
    double g[3];
    const double gn = gradient(r.owner, g);
    for (int d = 0; d < 3; ++d) normal[3 * i + d] = (Real)(-g[d] / gn);
    if (!scale) return;
    scale[2 * i] = (Real)gradient(r.slot, g);
    scale[2 * i + 1] = r.other >= 0 ? (Real)gradient(r.other, g) : Real(0);
}
}  // namespace

size_t face_list_bytes(int64_t n, int precision, bool scales) {
    return n * (sizeof(FaceRec) + (scales ? 5 : 3) * (precision == DG_FP64 ? 8 : 4));
}

cudaError_t setup_face_once(dg_mesh* m, const dg_mesh* whole, int64_t first, int64_t n_trace, bool scales, cudaStream_t s) {
    const int64_t slots = 4 * m->host.ne;
    int32_t nbnd = 0, nhalo = 0;
    for (int64_t i = 0; i < slots; ++i) {
        nbnd += m->host.nbr[i] < 0;
        nhalo += m->host.nbr[i] >= (int32_t)m->host.ne;
    }
    m->n_interior = (slots - nbnd - nhalo) / 2 + nhalo;
    const int64_t n = m->n_flist = m->n_interior + nbnd;
    m->n_trace = n_trace;
    cudaError_t e = cudaMalloc(&m->d_frec, face_list_bytes(n, m->precision, scales));   // records, normals, scales
    if (e != cudaSuccess) return e;
    const bool f64 = m->precision == DG_FP64;
    m->d_fnorm = m->d_frec + n;
    m->d_fscale = scales ? static_cast<char*>(m->d_fnorm) + 3 * n * (f64 ? 8 : 4) : nullptr;
    const ListArgs a{m->d_nbr, m->d_fcode, whole->d_nbr, whole->d_perm, m->host.ne, first};
    // the normals' place, written last, holds the counts: at least 24 bytes an element (n >= 2 ne) against 4 per LT slots
    int32_t* counts = static_cast<int32_t*>(m->d_fnorm);
    e = list_faces<false>(a, counts, m->d_frec, m->n_interior, s);
    if (e == cudaSuccess) e = list_faces<true>(a, counts, m->d_frec + m->n_interior, nbnd, s);
    if (e == cudaSuccess) {
        const unsigned grid = (unsigned)((n + 255) / 256);
        if (f64)
            k_face_geometry<double><<<grid, 256, 0, s>>>(whole->d_jinv64, m->d_frec, n, static_cast<double*>(m->d_fnorm),
                                                         static_cast<double*>(m->d_fscale));
        else
            k_face_geometry<float><<<grid, 256, 0, s>>>(whole->d_jinv64, m->d_frec, n, static_cast<float*>(m->d_fnorm),
                                                        static_cast<float*>(m->d_fscale));
        e = cudaGetLastError();
    }
    m->face_once = e == cudaSuccess;
    return e;   // a mesh whose launch failed is given up
}

cudaError_t launch_traces2(dg_mesh* m, const void* U, void* T, const void* U1, void* T1, cudaStream_t s) {
    const int64_t n = m->host.ne;
    const bool f64 = m->precision == DG_FP64;
    switch (m->p) {
        case 1: return f64 ? traces<double, 1>(U, T, U1, T1, n, s) : traces<float, 1>(U, T, U1, T1, n, s);
        case 2: return f64 ? traces<double, 2>(U, T, U1, T1, n, s) : traces<float, 2>(U, T, U1, T1, n, s);
        default: return f64 ? traces<double, 3>(U, T, U1, T1, n, s) : traces<float, 3>(U, T, U1, T1, n, s);
    }
}

cudaError_t launch_residual(dg_mesh* m, const void* U, const void* U0, void* out, int mode, double dt, double a,
                            double b, void* T, cudaStream_t s) {
    if (m->precision == DG_FP64) return dispatch<double>(m, U, U0, out, mode, dt, a, b, T, s);
    return dispatch<float>(m, U, U0, out, mode, dt, a, b, T, s);
}

}  // namespace dg
