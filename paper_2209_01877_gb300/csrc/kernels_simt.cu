// Residual and SSP-RK3 stage on the CUDA cores (FP64 and FP32), with every face's traces and
// numerical flux evaluated once.  Three launches per residual or stage:
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
// 1,296 elements 85 -> 62 us.
#include <algorithm>

#include "dg_internal.h"
#include "euler_device.cuh"
#include "face_flux.cuh"
#include "modal_ops.cuh"

namespace dg {

namespace {

constexpr int NT = 256;

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

constexpr int TT = 128;   // threads of k_traces
constexpr int FT = 128;   // threads of k_faces

// the trace of every (element, face, point): thread per (element, variable) row
template <typename Real, int P>
__global__ void __launch_bounds__(TT) k_traces(const Real* __restrict__ U, Real* __restrict__ T, int64_t nrow) {
    constexpr int NB = nb_of(P), NQF = nqf_of(P);
    const int64_t row = blockIdx.x * (int64_t)TT + threadIdx.x;
    if (row >= nrow) return;
    const int64_t e = row / 5;
    const int v = (int)(row - 5 * e);
    Real c[NB];
    load_row<NB>(U + row * NB, c);
    Real* t = T + (e * 20 + v) * NQF;
    modal::traces<Real, P>(c, [&](int f, const Real* u) { store_row<NQF>(t + f * 5 * NQF, u); });
}

template <typename Real>
struct FaceArgs {
    Real* T;                // face buffer [n_trace][4][5][Nqf]: traces in, fluxes out
    const Real* ncan;       // [ne][4][3] the owner's outward normal
    const uint8_t* fown;    // [ne][4] 1 where the slot's element owns the face
    const int32_t* flist;   // slots 4 e + f whose face this mesh evaluates, boundary faces last
    const int32_t* nbr;
    const uint8_t* fcode;
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
    const int64_t i = blockIdx.x * (int64_t)FT + threadIdx.x;
    if (i >= a.n) return;
    const int64_t li = i / NQF;
    const int q = (int)(i - li * NQF);
    const int64_t slot = a.flist[li];
    const Real* nc = a.ncan + slot * 3;
    const Real nv[3] = {nc[0], nc[1], nc[2]};
    Real* te = a.T + slot * 5 * NQF + q;
    Real Ue[5], Un[5], H[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) Ue[v] = te[v * NQF];
    const int32_t n = a.nbr[slot];
    bool okL, okR;
    if (n < 0) {
        if (n == -1 - DG_BC_WALL) wall_ghost(Ue, nv, Un);
        else farfield_ghost(Ue, nv, a.finf, a.gamma, Un);
        face_flux<Real, FLUX>(Ue, Un, nv, a.gamma, a.roe_eps, H, okL, okR);
        if (!okL) atomicOr(a.status, 1u);
#pragma unroll
        for (int v = 0; v < 5; ++v) te[v * NQF] = H[v];
        return;
    }
    const int code = a.fcode[slot];
    const int qn = a.fperm[(code >> 2) * NQF + q];
    Real* tn = a.T + ((int64_t)n * 4 + (code & 3)) * 5 * NQF + qn;
#pragma unroll
    for (int v = 0; v < 5; ++v) Un[v] = tn[v * NQF];
    const bool own = a.fown[slot] != 0;   // false only for a face shared with a halo element that owns it
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

constexpr int EE = 32;        // elements per tile of k_element
constexpr int ER = 5 * EE;    // rows (element, variable) = threads

template <typename Real, int P>
struct ElemPlan {
    static constexpr int NQ = nq_of(P);
    // shared memory (Reals): point states [NQ][ER], (W_0, W_1, W_2, p) [NQ][EE][4], J^-1 [EE][9],
    // |grad lambda_f| [EE][4]
    static constexpr int W = NQ * ER, J = W + NQ * EE * 4, G = J + EE * 9, REALS = G + EE * 4;
    static constexpr size_t BYTES = REALS * sizeof(Real);
};

template <typename Real, int P, bool RK>
__global__ void __launch_bounds__(ER) k_element(ResArgs<Real> a) {
    using S = ElemPlan<Real, P>;
    constexpr int NB = nb_of(P), NQ = nq_of(P), NQF = nqf_of(P), NM = modal::Tables<P>::NM;
    extern __shared__ __align__(16) unsigned char smem[];
    Real* sU = reinterpret_cast<Real*>(smem);
    Real* sW = sU + S::W;
    Real* sJ = sU + S::J;
    Real* sG = sU + S::G;
    const int t = threadIdx.x;
    const int64_t e0 = blockIdx.x * (int64_t)EE;
    const int nel = (a.ne - e0) < (int64_t)EE ? (int)(a.ne - e0) : EE;
    const bool live = t < 5 * nel;
    const int64_t row = e0 * 5 + t;
    for (int i = t; i < nel * 9; i += ER) sJ[i] = a.jinv[e0 * 9 + i];
    if (live) {
        Real c[NB], u[NQ];
        load_row<NB>(a.U + row * NB, c);
        modal::interpolate<Real, P>(c, u);
#pragma unroll
        for (int q = 0; q < NQ; ++q) sU[q * ER + t] = u[q];
    }
    __syncthreads();
    // |grad lambda_f| = 2 |S_f| / |det J|, by the threads that the point loop below leaves idle last
    if (t < nel * 4) {
        const Real* I = sJ + (t >> 2) * 9;
        const int f = t & 3;
        Real g[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) g[d] = f == 0 ? -(I[d] + I[3 + d] + I[6 + d]) : I[3 * (f - 1) + d];
        sG[t] = EulerOps<Real>::sqrt_(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    }
    // contravariant velocity W_k = sum_d (J^-1)_kd u_d and pressure at every (element, point)
    for (int i = t; i < NQ * EE; i += ER) {
        const int e = i % EE, q = i / EE;
        if (e >= nel) continue;
        const Real* u = sU + q * ER + 5 * e;
        const Real rho = u[0], ri = recip(rho);
        const Real x = u[1] * ri, y = u[2] * ri, z = u[3] * ri;
        const Real p = (a.gamma - Real(1)) * (u[4] - Real(0.5) * (u[1] * x + u[2] * y + u[3] * z));
        if (!(positive(rho) && positive(p))) atomicOr(a.status, 1u);
        const Real* I = sJ + e * 9;
        Real* w = sW + (q * EE + e) * 4;
        Real o[4] = {I[0] * x + I[1] * y + I[2] * z, I[3] * x + I[4] * y + I[5] * z, I[6] * x + I[7] * y + I[8] * z, p};
        store_row<4>(w, o);
    }
    __syncthreads();
    if (!live) return;
    const int e = t / 5, v = t - 5 * e;
    // G_k of variable v: W_k a + p J_k, a = U_v (+ p for the energy), J_k = (J^-1)_k,v-1 for a momentum
    const Real s4 = v == 4 ? Real(1) : Real(0);
    Real Jk[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) Jk[k] = v >= 1 && v <= 3 ? sJ[e * 9 + 3 * k + v - 1] : Real(0);
    Real M[3][NM];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int m = 0; m < NM; ++m) M[k][m] = 0;
    auto flux = [&](int q, Real* g) {
        Real w[4];
        load_row<4>(sW + (q * EE + e) * 4, w);
        const Real b = sU[q * ER + t] + s4 * w[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] = w[k] * b + w[3] * Jk[k];
    };
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int m = modal::kT<P>.vmir[q];
        if (m < q) continue;
        Real g[3], gm[3] = {0, 0, 0};
        flux(q, g);
        if (m != q) flux(m, gm);
#pragma unroll
        for (int k = 0; k < 3; ++k) modal::moments<Real, P, NM>(q, g[k], gm[k], M[k]);
    }
    Real r[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) r[j] = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) modal::grad_transposed<Real, P>(k, M[k], r);
    const Real s[4] = {-sG[4 * e], -sG[4 * e + 1], -sG[4 * e + 2], -sG[4 * e + 3]};
    const Real* h = a.Hs + ((e0 + e) * 20 + v) * NQF;
    modal::lift<Real, P>([&](int f, Real* x) { load_row<NQF>(h + f * 5 * NQF, x); }, s, r);
    if (RK) {
        Real c[NB];
        load_row<NB>(a.U + row * NB, c);
#pragma unroll
        for (int j = 0; j < NB; ++j) r[j] = a.b * (c[j] + a.dt * r[j]);
        if (a.a != Real(0)) {
            load_row<NB>(a.U0 + row * NB, c);
#pragma unroll
            for (int j = 0; j < NB; ++j) r[j] += a.a * c[j];
        }
    }
    store_row<NB>(a.out + row * NB, r);
}

template <typename Real, int P, bool RK>
cudaError_t launch_element(const ResArgs<Real>& r, cudaStream_t s) {
    constexpr size_t bytes = ElemPlan<Real, P>::BYTES;
    auto kern = k_element<Real, P, RK>;
    static bool init = false;
    if (!init) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        init = true;
    }
    kern<<<(unsigned)((r.ne + EE - 1) / EE), ER, bytes, s>>>(r);
    return cudaGetLastError();
}

template <typename Real, int P>
cudaError_t launch_face_once(dg_mesh* m, ResArgs<Real>& r, bool rk, cudaStream_t s) {
    FaceArgs<Real> f;
    f.T = static_cast<Real*>(m->d_T);
    f.ncan = static_cast<const Real*>(m->d_ncan);
    f.fown = m->d_fown;
    f.flist = m->d_flist;
    f.nbr = m->d_nbr;
    f.fcode = m->d_fcode;
    f.fperm = m->d_fperm;
    f.n = m->n_flist * nqf_of(P);
    f.gamma = r.gamma;
    f.roe_eps = r.roe_eps;
    for (int v = 0; v < 5; ++v) f.finf[v] = r.finf[v];
    f.status = m->d_status;
    const int64_t nrow = 5 * m->n_trace;
    k_traces<Real, P><<<(unsigned)((nrow + TT - 1) / TT), TT, 0, s>>>(r.U, f.T, nrow);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (f.n > 0) {
        const unsigned grid = (unsigned)((f.n + FT - 1) / FT);
        if (m->flux == DG_ROE) k_faces<Real, P, DG_ROE><<<grid, FT, 0, s>>>(f);
        else k_faces<Real, P, DG_RUSANOV><<<grid, FT, 0, s>>>(f);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    r.Hs = f.T;
    return rk ? launch_element<Real, P, true>(r, s) : launch_element<Real, P, false>(r, s);
}

template <typename Real>
cudaError_t dispatch(dg_mesh* m, const void* U, const void* U0, void* out, int mode, double dt, double ca,
                     double cb, cudaStream_t s) {
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
    if (m->face_once) {
        switch (m->p) {
            case 1: return launch_face_once<Real, 1>(m, r, rk, s);
            case 2: return launch_face_once<Real, 2>(m, r, rk, s);
            default: return launch_face_once<Real, 3>(m, r, rk, s);
        }
    }
    if constexpr (sizeof(Real) == 8) {
        return cudaErrorInvalidValue;   // FP64 meshes always hold a face buffer
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

cudaError_t setup_face_once(dg_mesh* m, const std::vector<uint8_t>& fown, const std::vector<double>& ncan,
                            int64_t n_trace, cudaStream_t s) {
    const int64_t ne = m->host.ne;
    std::vector<int32_t> list;
    // owned, or shared with a halo; boundary faces last, so that warps mostly run one kind
    for (int kind = 0; kind < 2; ++kind)
        for (int64_t sl = 0; sl < 4 * ne; ++sl)
            if ((fown[sl] || m->host.nbr[sl] >= ne) && (m->host.nbr[sl] < 0) == (kind == 1)) list.push_back((int32_t)sl);
    const size_t rbytes = m->precision == DG_FP64 ? sizeof(double) : sizeof(float);
    std::vector<float> n32;
    const void* nsrc = ncan.data();
    if (rbytes == sizeof(float)) {
        n32.assign(ncan.begin(), ncan.end());
        nsrc = n32.data();
    }
    cudaError_t e = cudaMalloc(&m->d_fown, fown.size());
    if (e == cudaSuccess) e = cudaMalloc(&m->d_ncan, ncan.size() * rbytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->d_flist, std::max<size_t>(list.size(), 1) * sizeof(int32_t));
    const size_t buf = (size_t)n_trace * 4 * m->nqf * 5 * rbytes;
    if (e == cudaSuccess) e = cudaMalloc(&m->d_T, buf);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->d_fown, fown.data(), fown.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->d_ncan, nsrc, ncan.size() * rbytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && !list.empty())
        e = cudaMemcpyAsync(m->d_flist, list.data(), list.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the host vectors go out of scope
    if (e != cudaSuccess) return e;
    m->n_flist = (int64_t)list.size();
    m->n_trace = n_trace;
    m->face_once = true;
    return cudaSuccess;
}

cudaError_t launch_residual(dg_mesh* m, const void* U, const void* U0, void* out, int mode, double dt, double a,
                            double b, cudaStream_t s) {
    if (m->precision == DG_FP64) return dispatch<double>(m, U, U0, out, mode, dt, a, b, s);
    return dispatch<float>(m, U, U0, out, mode, dt, a, b, s);
}

}  // namespace dg
