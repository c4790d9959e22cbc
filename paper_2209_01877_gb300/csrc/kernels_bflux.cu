// Boundary-flux integral: B_v = sum over boundary faces f of int_f H_v(Q-, Q_b, n) dS, the
// boundary-face line of Eq. 11 taken with the constant test function.  Interior face fluxes
// cancel in pairs, so d/dt int U_v dx = -B_v; the conservation bookkeeping of a run with
// walls and far-field faces integrates B over the RK stages.
//
// FP64 throughout, whatever the mesh's precision (the stored state is read as FP64, FP32, or
// the float-float pair of the mixed form): one thread per boundary face and quadrature point
// evaluates the trace, the ghost state (slip wall or characteristic far field) and the numerical
// flux (Rusanov or Roe), weighted by wf_q 2|S_f|; then a fixed-order two-pass sum (block, then one
// block over the block sums), so the result does not depend on timing.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "dg_internal.h"
#include "euler_device.cuh"

namespace dg {

namespace {

constexpr int BT = 256;
constexpr int MAX_BLOCKS = 1024;

__device__ __forceinline__ double det3x3(const double* A) {
    return A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) + A[2] * (A[3] * A[7] - A[4] * A[6]);
}

// Blocks of BF boundary faces, thread per (face, point): the faces' elements' coefficients and face
// basis in shared memory in FP64 (each coefficient converted once), block partials in a fixed order.
// Bound by the FP64 pipe; one thread per face, reading tables and coefficients per point, took 764 us
// for the 10,368 boundary faces of a 165,888-element P3 channel in the mixed form.
constexpr int BF = 16;

template <typename Real, int P, int FLUX>
__global__ void __launch_bounds__(BF * nqf_of(P)) k_bflux_local(const Real* __restrict__ U, const Real* __restrict__ Ulo,
                                                                const double* __restrict__ jinv, const double* __restrict__ tab,
                                                                const int32_t* __restrict__ bface, const int32_t* __restrict__ nbr,
                                                                int64_t nbf, double gamma, double eps, double f0, double f1,
                                                                double f2, double f3, double f4, double* __restrict__ block_sum) {
    constexpr int NB = nb_of(P), NQF = nqf_of(P), NT = BF * NQF, NV = 5 * NB;
    constexpr TabLayout L(P);   // followed by the volume points (3 NQ) and the face weights
    __shared__ double sC[BF][NV];
    __shared__ double sP[4 * NB * NQF];
    __shared__ double red[5][NT];
    const double finf[5] = {f0, f1, f2, f3, f4};
    const int t = threadIdx.x, b = t / NQF, q = t - b * NQF;
    for (int i = t; i < 4 * NB * NQF; i += NT) sP[i] = tab[L.phif + i];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int64_t g = blockIdx.x * (int64_t)BF; g < nbf; g += (int64_t)gridDim.x * BF) {
        const int nf = nbf - g < BF ? (int)(nbf - g) : BF;
        __syncthreads();
        for (int i = t; i < nf * NV; i += NT) {
            const int k = i / NV, j = i - k * NV;
            const int64_t at = (int64_t)(bface[g + k] >> 2) * NV + j;
            sC[k][j] = (double)U[at] + (Ulo ? (double)Ulo[at] : 0.0);
        }
        __syncthreads();
        if (b >= nf) continue;
        const int32_t code = bface[g + b];
        const int64_t e = code >> 2;
        const int f = code & 3;
        const int btype = -1 - nbr[e * 4 + f];
        const double* I = jinv + 9 * e;
        // grad_x lambda_f: row f - 1 of J^-1, and minus the sum of the rows for f = 0
        double gl[3];
        for (int d = 0; d < 3; ++d) gl[d] = f == 0 ? -(I[d] + I[3 + d] + I[6 + d]) : I[3 * (f - 1) + d];
        const double gn = sqrt(gl[0] * gl[0] + gl[1] * gl[1] + gl[2] * gl[2]);
        const double n[3] = {-gl[0] / gn, -gl[1] / gn, -gl[2] / gn};
        // 2 |S_f| = |grad lambda_f| |det J|
        const double w = tab[L.total + 3 * nq_of(P) + q] * (gn / fabs(det3x3(I)));
        double Um[5], G[5], H[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < NB; ++j) s += sC[b][v * NB + j] * sP[(f * NB + j) * NQF + q];
            Um[v] = s;
        }
        if (btype == DG_BC_WALL) wall_ghost(Um, n, G);
        else farfield_ghost(Um, n, finf, gamma, G);
        if (FLUX == DG_ROE) roe_flux(Um, G, n, gamma, eps, H);
        else rusanov_flux(Um, G, n, gamma, H);
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[v] += w * H[v];
    }
    for (int v = 0; v < 5; ++v) red[v][t] = acc[v];
    __syncthreads();
    // the block's sum: 16 partial sums per variable over the threads t = k (mod 16), then over k
    for (int u = t; u < 80; u += NT) {
        const int vv = u / 16, kk = u - 16 * vv;
        double s = 0.0;
        for (int i = kk; i < NT; i += 16) s += red[vv][i];
        red[vv][kk] = s;   // entry kk belongs to this sum alone
    }
    __syncthreads();
    if (t < 5) {
        double s = 0.0;
        for (int i = 0; i < 16; ++i) s += red[t][i];
        block_sum[blockIdx.x * 5 + t] = s;
    }
}

// the conservative mixed mode's own boundary flux: per boundary slot 4 e + f, the face's 2|S_f|
// times the flux integral the last stage used (one value per face, as in the mode-0 update)
__global__ void __launch_bounds__(BT) k_applied_bflux_local(const float* __restrict__ hs,
                                                            const double* __restrict__ farea,
                                                            const int32_t* __restrict__ bface, int64_t nbf,
                                                            double* __restrict__ block_sum) {
    __shared__ double red[5][BT];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int64_t i = blockIdx.x * (int64_t)BT + threadIdx.x; i < nbf; i += (int64_t)gridDim.x * BT) {
        const int64_t sl = bface[i];
        for (int v = 0; v < 5; ++v) acc[v] += farea[sl] * (double)hs[sl * 5 + v];
    }
    for (int v = 0; v < 5; ++v) red[v][threadIdx.x] = acc[v];
    __syncthreads();
    for (int s = BT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int v = 0; v < 5; ++v) red[v][threadIdx.x] += red[v][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 5) block_sum[blockIdx.x * 5 + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void __launch_bounds__(BT) k_bflux_final(const double* __restrict__ in, int nblk, double* __restrict__ out) {
    __shared__ double red[5][BT];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblk; b += BT)
        for (int v = 0; v < 5; ++v) acc[v] += in[b * 5 + v];
    for (int v = 0; v < 5; ++v) red[v][threadIdx.x] = acc[v];
    __syncthreads();
    for (int s = BT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int v = 0; v < 5; ++v) red[v][threadIdx.x] += red[v][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 5) out[threadIdx.x] = red[threadIdx.x][0];
}

}  // namespace

// d_partial holds at least 5 * 1024 doubles; d_out5 receives B
cudaError_t launch_boundary_flux(dg_mesh* m, const void* U, double* d_partial, double* d_out5, cudaStream_t s) {
    const int64_t nbf = m->host.n_bfaces;
    int nblk = (int)std::min<int64_t>((nbf + BF - 1) / BF, MAX_BLOCKS);
    if (nblk < 1) nblk = 1;
    const int64_t n = m->host.ne * 5 * m->nb;
    const double* fi = m->finf;
    auto go = [&](auto p, auto fl) {
        constexpr int P = decltype(p)::value, FL = decltype(fl)::value, NT = BF * nqf_of(P);
        if (m->precision == DG_FP64) {
            k_bflux_local<double, P, FL><<<nblk, NT, 0, s>>>(static_cast<const double*>(U), nullptr, m->d_jinv64, m->d_tab64,
                                                             m->d_bface, m->d_nbr, nbf, m->gamma, m->roe_eps, fi[0], fi[1],
                                                             fi[2], fi[3], fi[4], d_partial);
        } else {
            const float* u = static_cast<const float*>(U);
            k_bflux_local<float, P, FL><<<nblk, NT, 0, s>>>(u, m->precision == DG_FP32 ? nullptr : u + n, m->d_jinv64,
                                                            m->d_tab64, m->d_bface, m->d_nbr, nbf, m->gamma, m->roe_eps,
                                                            fi[0], fi[1], fi[2], fi[3], fi[4], d_partial);
        }
    };
    auto order = [&](auto fl) {
        if (m->p == 1) go(std::integral_constant<int, 1>(), fl);
        else if (m->p == 2) go(std::integral_constant<int, 2>(), fl);
        else go(std::integral_constant<int, 3>(), fl);
    };
    if (m->flux == DG_ROE) order(std::integral_constant<int, DG_ROE>());
    else order(std::integral_constant<int, DG_RUSANOV>());
    k_bflux_final<<<1, BT, 0, s>>>(d_partial, nblk, d_out5);
    return cudaGetLastError();
}

cudaError_t launch_applied_boundary_flux(dg_mesh* m, double* d_partial, double* d_out5, cudaStream_t s) {
    const int64_t nbf = m->host.n_bfaces;
    int nblk = (int)std::min<int64_t>((nbf + BT - 1) / BT, MAX_BLOCKS);
    if (nblk < 1) nblk = 1;
    k_applied_bflux_local<<<nblk, BT, 0, s>>>(m->d_hs, m->d_farea, m->d_bface, nbf, d_partial);
    k_bflux_final<<<1, BT, 0, s>>>(d_partial, nblk, d_out5);
    return cudaGetLastError();
}

}  // namespace dg
