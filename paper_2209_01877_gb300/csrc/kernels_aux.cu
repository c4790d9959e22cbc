// Auxiliary kernels: caller-order <-> internal-order state copies, the
// time-step reduction (Sec. III-C: local steps, then the global minimum by a
// two-pass block reduction), conservation / kinetic-energy integrals
// (fixed-order two-pass sums in FP64), L2 projection of pointwise values and
// the physical coordinates of the volume points.
#include <algorithm>
#include <cmath>

#include "dg_internal.h"
#include "ff_bits.cuh"
#include "modal_ops.cuh"

namespace dg {

namespace {

constexpr int RT = 256;   // reduction block size
constexpr double SQRT6 = 2.449489742783178098197284;

// ---- caller order <-> internal order ------------------------------------------------------------
// A block moves 32 elements (8 on a small mesh), a thread two values at a time, 16 bytes of the caller's FP64 array where
// that is aligned (8 where a caller's pointer is not).  Bound by memory; one value per thread with a
// 64-bit division per value was bound by issue: FP32 P3, 14,586 elements 12 us per call.
enum { MOVE_F64 = 0, MOVE_F32 = 1, MOVE_FF = 2 };   // internal format; FF: hi plane, then lo plane
constexpr int MT2 = 256;

template <bool VEC>
__device__ __forceinline__ double2 load2(const double* p) {
    if constexpr (VEC) return *reinterpret_cast<const double2*>(p);
    else return make_double2(p[0], p[1]);
}
template <bool VEC>
__device__ __forceinline__ void store2(double* p, double2 x) {
    if constexpr (VEC) {
        *reinterpret_cast<double2*>(p) = x;
    } else {
        p[0] = x.x;
        p[1] = x.y;
    }
}

template <int NV, int FMT, bool VEC, int ME>
__global__ void __launch_bounds__(MT2) k_gather(const double* __restrict__ user0, void* __restrict__ internal0,
                                                const double* __restrict__ user1, void* __restrict__ internal1,
                                                const int32_t* __restrict__ perm, int64_t ne) {
    constexpr int H = NV / 2;
    const double* __restrict__ user = blockIdx.y == 0 ? user0 : user1;   // one or (gridDim.y = 2) two arrays
    void* __restrict__ internal = blockIdx.y == 0 ? internal0 : internal1;
    const int64_t e0 = blockIdx.x * (int64_t)ME;
    const int n = (ne - e0 < ME ? (int)(ne - e0) : ME) * H;
    __shared__ int32_t sp[ME];
    if (threadIdx.x * H < n && threadIdx.x < ME) sp[threadIdx.x] = perm[e0 + threadIdx.x];
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += MT2) {
        const int e = i / H, k = 2 * (i - e * H);
        const double2 x = load2<VEC>(user + (int64_t)sp[e] * NV + k);
        const int64_t o = (e0 + e) * NV + k;
        if (FMT == MOVE_F64) {
            *reinterpret_cast<double2*>(static_cast<double*>(internal) + o) = x;
        } else {
            float* p = static_cast<float*>(internal) + o;
            if (FMT == MOVE_FF) {
                float2 h, l;
                ff::split(x.x, h.x, l.x);
                ff::split(x.y, h.y, l.y);
                *reinterpret_cast<float2*>(p) = h;
                *reinterpret_cast<float2*>(p + ne * NV) = l;
            } else {
                *reinterpret_cast<float2*>(p) = make_float2(ff::narrow(x.x), ff::narrow(x.y));
            }
        }
    }
}

template <int NV, int FMT, bool VEC, int ME>
__global__ void __launch_bounds__(MT2) k_scatter(const void* __restrict__ internal, double* __restrict__ user,
                                                 const int32_t* __restrict__ perm, int64_t ne) {
    constexpr int H = NV / 2;
    const int64_t e0 = blockIdx.x * (int64_t)ME;
    const int n = (ne - e0 < ME ? (int)(ne - e0) : ME) * H;
    __shared__ int32_t sp[ME];
    if (threadIdx.x * H < n && threadIdx.x < ME) sp[threadIdx.x] = perm[e0 + threadIdx.x];
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += MT2) {
        const int e = i / H, k = 2 * (i - e * H);
        const int64_t o = (e0 + e) * NV + k;
        double2 x;
        if (FMT == MOVE_F64) {
            x = *reinterpret_cast<const double2*>(static_cast<const double*>(internal) + o);
        } else {
            const float* p = static_cast<const float*>(internal) + o;
            const float2 h = *reinterpret_cast<const float2*>(p);
            if (FMT == MOVE_FF) {
                const float2 l = *reinterpret_cast<const float2*>(p + ne * NV);
                x = make_double2(ff::join(h.x, l.x), ff::join(h.y, l.y));
            } else {
                x = make_double2(ff::widen(h.x), ff::widen(h.y));
            }
        }
        store2<VEC>(user + (int64_t)sp[e] * NV + k, x);
    }
}

// user -> internal (gather; user1, internal1: a second pair, or null) or internal -> user
struct Move {
    bool gather;
    const void *from, *from1;
    void *to, *to1;
};

template <int NV, int FMT, int ME>
void move_elements(const Move& v, const int32_t* perm, int64_t ne, cudaStream_t s) {
    const unsigned grid = (unsigned)((ne + ME - 1) / ME);
    auto at16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    if (v.gather) {
        const double *u = static_cast<const double*>(v.from), *u1 = static_cast<const double*>(v.from1);
        const dim3 g(grid, u1 ? 2 : 1);
        if (at16(u) && at16(u1)) k_gather<NV, FMT, true, ME><<<g, MT2, 0, s>>>(u, v.to, u1, v.to1, perm, ne);
        else k_gather<NV, FMT, false, ME><<<g, MT2, 0, s>>>(u, v.to, u1, v.to1, perm, ne);
    } else {
        double* u = static_cast<double*>(v.to);
        if (at16(u)) k_scatter<NV, FMT, true, ME><<<grid, MT2, 0, s>>>(v.from, u, perm, ne);
        else k_scatter<NV, FMT, false, ME><<<grid, MT2, 0, s>>>(v.from, u, perm, ne);
    }
}

template <int NV, int FMT>
void move_elements(const Move& v, const int32_t* perm, int64_t ne, cudaStream_t s) {
    if (small_tiles(ne)) move_elements<NV, FMT, 8>(v, perm, ne, s);
    else move_elements<NV, FMT, 32>(v, perm, ne, s);
}

cudaError_t move_state(const dg_mesh* m, int fmt, const Move& v, cudaStream_t s) {
    const int64_t ne = m->host.ne;
    auto go = [&](auto nv) {
        constexpr int NV = decltype(nv)::value;
        if (fmt == MOVE_F64) move_elements<NV, MOVE_F64>(v, m->d_perm, ne, s);
        else if (fmt == MOVE_F32) move_elements<NV, MOVE_F32>(v, m->d_perm, ne, s);
        else move_elements<NV, MOVE_FF>(v, m->d_perm, ne, s);
    };
    if (m->p == 1) go(std::integral_constant<int, 20>());
    else if (m->p == 2) go(std::integral_constant<int, 50>());
    else go(std::integral_constant<int, 100>());
    return cudaGetLastError();
}

int format_of(const dg_mesh* m) {
    return m->precision == DG_FP64 ? MOVE_F64 : m->precision == DG_FP32 ? MOVE_F32 : MOVE_FF;
}

// h_e = 1 / max_f |grad lambda_f| = 3 vol / max face area (the root of the largest square is the
// largest root)
__device__ __forceinline__ double inv_h(const double* I) {
    double m = 0.0;
    for (int f = 0; f < 4; ++f) {
        double g0, g1, g2;
        if (f == 0) {
            g0 = -(I[0] + I[3] + I[6]);
            g1 = -(I[1] + I[4] + I[7]);
            g2 = -(I[2] + I[5] + I[8]);
        } else {
            g0 = I[3 * (f - 1)];
            g1 = I[3 * (f - 1) + 1];
            g2 = I[3 * (f - 1) + 2];
        }
        m = fmax(m, g0 * g0 + g1 * g1 + g2 * g2);
    }
    return sqrt(m);
}

__device__ __forceinline__ double det3(const double* I) {
    return I[0] * (I[4] * I[8] - I[5] * I[7]) - I[1] * (I[3] * I[8] - I[5] * I[6]) + I[2] * (I[3] * I[7] - I[4] * I[6]);
}

__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(float x) { return ff::widen(x); }

template <typename Real>
__global__ void __launch_bounds__(RT) k_dt_local(const Real* __restrict__ U, const Real* __restrict__ Ulo,
                                                 const double* __restrict__ jinv, int64_t ne,
                                                 int nb, int p, double gamma, double* __restrict__ block_min,
                                                 unsigned int* status) {
    __shared__ double red[RT];
    double best = 0.0;   // the largest reciprocal step: one division per thread, min(1 / x) = 1 / max(x)
    for (int64_t e = blockIdx.x * (int64_t)RT + threadIdx.x; e < ne; e += (int64_t)gridDim.x * RT) {
        double m[5];
        for (int v = 0; v < 5; ++v)   // element means
            m[v] = SQRT6 * (to_double(U[(e * 5 + v) * nb]) + (Ulo ? to_double(Ulo[(e * 5 + v) * nb]) : 0.0));
        const double rho = m[0];
        const double u2 = (m[1] * m[1] + m[2] * m[2] + m[3] * m[3]) / (rho * rho);
        const double pr = (gamma - 1.0) * (m[4] - 0.5 * rho * u2);
        if (!(rho > 0.0) || !(pr > 0.0)) atomicOr(status, 1u);
        const double c = sqrt(gamma * pr / rho);
        best = fmax(best, inv_h(jinv + 9 * e) * (2 * p + 1) * (sqrt(u2) + c));
    }
    red[threadIdx.x] = 1.0 / best;
    __syncthreads();
    for (int s = RT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) block_min[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(RT) k_min_final(const double* __restrict__ in, int n, double* __restrict__ out) {
    __shared__ double red[RT];
    double best = INFINITY;
    for (int i = threadIdx.x; i < n; i += RT) best = fmin(best, in[i]);
    red[threadIdx.x] = best;
    __syncthreads();
    for (int s = RT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

// Per element: |det J| * (int_T U_v = c_v0 / sqrt6) and |det J| * sum_q w_q |m|^2/(2 rho); block sums in
// a fixed order, a thread per element as far as the sums go.  The point values are a thread per
// (element, point) from shared memory (coefficients converted to FP64 once): bound by the FP64 pipe.  A
// thread per element reading tables and coefficients per point took 2.86 ms on 165,888 P3 elements in
// the mixed form, waiting on memory.  FP64 and FP32 meshes keep every operation of that form and its
// order (adjoint checks difference the kinetic energy at 1e-7 of the state, which its last bit
// decides); the mixed forms (FACTORED), which have no adjoint, interpolate a thread per (element,
// density or momentum) row with the factored operator: 896 -> 600 us.
template <typename Real, int P, bool FACTORED>
struct IntPlan {
    static constexpr int NB = nb_of(P), NQ = nq_of(P), SUB = FACTORED ? 64 : 32, NR = 4 * NB;
    // shared memory (doubles): coefficients of SUB elements (density and momenta) and the basis at the
    // points [NB][NQ], or (FACTORED) the point values [NQ][RT]; per element and point the kinetic
    // energy's term
    static constexpr int PH = SUB * NR, TERM = FACTORED ? NQ * RT : PH + NB * NQ, REALS = TERM + RT * (NQ + 1);
    static constexpr size_t BYTES = REALS * sizeof(double);
};

template <typename Real, int P, bool FACTORED>
__global__ void __launch_bounds__(RT) k_integrals_local(const Real* __restrict__ U, const Real* __restrict__ Ulo,
                                                        const double* __restrict__ jinv,
                                                        const double* __restrict__ tab, int64_t ne,
                                                        double* __restrict__ block_sum) {
    using S = IntPlan<Real, P, FACTORED>;
    constexpr int NB = S::NB, NQ = S::NQ, SUB = S::SUB, NR = S::NR;
    constexpr TabLayout L(P);
    extern __shared__ double sm[];
    double *sC = sm, *sP = sm + S::PH, *sT = sm + S::TERM;
    __shared__ double red[6][RT];
    const int t = threadIdx.x;
    if (!FACTORED)
        for (int i = t; i < NB * NQ; i += RT) sP[i] = tab[L.phiq + i];
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t base = blockIdx.x * (int64_t)RT; base < ne; base += (int64_t)gridDim.x * RT) {
        for (int sub = 0; sub < RT; sub += SUB) {
            const int64_t e0 = base + sub;
            const int nel = ne - e0 < SUB ? (int)(ne - e0) : SUB;
            if (nel <= 0) break;
            __syncthreads();
            if constexpr (FACTORED) {
                if (t < 4 * nel) {
                    const int64_t row = (e0 + (t >> 2)) * 5 + (t & 3);
                    Real x[NB], y[NB];
                    double c[NB];
                    load_row<NB>(U + row * NB, x);
                    load_row<NB>(Ulo + row * NB, y);
#pragma unroll
                    for (int j = 0; j < NB; ++j) c[j] = ff::join(x[j], y[j]);
                    modal::interpolate<double, P, NB, 0, NQ>(c, [&](int q, double u) { sC[q * RT + t] = u; });
                }
            } else {
                for (int i = t; i < nel * NR; i += RT) {
                    const int e = i / NR, k = i - e * NR;
                    const int64_t at = (e0 + e) * 5 * NB + k;
                    sC[i] = to_double(U[at]) + (Ulo ? to_double(Ulo[at]) : 0.0);
                }
            }
            __syncthreads();
            for (int i = t; i < nel * NQ; i += RT) {
                const int e = FACTORED ? i % nel : i / NQ, q = FACTORED ? i / nel : i - e * NQ;
                double Uq[4];
                if constexpr (FACTORED) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) Uq[v] = sC[q * RT + 4 * e + v];
                } else {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        double s = 0.0;
#pragma unroll
                        for (int j = 0; j < NB; ++j) s += sC[e * NR + v * NB + j] * sP[j * NQ + q];
                        Uq[v] = s;
                    }
                }
                sT[(sub + e) * (NQ + 1) + q] =
                    tab[L.wq + q] * 0.5 * (Uq[1] * Uq[1] + Uq[2] * Uq[2] + Uq[3] * Uq[3]) / Uq[0];
            }
        }
        __syncthreads();
        const int64_t e = base + t;
        if (e < ne) {
            const double detJ = 1.0 / fabs(det3(jinv + 9 * e));
            const Real* c = U + e * 5 * NB;
            const Real* cl = Ulo ? Ulo + e * 5 * NB : nullptr;
            for (int v = 0; v < 5; ++v) acc[v] += detJ * (to_double(c[v * NB]) + (cl ? to_double(cl[v * NB]) : 0.0)) / SQRT6;
            double ke = 0.0;
            for (int q = 0; q < NQ; ++q) ke += sT[t * (NQ + 1) + q];
            acc[5] += detJ * ke;
        }
    }
    for (int k = 0; k < 6; ++k) red[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = RT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int k = 0; k < 6; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 6) block_sum[blockIdx.x * 6 + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void __launch_bounds__(RT) k_sum_final(const double* __restrict__ in, int n, double* __restrict__ out) {
    __shared__ double red[6][RT];
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int i = threadIdx.x; i < n; i += RT)
        for (int k = 0; k < 6; ++k) acc[k] += in[i * 6 + k];
    for (int k = 0; k < 6; ++k) red[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = RT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int k = 0; k < 6; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 6) out[threadIdx.x] = red[threadIdx.x][0];
}

// U[e][v][j] = sum_q w_q f[e][q][v] phi_j(q)  (orthonormal basis; caller order)
__global__ void k_project(const double* __restrict__ f, double* __restrict__ U, const double* __restrict__ tab,
                          int64_t ne, int nb, int nq, int off_phiq, int off_wq) {
    const int64_t n = ne * 5 * nb;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / (5 * nb);
        const int r = (int)(i - e * 5 * nb), v = r / nb, j = r - v * nb;
        double s = 0.0;
        for (int q = 0; q < nq; ++q) s += tab[off_wq + q] * f[(e * nq + q) * 5 + v] * tab[off_phiq + j * nq + q];
        U[i] = s;
    }
}

__global__ void k_volume_points(const double* __restrict__ x0J, const double* __restrict__ xi, double* __restrict__ xyz,
                                int64_t ne, int nq) {
    const int64_t n = ne * nq;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / nq;
        const int q = (int)(i - e * nq);
        const double* g = x0J + 12 * e;
        for (int d = 0; d < 3; ++d)
            xyz[3 * i + d] = g[d] + g[3 + 3 * d] * xi[3 * q] + g[3 + 3 * d + 1] * xi[3 * q + 1] + g[3 + 3 * d + 2] * xi[3 * q + 2];
    }
}

// d/dU of int |m|^2/(2 rho) dx by the volume rule (caller order): out_vj = |det J| sum_q w_q g_v(q)
// phi_j(q), g = (-|m|^2/(2 rho^2), m/rho, 0).  Tiles of 32 elements: thread per (element, density or
// momentum) row, per (element, point), and rows again with the transposed interpolation.  One thread
// per element, accumulating in memory, took 5.1 ms on 196,608 P2 elements.
template <int P>
__global__ void __launch_bounds__(128) k_ke_grad(const double* __restrict__ U, double* __restrict__ out,
                                                 const int32_t* __restrict__ perm, const double* __restrict__ jinv, int64_t ne) {
    constexpr int NB = nb_of(P), NQ = nq_of(P);
    __shared__ double sU[NQ][128];
    __shared__ double sD[32];
    __shared__ int32_t sp[32];
    const int t = threadIdx.x, el = t >> 2, v = t & 3;
    const int64_t e0 = blockIdx.x * (int64_t)32;
    const int nel = ne - e0 < 32 ? (int)(ne - e0) : 32;
    if (t < nel) {
        sD[t] = 1.0 / fabs(det3(jinv + 9 * (e0 + t)));
        sp[t] = perm[e0 + t];
    }
    __syncthreads();
    const bool live = el < nel;
    const int64_t row = live ? (int64_t)sp[el] * 5 + v : 0;
    if (live) {
        double c[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) c[j] = U[row * NB + j];   // the caller's pointer: 8-byte aligned
        modal::interpolate<double, P, NB, 0, NQ>(c, [&](int q, double u) { sU[q][t] = u; });
    }
    __syncthreads();
    for (int i = t; i < NQ * 32; i += 128) {
        const int e = i & 31, q = i >> 5;
        if (e >= nel) continue;
        double* u = &sU[q][4 * e];
        const double ri = 1.0 / u[0], d = sD[e];
        const double x = u[1] * ri, y = u[2] * ri, z = u[3] * ri;
        u[0] = -0.5 * d * (x * x + y * y + z * z);
        u[1] = d * x;
        u[2] = d * y;
        u[3] = d * z;
    }
    __syncthreads();
    if (!live) return;
    double r[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) r[j] = 0.0;
    modal::unroll<0, NQ>([&](auto qc) {
        constexpr int q = qc.value, m = modal::kT<P>.vmir[q];
        if constexpr (m >= q) modal::moments<double, P, NB>(q, sU[q][t], m != q ? sU[m][t] : 0.0, r);
    });
#pragma unroll
    for (int j = 0; j < NB; ++j) out[row * NB + j] = r[j];
    if (v == 3) {   // the energy row
#pragma unroll
        for (int j = 0; j < NB; ++j) out[(row + 1) * NB + j] = 0.0;
    }
}

int grid_for(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 32));
}

}  // namespace

cudaError_t launch_gather(dg_mesh* m, const double* user, void* internal, cudaStream_t s) {
    return move_state(m, format_of(m), {true, user, nullptr, internal, nullptr}, s);
}

cudaError_t launch_gather2(dg_mesh* m, const double* user, void* internal, const double* user1, void* internal1, cudaStream_t s) {
    return move_state(m, format_of(m), {true, user, user1, internal, internal1}, s);
}

cudaError_t launch_gather_f32(dg_mesh* m, const double* user, float* internal, cudaStream_t s) {
    return move_state(m, MOVE_F32, {true, user, nullptr, internal, nullptr}, s);
}

cudaError_t launch_scatter(dg_mesh* m, const void* internal, double* user, cudaStream_t s) {
    return move_state(m, format_of(m), {false, internal, nullptr, user, nullptr}, s);
}

cudaError_t launch_scatter_f32(dg_mesh* m, const float* internal, double* user, cudaStream_t s) {
    return move_state(m, MOVE_F32, {false, internal, nullptr, user, nullptr}, s);
}

int reduction_blocks(int64_t ne) { return (int)std::max<int64_t>(1, std::min<int64_t>((ne + RT - 1) / RT, 1024)); }

cudaError_t launch_stable_dt(dg_mesh* m, const void* U, double* d_out, cudaStream_t s) {
    const int nblk = reduction_blocks(m->host.ne);
    const int64_t n = m->host.ne * 5 * m->nb;
    if (m->precision == DG_FP64)
        k_dt_local<double><<<nblk, RT, 0, s>>>(static_cast<const double*>(U), nullptr, m->d_jinv64, m->host.ne, m->nb,
                                               m->p, m->gamma, m->d_red, m->d_status);
    else
        k_dt_local<float><<<nblk, RT, 0, s>>>(static_cast<const float*>(U),
                                              m->precision == DG_FP32 ? nullptr : static_cast<const float*>(U) + n,
                                              m->d_jinv64, m->host.ne, m->nb, m->p, m->gamma, m->d_red, m->d_status);
    k_min_final<<<1, RT, 0, s>>>(m->d_red, nblk, d_out);
    return cudaGetLastError();
}

template <typename Real, int P, bool FACTORED>
static cudaError_t integrals_local(dg_mesh* m, const Real* U, const Real* Ulo, int nblk, cudaStream_t s) {
    constexpr size_t bytes = IntPlan<Real, P, FACTORED>::BYTES;
    auto kern = k_integrals_local<Real, P, FACTORED>;
    static bool init = false;
    if (!init) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        init = true;
    }
    kern<<<nblk, RT, bytes, s>>>(U, Ulo, m->d_jinv64, m->d_tab64, m->host.ne, m->d_red);
    return cudaGetLastError();
}

cudaError_t launch_integrals(dg_mesh* m, const void* U, double* d_out6, cudaStream_t s) {
    const int nblk = reduction_blocks(m->host.ne);
    const int64_t n = m->host.ne * 5 * m->nb;
    auto go = [&](auto p) {
        constexpr int P = decltype(p)::value;
        if (m->precision == DG_FP64) return integrals_local<double, P, false>(m, static_cast<const double*>(U), nullptr, nblk, s);
        const float* u = static_cast<const float*>(U);
        if (m->precision == DG_FP32) return integrals_local<float, P, false>(m, u, nullptr, nblk, s);
        return integrals_local<float, P, true>(m, u, u + n, nblk, s);
    };
    const cudaError_t e = m->p == 1 ? go(std::integral_constant<int, 1>())
                          : m->p == 2 ? go(std::integral_constant<int, 2>())
                                      : go(std::integral_constant<int, 3>());
    if (e != cudaSuccess) return e;
    k_sum_final<<<1, RT, 0, s>>>(m->d_red, nblk, d_out6);
    return cudaGetLastError();
}

cudaError_t launch_project(dg_mesh* m, const double* f, double* U, cudaStream_t s) {
    const TabLayout L(m->p);
    const int64_t n = m->host.ne * 5 * m->nb;
    k_project<<<grid_for(n, 256), 256, 0, s>>>(f, U, m->d_tab64, m->host.ne, m->nb, m->nq, L.phiq, L.wq);
    return cudaGetLastError();
}

cudaError_t launch_ke_grad(dg_mesh* m, const double* U_user, double* out_user, cudaStream_t s) {
    const int64_t ne = m->host.ne;
    const unsigned grid = (unsigned)((ne + 31) / 32);
    if (m->p == 1) k_ke_grad<1><<<grid, 128, 0, s>>>(U_user, out_user, m->d_perm, m->d_jinv64, ne);
    else if (m->p == 2) k_ke_grad<2><<<grid, 128, 0, s>>>(U_user, out_user, m->d_perm, m->d_jinv64, ne);
    else k_ke_grad<3><<<grid, 128, 0, s>>>(U_user, out_user, m->d_perm, m->d_jinv64, ne);
    return cudaGetLastError();
}

cudaError_t launch_volume_points(dg_mesh* m, const double* d_x0J, double* xyz, cudaStream_t s) {
    const int64_t n = m->host.ne * m->nq;
    const double* d_xi = m->d_tab64 + TabLayout(m->p).total;   // reference coordinates stored after the tables
    k_volume_points<<<grid_for(n, 256), 256, 0, s>>>(d_x0J, d_xi, xyz, m->host.ne, m->nq);
    return cudaGetLastError();
}

}  // namespace dg
