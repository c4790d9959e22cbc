// The numerical flux of a face point in its owner's orientation, evaluated once per face (FP64 and
// FP32 CUDA-core paths).  The formulas are rusanov_flux / roe_flux of euler_device.cuh; the Roe form
// shares each state's reciprocal and square root: one reciprocal square root per density and one
// for the Roe-averaged sound speed, each corrected by one Newton step to the accuracy of a division
// and a square root, in the place of four divisions and three square roots (FP64: ~165 operations
// of the FP64 pipe per point against ~240).
#pragma once

#include "euler_device.cuh"

namespace dg {

__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(float x) {
    const float r = __fdividef(1.f, x);
    return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }
__device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }

// 1 / x and sqrt(x) of x > 0
template <typename Real>
__device__ __forceinline__ void inv_and_sqrt(Real x, Real& inv, Real& sq) {
    const Real rs = rsqrt_(x);
    inv = rs * rs;
    inv += inv * (Real(1) - x * inv);
    sq = x * rs;
    sq += Real(0.5) * rs * (x - sq * sq);
}

// x > 0 (false for NaN) on the integer pipe: the FP64 pipe is the kernels' bound
__device__ __forceinline__ bool positive(double x) {
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }

// okL, okR: positive density and pressure of the two states
template <typename Real>
__device__ __forceinline__ void roe_face(const Real* L, const Real* R, const Real* n, Real gamma, Real eps, Real* H,
                                         bool& okL, bool& okR) {
    const Real g1 = gamma - Real(1);
    Real rL, sL, rR, sR;
    inv_and_sqrt(L[0], rL, sL);
    inv_and_sqrt(R[0], rR, sR);
    const Real uL[3] = {L[1] * rL, L[2] * rL, L[3] * rL}, uR[3] = {R[1] * rR, R[2] * rR, R[3] * rR};
    const Real pL = g1 * (L[4] - Real(0.5) * (L[1] * uL[0] + L[2] * uL[1] + L[3] * uL[2]));
    const Real pR = g1 * (R[4] - Real(0.5) * (R[1] * uR[0] + R[2] * uR[1] + R[3] * uR[2]));
    okL = positive(L[0]) && positive(pL);
    okR = positive(R[0]) && positive(pR);
    const Real nL = uL[0] * n[0] + uL[1] * n[1] + uL[2] * n[2], nR = uR[0] * n[0] + uR[1] * n[1] + uR[2] * n[2];
    const Real eL = L[4] + pL, eR = R[4] + pR;
    // Roe averages
    const Real w = recip(sL + sR), wL = sL * w, wR = sR * w;
    const Real u[3] = {wL * uL[0] + wR * uR[0], wL * uL[1] + wR * uR[1], wL * uL[2] + wR * uR[2]};
    const Real h = wL * (eL * rL) + wR * (eR * rR);
    const Real q2 = Real(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    Real ic2, c;
    inv_and_sqrt(g1 * (h - q2), ic2, c);
    const Real rho = sL * sR, un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
    const Real du[3] = {uR[0] - uL[0], uR[1] - uL[1], uR[2] - uL[2]};
    const Real dun = du[0] * n[0] + du[1] * n[1] + du[2] * n[2];
    const Real dp = pR - pL, t = rho * c * dun, hic2 = Real(0.5) * ic2;
    Real l1 = fabs(un - c), l5 = fabs(un + c);
    const Real l2 = fabs(un);
    if (eps > Real(0)) {
        const Real d = eps * c;
        if (l1 < d) l1 = (l1 * l1 + d * d) / (Real(2) * d);
        if (l5 < d) l5 = (l5 * l5 + d * d) / (Real(2) * d);
    }
    const Real w1 = l1 * ((dp - t) * hic2), w2 = l2 * ((R[0] - L[0]) - dp * ic2), w5 = l5 * ((dp + t) * hic2);
    // dissipation: w0 u + a n + b du in momentum, w0 = w1 + w2 + w5
    const Real w15 = w1 + w5, w0 = w15 + w2, b = l2 * rho, cd = (w5 - w1) * c;
    const Real a = cd - b * dun;
    const Real p = pL + pR, fL = L[0] * nL, fR = R[0] * nR;
    H[0] = Real(0.5) * ((fL + fR) - w0);
#pragma unroll
    for (int d = 0; d < 3; ++d)
        H[1 + d] = Real(0.5) * ((fL * uL[d] + fR * uR[d] + p * n[d]) - (w0 * u[d] + a * n[d] + b * du[d]));
    const Real ud = u[0] * du[0] + u[1] * du[1] + u[2] * du[2];
    H[4] = Real(0.5) * ((eL * nL + eR * nR) - (w15 * h + w2 * q2 + cd * un + b * (ud - dun * un)));
}

template <typename Real>
__device__ __forceinline__ void rusanov_face(const Real* L, const Real* R, const Real* n, Real gamma, Real* H, bool& okL,
                                             bool& okR) {
    const Real g1 = gamma - Real(1);
    const Real rL = recip(L[0]), rR = recip(R[0]);
    const Real uL[3] = {L[1] * rL, L[2] * rL, L[3] * rL}, uR[3] = {R[1] * rR, R[2] * rR, R[3] * rR};
    const Real pL = g1 * (L[4] - Real(0.5) * (L[1] * uL[0] + L[2] * uL[1] + L[3] * uL[2]));
    const Real pR = g1 * (R[4] - Real(0.5) * (R[1] * uR[0] + R[2] * uR[1] + R[3] * uR[2]));
    okL = positive(L[0]) && positive(pL);
    okR = positive(R[0]) && positive(pR);
    const Real nL = uL[0] * n[0] + uL[1] * n[1] + uL[2] * n[2], nR = uR[0] * n[0] + uR[1] * n[1] + uR[2] * n[2];
    const Real aL = fabs(nL) + EulerOps<Real>::sqrt_(gamma * pL * rL), aR = fabs(nR) + EulerOps<Real>::sqrt_(gamma * pR * rR);
    const Real s = aL >= aR ? aL : aR, p = pL + pR, fL = L[0] * nL, fR = R[0] * nR;
    H[0] = Real(0.5) * ((fL + fR) - s * (R[0] - L[0]));
#pragma unroll
    for (int d = 0; d < 3; ++d)
        H[1 + d] = Real(0.5) * ((fL * uL[d] + fR * uR[d] + p * n[d]) - s * (R[1 + d] - L[1 + d]));
    H[4] = Real(0.5) * (((L[4] + pL) * nL + (R[4] + pR) * nR) - s * (R[4] - L[4]));
}

template <typename Real, int FLUX>
__device__ __forceinline__ void face_flux(const Real* L, const Real* R, const Real* n, Real gamma, Real eps, Real* H,
                                          bool& okL, bool& okR) {
    if (FLUX == DG_ROE) roe_face(L, R, n, gamma, eps, H, okL, okR);
    else rusanov_face(L, R, n, gamma, H, okL, okR);
}

}  // namespace dg
