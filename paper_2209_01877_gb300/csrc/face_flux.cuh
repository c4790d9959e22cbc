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

// ---- reverse mode ---------------------------------------------------------------------------------
// The transposed Jacobians of the face flux applied to a cotangent Hb of H: (Lb, Rb) = (dH/dL, dH/dR)^T
// Hb, one reverse sweep through the formulas above.  At a kink (|x| at x = 0, max at a tie) the
// derivative is that of the branch an evaluation with the interior side first would take: tie = +1
// for the residual of L's element, -1 for that of R's (whose flux sees the opposite normal).  Returns
// whether a kink was hit, in which case the two residuals' cotangents need a sweep each.
template <typename Real>
__device__ __forceinline__ Real sign_at(Real x, Real tie, bool& kink) {
    if (x == Real(0)) kink = true;
    return x < Real(0) ? Real(-1) : x > Real(0) ? Real(1) : tie;
}

// one side's part: the cotangent f of its normal flux, with those of its velocity, pressure,
// specific total enthalpy and density from elsewhere, onto its conserved state
template <typename Real>
__device__ __forceinline__ void side_reverse(const Real* U, const Real* u, Real ri, Real p, Real un, const Real* n, Real g1,
                                             const Real* f, const Real* ub, Real pb, Real hb, Real rb, Real unb, Real* out) {
    const Real e = U[4] + p, k = Real(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const Real fb = f[0] + f[1] * u[0] + f[2] * u[1] + f[3] * u[2];   // of the mass flux rho un
    const Real nb = unb + f[4] * e + fb * U[0];                       // of un
    const Real eb = f[4] * un + hb * ri;                              // of E + p
    const Real pt = pb + eb + f[1] * n[0] + f[2] * n[1] + f[3] * n[2];
    const Real m = U[0] * un;
    Real uu = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const Real x = ub[d] + m * f[1 + d] + nb * n[d];              // of u_d
        uu += x * u[d];
        out[1 + d] = x * ri - g1 * pt * u[d];
    }
    out[4] = eb + g1 * pt;
    out[0] = rb + fb * un - ri * (uu + hb * (e * ri)) + g1 * pt * k;
}

template <typename Real>
__device__ __forceinline__ bool roe_reverse(const Real* L, const Real* R, const Real* n, Real gamma, Real eps, const Real* Hb,
                                            Real tie, Real* Lb, Real* Rb) {
    const Real g1 = gamma - Real(1);
    Real rL, sL, rR, sR;
    inv_and_sqrt(L[0], rL, sL);
    inv_and_sqrt(R[0], rR, sR);
    const Real uL[3] = {L[1] * rL, L[2] * rL, L[3] * rL}, uR[3] = {R[1] * rR, R[2] * rR, R[3] * rR};
    const Real pL = g1 * (L[4] - Real(0.5) * (L[1] * uL[0] + L[2] * uL[1] + L[3] * uL[2]));
    const Real pR = g1 * (R[4] - Real(0.5) * (R[1] * uR[0] + R[2] * uR[1] + R[3] * uR[2]));
    const Real nL = uL[0] * n[0] + uL[1] * n[1] + uL[2] * n[2], nR = uR[0] * n[0] + uR[1] * n[1] + uR[2] * n[2];
    const Real hL = (L[4] + pL) * rL, hR = (R[4] + pR) * rR;
    const Real w = recip(sL + sR), wL = sL * w, wR = sR * w;
    const Real u[3] = {wL * uL[0] + wR * uR[0], wL * uL[1] + wR * uR[1], wL * uL[2] + wR * uR[2]};
    const Real h = wL * hL + wR * hR, q2 = Real(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    Real ic2, c;
    inv_and_sqrt(g1 * (h - q2), ic2, c);
    const Real rho = sL * sR, un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
    const Real du[3] = {uR[0] - uL[0], uR[1] - uL[1], uR[2] - uL[2]};
    const Real dun = du[0] * n[0] + du[1] * n[1] + du[2] * n[2];
    const Real dp = pR - pL, t = rho * c * dun, hic2 = Real(0.5) * ic2;
    bool kink = false;
    const Real s1 = sign_at(un - c, tie, kink), s2 = sign_at(un, tie, kink), s5 = sign_at(un + c, tie, kink);
    const Real r1 = fabs(un - c), l2 = fabs(un), r5 = fabs(un + c);
    Real l1 = r1, l5 = r5;
    const Real d = eps * c;
    const bool h1 = eps > Real(0) && r1 < d, h5 = eps > Real(0) && r5 < d;
    if (h1) l1 = (r1 * r1 + d * d) / (Real(2) * d);
    if (h5) l5 = (r5 * r5 + d * d) / (Real(2) * d);
    const Real a1 = (dp - t) * hic2, a2 = (R[0] - L[0]) - dp * ic2, a5 = (dp + t) * hic2;
    const Real w1 = l1 * a1, w2 = l2 * a2, w5 = l5 * a5;
    const Real w15 = w1 + w5, w0 = w15 + w2, b = l2 * rho, cd = (w5 - w1) * c;
    const Real ud = u[0] * du[0] + u[1] * du[1] + u[2] * du[2];

    const Real f[5] = {Real(0.5) * Hb[0], Real(0.5) * Hb[1], Real(0.5) * Hb[2], Real(0.5) * Hb[3], Real(0.5) * Hb[4]};
    const Real d0 = -f[0], d4 = -f[4], dm[3] = {-f[1], -f[2], -f[3]};
    // dissipation: mass w0; momentum w0 u + (cd - b dun) n + b du; energy w15 h + w2 q2 + cd un + b (u.du - dun un)
    const Real w0b = d0 + dm[0] * u[0] + dm[1] * u[1] + dm[2] * u[2];
    const Real ab = dm[0] * n[0] + dm[1] * n[1] + dm[2] * n[2];
    const Real bb = dm[0] * du[0] + dm[1] * du[1] + dm[2] * du[2] + d4 * (ud - dun * un) - ab * dun;
    const Real cdb = ab + d4 * un, d4b = d4 * b;
    Real dunb = -b * (ab + d4 * un), unb = d4 * (cd - b * dun);
    Real hb = d4 * w15, q2b = d4 * w2;
    const Real w15b = w0b + d4 * h, w2b = w0b + d4 * q2;
    const Real w1b = w15b - cdb * c, w5b = w15b + cdb * c;
    Real cb = cdb * (w5 - w1), rhob = bb * l2;
    const Real l2b = bb * rho + w2b * a2;
    Real l1b = w1b * a1, l5b = w5b * a5;
    const Real a1b = w1b * l1, a2b = w2b * l2, a5b = w5b * l5;
    if (h1) {
        const Real x = r1 / d;
        cb += l1b * eps * Real(0.5) * (Real(1) - x * x);
        l1b *= x;
    }
    if (h5) {
        const Real x = r5 / d;
        cb += l5b * eps * Real(0.5) * (Real(1) - x * x);
        l5b *= x;
    }
    unb += s1 * l1b + s5 * l5b + s2 * l2b;
    cb += s5 * l5b - s1 * l1b;
    const Real dpb = (a1b + a5b) * hic2 - a2b * ic2, tb = (a5b - a1b) * hic2;
    const Real ic2b = Real(0.5) * (a1b * (dp - t) + a5b * (dp + t)) - a2b * dp;
    rhob += tb * c * dun;
    cb += tb * rho * dun;
    dunb += tb * rho * c;
    const Real c2b = Real(0.5) * cb * c * ic2 - ic2b * ic2 * ic2;   // 1 / c = c ic2
    hb += g1 * c2b;
    q2b -= g1 * c2b;
    Real ubL[3], ubR[3], wLb = hb * hL, wRb = hb * hR;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const Real x = w0 * dm[k] + d4b * du[k] + q2b * u[k] + unb * n[k];   // of u_k
        const Real y = b * dm[k] + d4b * u[k];                                // of du_k (dun's part below)
        ubL[k] = wL * x - y;
        ubR[k] = wR * x + y;
        wLb += x * uL[k];
        wRb += x * uR[k];
    }
    const Real wd = w * (wLb - wRb);
    const Real sLb = wR * wd + rhob * sR, sRb = rhob * sL - wL * wd;
    side_reverse(L, uL, rL, pL, nL, n, g1, f, ubL, -dpb, wL * hb, Real(0.5) * sLb * sL * rL - a2b, -dunb, Lb);
    side_reverse(R, uR, rR, pR, nR, n, g1, f, ubR, dpb, wR * hb, Real(0.5) * sRb * sR * rR + a2b, dunb, Rb);
    return kink;
}

template <typename Real>
__device__ __forceinline__ bool rusanov_reverse(const Real* L, const Real* R, const Real* n, Real gamma, const Real* Hb, Real tie,
                                                Real* Lb, Real* Rb) {
    const Real g1 = gamma - Real(1);
    const Real rL = recip(L[0]), rR = recip(R[0]);
    const Real uL[3] = {L[1] * rL, L[2] * rL, L[3] * rL}, uR[3] = {R[1] * rR, R[2] * rR, R[3] * rR};
    const Real pL = g1 * (L[4] - Real(0.5) * (L[1] * uL[0] + L[2] * uL[1] + L[3] * uL[2]));
    const Real pR = g1 * (R[4] - Real(0.5) * (R[1] * uR[0] + R[2] * uR[1] + R[3] * uR[2]));
    const Real nL = uL[0] * n[0] + uL[1] * n[1] + uL[2] * n[2], nR = uR[0] * n[0] + uR[1] * n[1] + uR[2] * n[2];
    Real icL, cL, icR, cR;   // 1 / c^2 and c
    inv_and_sqrt(gamma * pL * rL, icL, cL);
    inv_and_sqrt(gamma * pR * rR, icR, cR);
    const Real aL = fabs(nL) + cL, aR = fabs(nR) + cR;
    Real diff = aL - aR;
    if constexpr (sizeof(Real) == 4) {
        // two wave speeds that only round to the same FP32 number (common where the flow is nearly
        // uniform) are no tie: |nL| - |nR| + (cL^2 - cR^2) / (cL + cR), the products' difference exact
        if (diff == 0.f) {
            const float x = pR * L[0], dx = fmaf(pL, R[0], -x), ex = fmaf(-pR, L[0], x);
            diff = (fabs(nL) - fabs(nR)) + gamma * (dx + ex) * rL * rR / (cL + cR);
        }
    }
    bool kink = diff == Real(0);
    const bool left = diff > Real(0) || (kink && tie > Real(0));
    const Real s = left ? aL : aR;
    Real f[5], sb = 0;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        f[v] = Real(0.5) * Hb[v];
        sb -= f[v] * (R[v] - L[v]);
    }
    // s = |un| + c of the faster side, c^2 = gamma p / rho
    const Real nb = sb * sign_at(left ? nL : nR, tie, kink);
    const Real cb = Real(0.5) * sb * (left ? cL * icL : cR * icR);   // of c^2
    const Real pb = cb * gamma * (left ? rL : rR), rb = -pb * (left ? pL * rL : pR * rR);
    const Real z[3] = {0, 0, 0};
    side_reverse(L, uL, rL, pL, nL, n, g1, f, z, left ? pb : Real(0), Real(0), left ? rb : Real(0), left ? nb : Real(0), Lb);
    side_reverse(R, uR, rR, pR, nR, n, g1, f, z, left ? Real(0) : pb, Real(0), left ? Real(0) : rb, left ? Real(0) : nb, Rb);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        Lb[v] += s * f[v];
        Rb[v] -= s * f[v];
    }
    return kink;
}

template <typename Real, int FLUX>
__device__ __forceinline__ bool face_reverse(const Real* L, const Real* R, const Real* n, Real gamma, Real eps, const Real* Hb,
                                             Real tie, Real* Lb, Real* Rb) {
    if (FLUX == DG_ROE) return roe_reverse(L, R, n, gamma, eps, Hb, tie, Lb, Rb);
    return rusanov_reverse(L, R, n, gamma, Hb, tie, Lb, Rb);
}

}  // namespace dg
