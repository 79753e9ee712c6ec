// lbm_bgk_collide.cuh -- the per-node collision of the D3Q19 BGK-Smagorinsky
// fluid with the D3Q7 scalar and the Boussinesq force, shared by the AA step
// kernels, the out-of-place recompute and the adjoint.
//
// Per node and step (lattice units, c_s^2 = 1/3, populations held as
// deviations f - w from the rest weights so FP32 keeps its digits):
//   chi = sum_k Phi_k                                        (Eq. 27)
//   F = g' chi e^g                                           (Eq. 11)
//   rho = 1 + sum_i (f_i - w_i), rho u = sum_i c_i f_i + F/2  (Eq. 19-20, 52-53)
//   Pi = sum_i c_i c_i (f_i - feq_i) = M - (delta rho / 3) I - rho u u
//   q = |Pi|, tau = (tau0 + sqrt(tau0^2 + 18 sqrt2 C_s^2 q / rho)) / 2
//                                                   (Eq. 32-34, reading R3)
//   f*_i = f_i - (f_i - feq_i)/tau + (1 - 1/2tau) w_i [3 (c_i - u) + 9 (c_i.u) c_i].F
//                                                   (Eq. 17, 21, 22, 26)
//   tau_Phi = 1/2 + 4 (D + nu_T / Sc_T), nu_T = (tau - tau0) / 3   (Eq. 30, 35)
//   Phi*_k = Phi_k - (Phi_k - w_k chi (1 + 4 c_k.u)) / tau_Phi     (Eq. 28-29)
#pragma once

#include "lbm_lanes.cuh"

namespace lbmgpu {

// Replaces f (held as f - w) and Phi (held as Phi - w) by their
// post-collision values.  Directions come in opposite pairs (i, i + 1 for odd
// i): with s = f_i + f_opp and d = f_i - f_opp the moments need half the
// additions, and the equilibrium and the Guo source split into a part even
// in c (shared by the pair) and a part odd in c (sign-flipped).
//
// L: One or Two (lbm_lanes.cuh), the nodes collided at once.  g: the force
// g' e^g per unit chi, with the sign of the velocity set that f and p are
// named in: every operation is odd or even under c -> -c, so a caller that
// names each population by its opposite passes -g and gets the same bits.
//
// SL: scalar lattice, D3Q7 (c_s^2 = 1/4) or D3Q6 (Eq. 29-31 as printed,
// c_s^2 = 1/3, w = 1/6, no rest population).
template <typename L, int SL>
__device__ __forceinline__ void collide_bgk_lanes(const KParams& kp, float gx, float gy, float gz,
                                                  typename L::V (&f)[19],
                                                  typename L::V (&p)[ScalarLat<SL>::NS]) {
    static_assert(SL == 7 || SL == 6, "BGK runs with the D3Q7 or D3Q6 scalar");
    using V = typename L::V;
    constexpr int K0 = SL == 7 ? 1 : 0;   // first moving scalar population
    // chi - 1, by opposite pairs
    const V q1 = L::add(p[K0], p[K0 + 1]), q2 = L::add(p[K0 + 2], p[K0 + 3]),
            q3 = L::add(p[K0 + 4], p[K0 + 5]);
    V chs = L::add(L::add(q1, q2), q3);
    if constexpr (SL == 7) chs = L::add(chs, p[0]);
    const V chi = L::add(chs, L::set(1.0f));
    const V Fx = L::mul(L::set(gx), chi), Fy = L::mul(L::set(gy), chi), Fz = L::mul(L::set(gz), chi);

    // moments: drho = sum f, j = sum c f, m_ab = sum c_a c_b f
    V sm[9], dm[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) {
        sm[m] = L::add(f[2 * m + 1], f[2 * m + 2]);
        dm[m] = L::sub(f[2 * m + 1], f[2 * m + 2]);
    }
    const V axy = L::add(sm[3], sm[4]), axz = L::add(sm[5], sm[6]), ayz = L::add(sm[7], sm[8]);
    const V drho = L::add(f[0], L::add(L::add(L::add(sm[0], sm[1]), sm[2]), L::add(L::add(axy, axz), ayz)));
    const V jx = L::add(dm[0], L::add(L::add(dm[3], dm[4]), L::add(dm[5], dm[6])));
    const V jy = L::add(dm[1], L::add(L::sub(dm[3], dm[4]), L::add(dm[7], dm[8])));
    const V jz = L::add(dm[2], L::add(L::sub(dm[5], dm[6]), L::sub(dm[7], dm[8])));
    const V mxx = L::add(sm[0], L::add(axy, axz)), myy = L::add(sm[1], L::add(axy, ayz)),
            mzz = L::add(sm[2], L::add(axz, ayz));
    const V mxy = L::sub(sm[3], sm[4]), mxz = L::sub(sm[5], sm[6]), myz = L::sub(sm[7], sm[8]);
    const V half = L::set(0.5f);
    const V rho = L::add(drho, L::set(1.0f));
    const V irho = lane_rcp<L>(rho);
    // momentum with the half-force shift and velocity
    const V hx = L::fma(half, Fx, jx), hy = L::fma(half, Fy, jy), hz = L::fma(half, Fz, jz);
    const V ux = L::mul(hx, irho), uy = L::mul(hy, irho), uz = L::mul(hz, irho);
    // rho u.u
    const V rusq = L::fma(hx, ux, L::fma(hy, uy, L::mul(hz, uz)));
    // non-equilibrium second moment (sum c c feq = rho (I/3 + u u), sum c c w = I/3)
    const V nx = L::neg(hx), ny = L::neg(hy), nz = L::neg(hz);
    const V n3 = L::set(-1.0f / 3.0f);
    const V pxx = L::fma(nx, ux, L::fma(n3, drho, mxx));
    const V pyy = L::fma(ny, uy, L::fma(n3, drho, myy));
    const V pzz = L::fma(nz, uz, L::fma(n3, drho, mzz));
    const V pxy = L::fma(nx, uy, mxy), pxz = L::fma(nx, uz, mxz), pyz = L::fma(ny, uz, myz);
    const V qd = L::fma(pxx, pxx, L::fma(pyy, pyy, L::mul(pzz, pzz)));
    const V qo = L::fma(pxy, pxy, L::fma(pxz, pxz, L::mul(pyz, pyz)));
    const V q = lane_sqrt<L>(L::fma(L::set(2.0f), qo, qd));
    // tau = (tau0 + s) / 2, s = sqrt(tau0^2 + X); 1 / tau = 2 r and tau - tau0
    // = X r / 2 (no cancellation) with r = 1 / (s + tau0)
    const V Aq = L::mul(L::set(kp.A), q);
    const V r = lane_rcp<L>(
        L::add(lane_sqrt<L>(L::fma(Aq, irho, L::set(__fmul_rn(kp.tau0, kp.tau0)))), L::set(kp.tau0)));
    // feq_i - w_i = w_i (drho + rho (3 cu + 4.5 cu^2 - 1.5 u.u)),
    // S_i = (1 - om/2) w_i (3 cF - 3 u.F + 9 cu cF): with, at the weight of the
    // axis directions (w = 1/18, the diagonals carry half of it),
    //   V = w (3 om rho u + 3 (1 - om/2) F),  W = w (4.5 om rho u + 9 (1 - om/2) F),
    //   A = om (drho - 1.5 rho u.u) - 3 (1 - om/2) u.F
    // w_i (om (feq_i - w_i) / w_i + ...) = w_i A + cu (c.W) + c.V, parts even and
    // odd in c.  o = om / 6 is rounded once, and 1 - om and the weights of A are
    // taken from what it rounded to (1 - 6 o; A - 12 w A at rest), so that the
    // update keeps mass and momentum to the rounding of its results.
    const V o = L::mul(L::add(r, r), L::set(1.0f / 6.0f));
    const V keep = L::fma(L::set(-6.0f), o, L::set(1.0f));
    const V g3 = L::fma(L::set(-3.0f), r, L::set(3.0f));          // 3 (1 - om/2)
    const V gw = L::mul(g3, L::set(w19(1)));
    const V uF = L::fma(ux, Fx, L::fma(uy, Fy, L::mul(uz, Fz)));
    const V A = L::fma(L::neg(g3), uF,
                       L::mul(L::mul(L::set(6.0f), o), L::fma(L::set(-1.5f), rusq, drho)));
    const V A1 = L::mul(L::set(w19(1)), A);
    const V ox = L::mul(o, hx), oy = L::mul(o, hy), oz = L::mul(o, hz);
    const V Vx = L::fma(gw, Fx, ox), Vy = L::fma(gw, Fy, oy), Vz = L::fma(gw, Fz, oz);
    const V g9 = L::mul(L::set(3.0f), gw), c15 = L::set(1.5f);
    const V Wx = L::fma(g9, Fx, L::mul(c15, ox)), Wy = L::fma(g9, Fy, L::mul(c15, oy)),
            Wz = L::fma(g9, Fz, L::mul(c15, oz));
    f[0] = L::fma(keep, f[0], L::fma(L::set(-12.0f), A1, A));
    auto pair = [&](int i, V even, V odd) {
        f[i] = L::fma(keep, f[i], L::add(even, odd));
        f[i + 1] = L::fma(keep, f[i + 1], L::sub(even, odd));
    };
    pair(1, L::fma(ux, Wx, A1), Vx);
    pair(3, L::fma(uy, Wy, A1), Vy);
    pair(5, L::fma(uz, Wz, A1), Vz);
    const V A2 = L::mul(half, A1);
    const V vx = L::mul(half, Vx), vy = L::mul(half, Vy), vz = L::mul(half, Vz);
    const V wx = L::mul(half, Wx), wy = L::mul(half, Wy), wz = L::mul(half, Wz);
    pair(7, L::fma(L::add(ux, uy), L::add(wx, wy), A2), L::add(vx, vy));
    pair(9, L::fma(L::sub(ux, uy), L::sub(wx, wy), A2), L::sub(vx, vy));
    pair(11, L::fma(L::add(ux, uz), L::add(wx, wz), A2), L::add(vx, vz));
    pair(13, L::fma(L::sub(ux, uz), L::sub(wx, wz), A2), L::sub(vx, vz));
    pair(15, L::fma(L::add(uy, uz), L::add(wy, wz), A2), L::add(vy, vz));
    pair(17, L::fma(L::sub(uy, uz), L::sub(wy, wz), A2), L::sub(vy, vz));

    // scalar: Phi_eq - w = w (chi - 1) + w chi c.u / c_s^2.  Only the
    // non-equilibrium parts are relaxed, and their sum is closed to zero
    // (through the rest population on D3Q7, by removing the mean on D3Q6), so
    // the update conserves sum Phi up to the rounding of the stored results
    // (relaxing towards the rounded chi would inject omega times the rounding
    // error of the sum at every node)
    const V dtau = L::mul(L::mul(half, L::mul(Aq, irho)), r);
    const V omp = lane_rcp<L>(L::fma(L::set(kp.kT), dtau, L::set(kp.taup0)));
    const V nomp = L::neg(omp);
    constexpr float wk = SL == 7 ? 0.125f : 1.0f / 6.0f;
    const V pe = L::mul(L::set(wk), chs);
    const V pa = L::mul(half, chi);   // w / c_s^2 = 1/2 on both lattices
    const V npa = L::neg(pa);
    V nq[6];
    nq[0] = L::sub(p[K0], L::fma(pa, ux, pe));
    nq[1] = L::sub(p[K0 + 1], L::fma(npa, ux, pe));
    nq[2] = L::sub(p[K0 + 2], L::fma(pa, uy, pe));
    nq[3] = L::sub(p[K0 + 3], L::fma(npa, uy, pe));
    nq[4] = L::sub(p[K0 + 4], L::fma(pa, uz, pe));
    nq[5] = L::sub(p[K0 + 5], L::fma(npa, uz, pe));
    const V sum = L::add(L::add(L::add(nq[0], nq[1]), L::add(nq[2], nq[3])), L::add(nq[4], nq[5]));
    if constexpr (SL == 7) {
        p[0] = L::fma(omp, sum, p[0]);
#pragma unroll
        for (int k = 0; k < 6; ++k) p[1 + k] = L::fma(nomp, nq[k], p[1 + k]);
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k)
            p[k] = L::fma(nomp, L::fma(L::set(-1.0f / 6.0f), sum, nq[k]), p[k]);
    }
}

// The same on one node in the 16-bit storage forms (SCALED) or in plain FP32
// units, with contraction left to the compiler.  The 16-bit kernels keep this
// form: their results, the FP32 rest row above all, follow every rounding of
// the collision through the storage roundings, and a form that rounds
// differently gives other (equally accurate) 16-bit runs.  Directions come in opposite pairs (i, i + 1 for odd
// i): with s = f_i + f_opp and d = f_i - f_opp the moments need half the
// additions, and the equilibrium and the Guo source split into a part even
// in c (shared by the pair) and a part odd in c (sign-flipped), which halves
// the per-direction arithmetic.
//
// SCALED: f and p hold the 16-bit storage units scale_f (f - w) and
// scale_phi (Phi - w); the scales are applied to the few moments and output
// terms instead of to every population, and the divisions and square roots
// use the hardware approximations (crcp, cdiv, csqrt).
//
// SL: scalar lattice, D3Q7 (c_s^2 = 1/4) or D3Q6 (Eq. 29-31 as printed,
// c_s^2 = 1/3, w = 1/6, no rest population).
template <bool SCALED = false, int SL = 7>
__device__ __forceinline__ void collide_bgk(const KParams& kp, float (&f)[19],
                                            float (&p)[ScalarLat<SL>::NS]) {
    static_assert(SL == 7 || SL == 6, "BGK runs with the D3Q7 or D3Q6 scalar");
    constexpr int NS = ScalarLat<SL>::NS;
    const float isf = SCALED ? kp.isf : 1.0f, isp = SCALED ? kp.isp : 1.0f;
    const float sf = SCALED ? kp.sf : 1.0f, sp = SCALED ? kp.sp : 1.0f;
    float chs = 0.0f;  // scale_phi (chi - 1)
#pragma unroll
    for (int k = 0; k < NS; ++k) chs += p[k];
    const float chit = chs * isp;  // chi - chi_s
    const float chi = kp.chi_s + chit;
    const float Fx = kp.gx * chi, Fy = kp.gy * chi, Fz = kp.gz * chi;

    float drho = f[0], jx = 0.0f, jy = 0.0f, jz = 0.0f;
    float mxx = 0.0f, myy = 0.0f, mzz = 0.0f, mxy = 0.0f, mxz = 0.0f, myz = 0.0f;
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
        const float sm = f[i] + f[i + 1], dm = f[i] - f[i + 1];
        drho += sm;
        if (cx27(i)) { jx += cx27(i) * dm; mxx += sm; }
        if (cy27(i)) { jy += cy27(i) * dm; myy += sm; }
        if (cz27(i)) { jz += cz27(i) * dm; mzz += sm; }
        if (cx27(i) * cy27(i)) mxy += cx27(i) * cy27(i) * sm;
        if (cx27(i) * cz27(i)) mxz += cx27(i) * cz27(i) * sm;
        if (cy27(i) * cz27(i)) myz += cy27(i) * cz27(i) * sm;
    }
    if (SCALED) {
        drho *= isf; jx *= isf; jy *= isf; jz *= isf;
        mxx *= isf; myy *= isf; mzz *= isf; mxy *= isf; mxz *= isf; myz *= isf;
    }
    const float rho = 1.0f + drho;
    const float irho = crcp<SCALED>(rho);
    const float ux = (jx + 0.5f * Fx) * irho;
    const float uy = (jy + 0.5f * Fy) * irho;
    const float uz = (jz + 0.5f * Fz) * irho;
    const float usq = ux * ux + uy * uy + uz * uz;

    // non-equilibrium second moment (sum c c feq = rho (I/3 + u u), sum c c w = I/3)
    const float d3 = drho * (1.0f / 3.0f);
    const float pxx = mxx - d3 - rho * ux * ux;
    const float pyy = myy - d3 - rho * uy * uy;
    const float pzz = mzz - d3 - rho * uz * uz;
    const float pxy = mxy - rho * ux * uy;
    const float pxz = mxz - rho * ux * uz;
    const float pyz = myz - rho * uy * uz;
    const float q = csqrt<SCALED>(pxx * pxx + pyy * pyy + pzz * pzz +
                          2.0f * (pxy * pxy + pxz * pxz + pyz * pyz));
    // tau - tau0 without cancellation: X / (2 (s + tau0)), s = sqrt(tau0^2 + X)
    const float X = kp.A * q * irho;
    const float s = csqrt<SCALED>(kp.tau0 * kp.tau0 + X);
    const float dtau = cdiv<SCALED>(0.5f * X, s + kp.tau0);
    const float om = crcp<SCALED>(kp.tau0 + dtau);
    const float keep = 1.0f - om;
    const float guo = 1.0f - 0.5f * om;
    const float uF = ux * Fx + uy * Fy + uz * Fz;
    // feq_i - w_i = w_i (drho + rho (3 cu + 4.5 cu^2 - 1.5 u.u)),
    // S_i = guo w_i (3 cF - 3 u.F + 9 cu cF)
    const float base = drho - 1.5f * rho * usq;       // even part of (feq - w)/w at cu = 0
    const float gbase = -3.0f * guo * uF;             // even part of S/w at cF = 0
    // node-wide coefficients, so that each direction pair costs
    // even = w (A0 + cu (Bq cu + Cq cF)), odd = w (Dq cu + Eq cF)
    // (A0 = om base + gbase; measured 1-2 % faster than expanding the terms
    // per direction)
    const float A0 = om * base + gbase;
    const float Bq = 4.5f * om * rho, Cq = 9.0f * guo;
    const float Dq = 3.0f * om * rho, Eq = 3.0f * guo;
    const float wa = sf * w19(1), wd = sf * w19(7);
    f[0] = keep * f[0] + sf * w19(0) * A0;
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
        const float cu = cx27(i) * ux + cy27(i) * uy + cz27(i) * uz;
        const float cF = cx27(i) * Fx + cy27(i) * Fy + cz27(i) * Fz;
        const float w = i < 7 ? wa : wd;
        const float even = w * fmaf(cu, fmaf(Bq, cu, Cq * cF), A0);
        const float odd = w * fmaf(Dq, cu, Eq * cF);
        f[i] = fmaf(keep, f[i], even + odd);
        f[i + 1] = fmaf(keep, f[i + 1], even - odd);
    }

    const float omp = crcp<SCALED>(kp.taup0 + kp.kT * dtau);
    if constexpr (SL == 7) {
        // scalar: Phi_eq - w = w (chi - 1 + 4 chi c.u).  Only the non-equilibrium
        // parts are relaxed, and the rest population's part closes their sum to
        // zero, so the update conserves sum Phi exactly up to the rounding of the
        // stored results (relaxing towards the rounded chi would inject
        // omega times the rounding error of the 7-term sum at every node)
        const float pe = w7(1) * chs, pa = sp * w7(1) * 4.0f * chi;
        float nq[7];
        nq[1] = p[1] - (pe + pa * ux);
        nq[2] = p[2] - (pe - pa * ux);
        nq[3] = p[3] - (pe + pa * uy);
        nq[4] = p[4] - (pe - pa * uy);
        nq[5] = p[5] - (pe + pa * uz);
        nq[6] = p[6] - (pe - pa * uz);
        nq[0] = -(((nq[1] + nq[2]) + (nq[3] + nq[4])) + (nq[5] + nq[6]));
#pragma unroll
        for (int k = 0; k < 7; ++k) p[k] -= omp * nq[k];
    } else {
        // D3Q6: Phi_eq - w = (chi - 1 + 3 chi c.u) / 6; with no rest population
        // the non-equilibrium parts are centred on their mean instead
        const float pe = chs * (1.0f / 6.0f), pa = sp * 0.5f * chi;
        float nq[6];
        nq[0] = p[0] - (pe + pa * ux);
        nq[1] = p[1] - (pe - pa * ux);
        nq[2] = p[2] - (pe + pa * uy);
        nq[3] = p[3] - (pe - pa * uy);
        nq[4] = p[4] - (pe + pa * uz);
        nq[5] = p[5] - (pe - pa * uz);
        const float r = (((nq[0] + nq[1]) + (nq[2] + nq[3])) + (nq[4] + nq[5])) * (1.0f / 6.0f);
#pragma unroll
        for (int k = 0; k < 6; ++k) p[k] -= omp * (nq[k] - r);
    }
}

}  // namespace lbmgpu
