// lbm_cumulant_lanes.cuh -- the cumulant collision of lbm_cumulant_collide.cuh
// with the D3Q7 scalar, in FP32, on one node or on two side by side
// (lbm_lanes.cuh), every operation written out.
//
// Same map: moments of order <= 2 by lines, relaxation of the covariance, the
// Gaussian central moments, and the per-axis inverse stages on z, y and x, in
// place on one array of 27 values (the populations are dead once their moments
// are taken), leaving out the terms that are zero.  Every operation is odd or
// even under c -> -c.
#pragma once

#include "lbm_cumulant_collide.cuh"
#include "lbm_lanes.cuh"

namespace lbmgpu {

// Inverse of the central-moment map along one axis (axis_inverse): the line
// (d0, d1, d2), held as deviations from s (1, 0, 1/3) in the frame moving with
// v, becomes (p(-1), p(0), p(+1)).  hv2 = v^2 / 2.  D0, D1, D2: which entries are
// not zero; S: s is not zero.
template <typename L, bool S, bool D0, bool D1, bool D2>
__device__ __forceinline__ void line_inverse(float s, typename L::V v, typename L::V v2,
                                             typename L::V& d0, typename L::V& d1,
                                             typename L::V& d2) {
    using V = typename L::V;
    const V half = L::set(0.5f);
    if constexpr (!S && !D0) {
        // only d1: a = 2 v d1, b = d1
        const V h = L::mul(v, d1), b = L::mul(half, d1);
        d0 = L::sub(h, b);
        d1 = L::mul(L::set(-2.0f), h);
        d2 = L::add(h, b);
    } else {
        const V k0 = !S ? d0 : (D0 ? L::add(d0, L::set(s)) : L::set(s));
        V a, b;
        if constexpr (D1) {
            const V t = L::add(v, v);
            a = L::fma(v2, k0, D2 ? L::fma(t, d1, d2) : L::mul(t, d1));
            b = L::fma(v, k0, d1);
        } else {
            a = D2 ? L::fma(v2, k0, d2) : L::mul(v2, k0);
            b = L::mul(v, k0);
        }
        const V h = L::mul(half, a);
        const V p0 = D0 ? L::sub(d0, a) : L::neg(a);
        d0 = L::fma(L::set(-0.5f), b, h);
        d2 = L::fma(half, b, h);
        d1 = p0;
    }
}

// The fluid: replaces f by its post-collision populations, given chit = chi - 1
// and the force F per unit chi (with the sign of the velocity set that f is
// named in); returns chi and the half-force velocity h.
template <typename L>
__device__ __forceinline__ void cumulant_fluid_lanes(const KParams& kp, float gx, float gy,
                                                     float gz, typename L::V (&f)[27],
                                                     typename L::V chit, typename L::V& chi,
                                                     typename L::V& hx, typename L::V& hy,
                                                     typename L::V& hz) {
    using V = typename L::V;
    chi = L::add(chit, L::set(1.0f));
    const V Fx = L::mul(L::set(gx), chi), Fy = L::mul(L::set(gy), chi), Fz = L::mul(L::set(gz), chi);

    // moments by lines: along x, then y, then z
    V m00[3], m10[3], m01[3], m02[3], m11[3], m20[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        V L0[3], L1[3], L2[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const V pm = f[dir27(-1, b - 1, c - 1)], pp = f[dir27(1, b - 1, c - 1)];
            L2[b] = L::add(pp, pm);
            L0[b] = L::add(L2[b], f[dir27(0, b - 1, c - 1)]);
            L1[b] = L::sub(pp, pm);
        }
        m02[c] = L::add(L0[0], L0[2]);
        m00[c] = L::add(m02[c], L0[1]);
        m01[c] = L::sub(L0[2], L0[0]);
        m10[c] = L::add(L::add(L1[0], L1[2]), L1[1]);
        m11[c] = L::sub(L1[2], L1[0]);
        m20[c] = L::add(L::add(L2[0], L2[2]), L2[1]);
    }
    const V mzz = L::add(m00[2], m00[0]), drho = L::add(mzz, m00[1]);
    const V jx = L::add(L::add(m10[0], m10[2]), m10[1]);
    const V jy = L::add(L::add(m01[0], m01[2]), m01[1]);
    const V jz = L::sub(m00[2], m00[0]);
    const V mxx = L::add(L::add(m20[0], m20[2]), m20[1]);
    const V myy = L::add(L::add(m02[0], m02[2]), m02[1]);
    const V mxy = L::add(L::add(m11[0], m11[2]), m11[1]);
    const V mxz = L::sub(m10[2], m10[0]), myz = L::sub(m01[2], m01[0]);

    const V rho = L::add(drho, L::set(1.0f));
    const V irho = lane_rcp<L>(rho);
    // covariance (deviation of the diagonal from 1/3), relaxed
    const V vx = L::mul(jx, irho), vy = L::mul(jy, irho), vz = L::mul(jz, irho);
    const V nx = L::neg(vx), ny = L::neg(vy), nz = L::neg(vz), n3 = L::set(-1.0f / 3.0f);
    const V cxx = L::fma(nx, vx, L::mul(L::fma(n3, drho, mxx), irho));
    const V cyy = L::fma(ny, vy, L::mul(L::fma(n3, drho, myy), irho));
    const V czz = L::fma(nz, vz, L::mul(L::fma(n3, drho, mzz), irho));
    const V r1 = L::set(1.0f - kp.om1);
    const V sxy = L::mul(r1, L::fma(nx, vy, L::mul(mxy, irho)));
    const V sxz = L::mul(r1, L::fma(nx, vz, L::mul(mxz, irho)));
    const V syz = L::mul(r1, L::fma(ny, vz, L::mul(myz, irho)));
    const V E1 = L::mul(r1, L::sub(cxx, cyy)), E2 = L::mul(r1, L::sub(cxx, czz));
    const V T = L::mul(L::set(1.0f - kp.om2), L::add(L::add(cxx, cyy), czz));
    const V t3 = L::set(1.0f / 3.0f);
    const V sxx = L::mul(L::add(T, L::add(E1, E2)), t3);
    const V syy = L::sub(sxx, E1), szz = L::sub(sxx, E2);
    // post-collision velocity
    const V ux = L::mul(L::add(jx, Fx), irho), uy = L::mul(L::add(jy, Fy), irho),
            uz = L::mul(L::add(jz, Fz), irho);
    const V half = L::set(0.5f);
    hx = L::mul(L::fma(half, Fx, jx), irho);
    hy = L::mul(L::fma(half, Fy, jy), irho);
    hz = L::mul(L::fma(half, Fz, jz), irho);

    // central-moment deviations of the Gaussian, index 9 a + 3 b + c
    const V gx3 = L::add(sxx, t3), gy3 = L::add(syy, t3), gz3 = L::add(szz, t3);
    const V axy = L::add(sxy, sxy), axz = L::add(sxz, sxz), ayz = L::add(syz, syz);
    V K[27];
    K[18] = sxx; K[6] = syy; K[2] = szz;
    K[12] = sxy; K[10] = sxz; K[4] = syz;
    const V pxy = L::mul(sxx, syy);
    K[24] = L::fma(axy, sxy, L::fma(L::add(sxx, syy), t3, pxy));
    K[20] = L::fma(axz, sxz, L::fma(L::add(sxx, szz), t3, L::mul(sxx, szz)));
    K[8] = L::fma(ayz, syz, L::fma(L::add(syy, szz), t3, L::mul(syy, szz)));
    K[22] = L::fma(axy, sxz, L::mul(gx3, syz));
    K[16] = L::fma(axy, syz, L::mul(gy3, sxz));
    K[14] = L::fma(axz, syz, L::mul(gz3, sxy));
    {
        // s_xx s_yy s_zz of the full covariance minus 1/27, the pairs and the triple
        const V q = L::fma(sxx, szz, L::fma(syy, szz, pxy));
        V k = L::fma(L::add(L::add(sxx, syy), szz), L::set(1.0f / 9.0f), L::mul(q, t3));
        k = L::fma(pxy, szz, k);
        k = L::fma(L::mul(gx3, ayz), syz, k);
        k = L::fma(L::mul(gy3, axz), sxz, k);
        k = L::fma(L::mul(gz3, axy), sxy, k);
        K[26] = L::fma(L::mul(L::mul(L::set(4.0f), axy), sxz), syz, k);
    }
    // inverse stages, in place: z
    const V z2 = L::mul(uz, uz), y2 = L::mul(uy, uy), x2 = L::mul(ux, ux);
    constexpr float c9 = 1.0f / 9.0f, c3 = 1.0f / 3.0f;
    line_inverse<L, true, false, false, true>(1.0f, uz, z2, K[0], K[1], K[2]);
    line_inverse<L, false, false, true, false>(0.0f, uz, z2, K[3], K[4], K[5]);
    line_inverse<L, true, true, false, true>(c3, uz, z2, K[6], K[7], K[8]);
    line_inverse<L, false, false, true, false>(0.0f, uz, z2, K[9], K[10], K[11]);
    line_inverse<L, false, true, false, true>(0.0f, uz, z2, K[12], K[13], K[14]);
    line_inverse<L, false, false, true, false>(0.0f, uz, z2, K[15], K[16], K[17]);
    line_inverse<L, true, true, false, true>(c3, uz, z2, K[18], K[19], K[20]);
    line_inverse<L, false, false, true, false>(0.0f, uz, z2, K[21], K[22], K[23]);
    line_inverse<L, true, true, false, true>(c9, uz, z2, K[24], K[25], K[26]);
    // y: rest values R[a] W1[c]
    constexpr float W1[3] = {1.0f / 6.0f, 2.0f / 3.0f, 1.0f / 6.0f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        line_inverse<L, true, true, true, true>(W1[c], uy, y2, K[c], K[3 + c], K[6 + c]);
        line_inverse<L, false, true, true, true>(0.0f, uy, y2, K[9 + c], K[12 + c], K[15 + c]);
        line_inverse<L, true, true, true, true>(c3 * W1[c], uy, y2, K[18 + c], K[21 + c], K[24 + c]);
    }
    // x, and f*_i - w_i = drho w_i + rho (P_i - w_i)
    const V dw[4] = {L::mul(drho, L::set(w27(0))), L::mul(drho, L::set(w27(1))),
                     L::mul(drho, L::set(w27(7))), L::mul(drho, L::set(w27(19)))};
    const V t = L::add(ux, ux), hr = L::mul(half, rho);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const V d0 = K[3 * b + c], d1 = K[9 + 3 * b + c], d2 = K[18 + 3 * b + c];
            const V k0 = L::add(d0, L::set(W1[b] * W1[c]));
            const V a = L::fma(x2, k0, L::fma(t, d1, d2)), e = L::fma(ux, k0, d1);
            const int n0 = (b != 1) + (c != 1);   // class of the weight of c_x = 0
            f[dir27(0, b - 1, c - 1)] = L::fma(rho, L::sub(d0, a), dw[n0]);
            f[dir27(-1, b - 1, c - 1)] = L::fma(hr, L::sub(a, e), dw[n0 + 1]);
            f[dir27(1, b - 1, c - 1)] = L::fma(hr, L::add(a, e), dw[n0 + 1]);
        }
}

// chi - 1 of the D3Q7 scalar.
template <typename L>
__device__ __forceinline__ typename L::V scalar7_chit(const typename L::V (&p)[7]) {
    return L::add(p[0], L::add(L::add(L::add(p[1], p[2]), L::add(p[3], p[4])), L::add(p[5], p[6])));
}

// D3Q7 BGK with the molecular D, in the non-equilibrium form whose parts sum to
// zero (collide_cumulant).
template <typename L>
__device__ __forceinline__ void scalar7_lanes(const KParams& kp, typename L::V (&p)[7],
                                              typename L::V chit, typename L::V chi,
                                              typename L::V hx, typename L::V hy,
                                              typename L::V hz) {
    using V = typename L::V;
    const V pe = L::mul(L::set(0.125f), chit), pa = L::mul(L::set(0.5f), chi), na = L::neg(pa);
    V nq[6];
    nq[0] = L::sub(p[1], L::fma(pa, hx, pe));
    nq[1] = L::sub(p[2], L::fma(na, hx, pe));
    nq[2] = L::sub(p[3], L::fma(pa, hy, pe));
    nq[3] = L::sub(p[4], L::fma(na, hy, pe));
    nq[4] = L::sub(p[5], L::fma(pa, hz, pe));
    nq[5] = L::sub(p[6], L::fma(na, hz, pe));
    const V sum = L::add(L::add(L::add(nq[0], nq[1]), L::add(nq[2], nq[3])), L::add(nq[4], nq[5]));
    const V om = L::set(kp.omp0), no = L::set(-kp.omp0);
    p[0] = L::fma(om, sum, p[0]);
#pragma unroll
    for (int k = 0; k < 6; ++k) p[1 + k] = L::fma(no, nq[k], p[1 + k]);
}

// The collision, g with the sign of the velocity set that f and p are named in.
template <typename L>
__device__ __forceinline__ void collide_cumulant_lanes(const KParams& kp, float gx, float gy,
                                                       float gz, typename L::V (&f)[27],
                                                       typename L::V (&p)[7]) {
    typename L::V chi, hx, hy, hz;
    const typename L::V chit = scalar7_chit<L>(p);
    cumulant_fluid_lanes<L>(kp, gx, gy, gz, f, chit, chi, hx, hy, hz);
    scalar7_lanes<L>(kp, p, chit, chi, hx, hy, hz);
}

}  // namespace lbmgpu
