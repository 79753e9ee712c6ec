// lbm_bgk.cu -- fused AA stream + collide kernels of the D3Q19 BGK-Smagorinsky
// fluid with the D3Q7 scalar and the Boussinesq force.
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
// followed by streaming (Eq. 17) in the AA pattern of lbm_common.cuh.
//
// FP32: two nodes per thread, x and x + 32 of a 64-node segment of a row
// (lbm_pair.cuh), collided in packed arithmetic.  Large boxes are bound by HBM
// (208 bytes per node update, about 2 flop per byte) when steps are launched one
// by one: 32.8 G node updates/s at 2048x128x256, 1.00 of the measured copy rate, as
// the form before it (pairs of adjacent nodes, collided one after the other).
// Boxes that fit the L2 and rows of odd length were bound by instruction issue: 322
// instructions per node on both parities (456 / 634 before on even / odd steps)
// took the step from 17.4 to 12.8 us at 256x32x64 and from 35.3 to 28.8 us at
// 333x47x59, overlapped launches (launch_after) to 10.9 and 25.9.
//
// 16-bit storage: adjacent pairs (lbm_aa2.cuh) and, on even steps with nx a
// multiple of 4, packed quads (lbm_quad.cuh); nx odd: one node per thread.
// No shared memory, no tensor cores.
#include <type_traits>

#include "lbm_aa2.cuh"
#include "lbm_bgk_collide.cuh"
#include "lbm_chain.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_quad.cuh"

namespace lbmgpu {

// CONTRACT: FP32 in the compiler-contracted arithmetic (collide_bgk), as the
// 16-bit forms always.
template <bool ODD, bool SAVE, typename S, int SL, typename Off = unsigned, bool CONTRACT = false>
__global__ void __launch_bounds__(128, LBM_STEP_MINB) bgk_step_kernel(KParams kp, S* __restrict__ f,
                                                       S* __restrict__ phi,
                                                       float* __restrict__ save) {
    step_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= kp.nx) return;
    const Stencil st = make_stencil(kp, x, blockIdx.y, blockIdx.z);
    const unsigned n = st.n;

    constexpr int NS = ScalarLat<SL>::NS, D0 = ScalarLat<SL>::D0;
    constexpr bool R32 = rest32<S, SL>();
    float fv[19], pv[NS];
    gather<19, ODD, S, 0, false, true, Off>(kp, f, st, fv);
    gather<NS, ODD, S, D0, R32, true, Off>(kp, phi, st, pv);
    constexpr bool s16 = !std::is_same<S, float>::value;   // populations in storage units
    if (SAVE) {
#pragma unroll
        for (int i = 0; i < 19; ++i) save_pop(kp, save, 19 + NS, i, n, s16 ? fv[i] * kp.isf : fv[i]);
#pragma unroll
        for (int k = 0; k < NS; ++k)
            save_pop(kp, save, 19 + NS, 19 + k, n,
                     s16 ? phi_canonical(kp, pv[k], ScalarLat<SL>::w(k)) : pv[k]);
    }
    if (!(kp.flags & LBM_FLAG_NO_COLLIDE)) {
        if constexpr (s16 || CONTRACT) collide_bgk<s16, SL>(kp, fv, pv);
        else collide_bgk_lanes<One, SL>(kp, kp.gx, kp.gy, kp.gz, fv, pv);
    }
    if constexpr (R32) feed_rest<S>(pv);
    scatter<19, ODD, S, 0, false, true, Off>(kp, f, st, fv);
    scatter<NS, ODD, S, D0, R32, true, Off>(kp, phi, st, pv);
}


// FP32: two nodes per thread, x and x + 32 (lbm_pair.cuh), one code for both
// parities, packed arithmetic.
template <int SL, bool EDGE, bool WIDE>
__device__ __forceinline__ void bgk_pair_step(const KParams& kp, const PairTable<9, 3>& tab,
                                              float* __restrict__ f, float* __restrict__ phi,
                                              bool odd, int x0, int y, int z) {
    constexpr int NS = ScalarLat<SL>::NS, D0 = ScalarLat<SL>::D0;
    const PairNodes pn = pair_nodes(kp, x0, y, z, odd);
    const int cls = pair_class(kp, odd, y, z);
    const size_t fe = (size_t)19 * kp.N, pe = (size_t)NS * kp.N;
    float2 fv[19], pv[NS];
    pair_gather<9, 0, 19, float, EDGE, WIDE>(kp, f, pn, tab.f[cls], fv);
    pair_gather<3, D0, NS, float, EDGE, WIDE>(kp, phi, pn, tab.g[cls], pv);
    fv[0] = pair_ld_rest<float, EDGE>(kp, f, fe, pn);
    if constexpr (SL == 7) pv[0] = pair_ld_rest<float, EDGE>(kp, phi, pe, pn);
    if (!(kp.flags & LBM_FLAG_NO_COLLIDE)) {
        const float s = odd ? 1.0f : -1.0f;   // even steps see the mirrored velocity set
        collide_bgk_lanes<Two, SL>(kp, s * kp.gx, s * kp.gy, s * kp.gz, fv, pv);
    }
    pair_scatter<9, 0, 19, float, EDGE, WIDE>(kp, f, pn, tab.f[cls], fv);
    pair_scatter<3, D0, NS, float, EDGE, WIDE>(kp, phi, pn, tab.g[cls], pv);
    pair_st_rest<float, EDGE>(kp, f, fe, pn, fv[0]);
    if constexpr (SL == 7) pair_st_rest<float, EDGE>(kp, phi, pe, pn, pv[0]);
}

template <int SL, bool WIDE>
__global__ void __launch_bounds__(128, LBM_PAIR_MINB)
    bgk_pair_kernel(const __grid_constant__ KParams kp,
                    const __grid_constant__ PairTable<9, 3> tab, float* __restrict__ f,
                    float* __restrict__ phi, bool odd) {
    step_begin();
    const int x0 = 64 * (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (x0 >= kp.nx) return;
    if (pair_inner(kp, x0))
        bgk_pair_step<SL, false, WIDE>(kp, tab, f, phi, odd, x0, blockIdx.y, blockIdx.z);
    else
        bgk_pair_step<SL, true, WIDE>(kp, tab, f, phi, odd, x0, blockIdx.y, blockIdx.z);
}

#ifndef LBM_BGK_ZSPLIT
#define LBM_BGK_ZSPLIT 1
#endif
#ifndef LBM_BGK_FAST
#define LBM_BGK_FAST 1
#endif

// The 16-bit instantiations are issue-bound rather than HBM-bound, so they
// may trade registers for resident warps differently (LBM_STEP2_MINB16).
#ifndef LBM_STEP2_MINB16
#define LBM_STEP2_MINB16 LBM_STEP2_MINB
#endif

template <bool ODD, bool SAVE, typename S, int SL, bool ZW, bool FAST, typename Off>
__device__ __forceinline__ void bgk_step2_body(const KParams& kp, S* __restrict__ f,
                                               S* __restrict__ phi, float* __restrict__ save,
                                               const Stencil2& st) {
    constexpr int NS = ScalarLat<SL>::NS, D0 = ScalarLat<SL>::D0;
    constexpr bool R32 = rest32<S, SL>();
    float f0[19], f1[19], p0[NS], p1[NS];
    gather2<19, ODD, S, 0, false, ZW, FAST, Off>(kp, f, st, f0, f1);
    gather2<NS, ODD, S, D0, R32, ZW, FAST, Off>(kp, phi, st, p0, p1);
    constexpr bool s16 = !std::is_same<S, float>::value;   // populations in storage units
    if (SAVE && st.active) {
        const unsigned N = kp.N;
        const float a = s16 ? kp.isf : 1.0f;
#pragma unroll
        for (int i = 0; i < 19; ++i)
            *reinterpret_cast<float2*>(save + (size_t)i * N + st.n) = make_float2(a * f0[i], a * f1[i]);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const float w = ScalarLat<SL>::w(k);
            *reinterpret_cast<float2*>(save + (size_t)(19 + k) * N + st.n) =
                s16 ? make_float2(phi_canonical(kp, p0[k], w), phi_canonical(kp, p1[k], w))
                    : make_float2(p0[k], p1[k]);
        }
    }
    if (!(kp.flags & LBM_FLAG_NO_COLLIDE)) {
        collide_bgk<s16, SL>(kp, f0, p0);
        collide_bgk<s16, SL>(kp, f1, p1);
    }
    if constexpr (R32) feed_rest2<S>(p0, p1);
    scatter2<19, ODD, S, 0, false, ZW, FAST, Off>(kp, f, st, f0, f1);
    scatter2<NS, ODD, S, D0, R32, ZW, FAST, Off>(kp, phi, st, p0, p1);
}

// Two x-adjacent nodes per thread (nx even): paired population accesses, see
// lbm_aa2.cuh.  Same arithmetic per node as bgk_step_kernel.  On odd steps
// the rows away from the z walls (uniform per block) take a body without the
// wall selects.
template <bool ODD, bool SAVE, typename S, int SL, typename Off = unsigned>
__global__ void __launch_bounds__(128, std::is_same<S, float>::value ? LBM_STEP2_MINB : LBM_STEP2_MINB16) bgk_step2_kernel(KParams kp, S* __restrict__ f,
                                                                    S* __restrict__ phi,
                                                                    float* __restrict__ save) {
    step_begin();
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const Stencil2 st = make_stencil2(kp, x, blockIdx.y, blockIdx.z);
    const int z = blockIdx.z;
    const bool zwall = ODD && (!LBM_BGK_ZSPLIT ||
                               (!(kp.flags & LBM_FLAG_PERIODIC_Z) && (z == 0 || z == kp.nz - 1)));
    if (!ODD) bgk_step2_body<ODD, SAVE, S, SL, false, false, Off>(kp, f, phi, save, st);
    else if (LBM_BGK_FAST && block_interior2(kp))
        bgk_step2_body<ODD, SAVE, S, SL, false, true, Off>(kp, f, phi, save, st);
    else if (!zwall) bgk_step2_body<ODD, SAVE, S, SL, false, false, Off>(kp, f, phi, save, st);
    else bgk_step2_body<ODD, SAVE, S, SL, true, false, Off>(kp, f, phi, save, st);
}

#ifndef LBM_STEP4_MINB
#define LBM_STEP4_MINB 3
#endif

// Even steps with 16-bit storage and nx a multiple of 4: four x-adjacent
// nodes per thread, each population row moved as one aligned 8-byte word
// (a warp reads and writes 256-byte row segments, as the FP32 pair kernel
// does, against 128 for 16-bit pairs).  Even steps are local (slot i of node
// n is read, slot opp(i) of the same node written), so the words need no
// shifting; the four nodes are unpacked, collided and packed back one at a
// time.  Same arithmetic per node as bgk_step_kernel.  Odd steps stay with
// bgk_step2_kernel: there the x-shifted rows of a packed quad need shuffles
// and byte permutes and measured slower than the paired form.
struct BgkQuadCollide {
    template <int SL, typename S>
    static __device__ __forceinline__ void run(const KParams& kp, float (&f)[19],
                                               float (&p)[ScalarLat<SL>::NS]) {
        collide_bgk<true, SL>(kp, f, p);
    }
};

template <typename S, int SL, typename Off = unsigned>
__global__ void __launch_bounds__(128, LBM_STEP4_MINB) bgk_even4_kernel(KParams kp, S* __restrict__ f,
                                                                       S* __restrict__ phi) {
    step_begin();
    even4_body<19, SL, S, Off, BgkQuadCollide>(kp, f, phi);
}

// Many steps in one launch (lbm_chain.cuh).  14 computing warps: 128 registers
// without spills (18 warps at 96 registers spill 244 bytes and measured 28
// against 39 G node updates/s at 2048x128x256).  The body has to be small: with
// the former step kernels inlined (four bodies of 17 to 20 KB) the mixed
// parities missed the instruction cache (3.3 of 11.6 cycles per issue) and ran
// at 26 G.  Per step, one overlapped launch each -> chain: 256x32x64
// 11.1 -> 10.5 us, 333x47x59 25.9 -> 23.2, 1024x64x128 252 -> 183, 2048x128x256
// 2050 -> 1680 (39.9 G node updates/s, 8.3 TB/s of populations); boxes of fewer
// rows are faster one launch at a time (chain_plan).
template <int SL>
__global__ void __launch_bounds__(CHAIN_THREADS, 1)
    bgk_chain_kernel(const __grid_constant__ KParams kp, const __grid_constant__ ChainParams cp,
                     const __grid_constant__ PairTable<9, 3> tab, float* __restrict__ f,
                     float* __restrict__ phi) {
    chain_run<CHAIN_WARPS>(kp, cp, [&](bool odd, int seg, int y, int z) {
        const int x0 = 64 * seg;
        if (pair_inner(kp, x0))
            bgk_pair_step<SL, false, false>(kp, tab, f, phi, odd, x0, y, z);
        else
            bgk_pair_step<SL, true, false>(kp, tab, f, phi, odd, x0, y, z);
    });
}

template <int SL>
static cudaError_t launch_chain(const KParams& kp, const ChainPlan& pl, const Views& v,
                                cudaStream_t st) {
    bgk_chain_kernel<SL><<<pl.grid, CHAIN_THREADS, 0, st>>>(
        kp, pl.p, pair_view<9, 3>(*v.sides), (float*)v.f, (float*)v.phi);
    return cudaGetLastError();
}

cudaError_t launch_bgk_chain(const KParams& kp, Kind k, bool odd, int nsteps, const Views& v,
                             int& done, cudaStream_t st) {
    ChainPlan pl;
    const cudaError_t e = chain_prepare(kp, k, v, nsteps, odd, pl, done, st);
    if (e != cudaSuccess || !done) return e;
    return k.scalar == LBM_SCALAR_Q7 ? launch_chain<7>(kp, pl, v, st) : launch_chain<6>(kp, pl, v, st);
}

// The steps in the contracted arithmetic: every 16-bit step, and in FP32 the
// saved steps, the trajectory of an objective (lbm_objective_forward) and, in
// lbm_adjoint.cu, its recompute in the reverse sweep, which have to retrace each
// other.  (A gradient of the front divides by differences of chi of a few 1e-3
// at chi ~ 0.02, held as chi - 1 in FP32: its error, 1e-6 to 3e-5, is the
// rounding of this one trajectory, so another arithmetic, however accurate,
// gives another error of the same size; these paths keep theirs.)
template <typename S, int SL, typename Off>
static cudaError_t launch_bgk_contracted(const KParams& kp, bool odd, S* f, S* phi, float* save,
                                         cudaStream_t st) {
    // saved steps need (Q + NS) N < 2^32
    constexpr bool narrow = std::is_same<Off, unsigned>::value;
    if (save && !narrow) return cudaErrorInvalidValue;
    if ((kp.flags & LBM_FLAG_ONE_NODE) || kp.nx % 2) {
        dim3 block(128), grid((kp.nx + 127) / 128, kp.ny, kp.nz);
        if (save) {
            if (odd) launch_after(bgk_step_kernel<true, true, S, SL, unsigned, true>, grid, block, st, kp, f, phi, save);
            else launch_after(bgk_step_kernel<false, true, S, SL, unsigned, true>, grid, block, st, kp, f, phi, save);
        } else {
            if (odd) launch_after(bgk_step_kernel<true, false, S, SL, Off, true>, grid, block, st, kp, f, phi, nullptr);
            else launch_after(bgk_step_kernel<false, false, S, SL, Off, true>, grid, block, st, kp, f, phi, nullptr);
        }
        return cudaGetLastError();
    }
    if constexpr (!std::is_same<S, float>::value) {
        if (!odd && !save && kp.nx % 4 == 0) {
            dim3 block(128), grid((kp.nx / 4 + 127) / 128, kp.ny, kp.nz);
            launch_after(bgk_even4_kernel<S, SL, Off>, grid, block, st, kp, f, phi);
            return cudaGetLastError();
        }
    }
    dim3 block(128), grid((kp.nx / 2 + 127) / 128, kp.ny, kp.nz);
    if (save) {
        if (odd) launch_after(bgk_step2_kernel<true, true, S, SL>, grid, block, st, kp, f, phi, save);
        else launch_after(bgk_step2_kernel<false, true, S, SL>, grid, block, st, kp, f, phi, save);
    } else {
        if (odd) launch_after(bgk_step2_kernel<true, false, S, SL, Off>, grid, block, st, kp, f, phi, nullptr);
        else launch_after(bgk_step2_kernel<false, false, S, SL, Off>, grid, block, st, kp, f, phi, nullptr);
    }
    return cudaGetLastError();
}

template <int SL, bool WIDE>
static cudaError_t launch_bgk_fp32(const KParams& kp, const Sides& sides, bool odd, float* f,
                                   float* phi, cudaStream_t st) {
    if (kp.flags & LBM_FLAG_ONE_NODE) {
        using Off = std::conditional_t<WIDE, size_t, unsigned>;
        dim3 block(128), grid((kp.nx + 127) / 128, kp.ny, kp.nz);
        if (odd) launch_after(bgk_step_kernel<true, false, float, SL, Off>, grid, block, st, kp, f, phi, nullptr);
        else launch_after(bgk_step_kernel<false, false, float, SL, Off>, grid, block, st, kp, f, phi, nullptr);
        return cudaGetLastError();
    }
    const int ns = (kp.nx + 63) / 64, w = pair_warps(ns);
    dim3 block(32 * w), grid((ns + w - 1) / w, kp.ny, kp.nz);
    launch_after(bgk_pair_kernel<SL, WIDE>, grid, block, st, kp, pair_view<9, 3>(sides), f, phi, odd);
    return cudaGetLastError();
}

void fill_bgk_sides(const KParams& kp, int scalar, Sides& s) {
    pair_table(kp, scalar == LBM_SCALAR_Q6 ? 1 : 0, pair_view<9, 3>(s));
}

template <typename S, int SL>
static cudaError_t launch_bgk_typed(const KParams& kp, bool odd, const Views& v, float* save,
                                    bool trajectory, cudaStream_t st) {
    S *f = (S*)v.f, *phi = (S*)v.phi;
    if constexpr (std::is_same<S, float>::value) {
        if (!save && !trajectory)
            return kp.wide ? launch_bgk_fp32<SL, true>(kp, *v.sides, odd, f, phi, st)
                           : launch_bgk_fp32<SL, false>(kp, *v.sides, odd, f, phi, st);
    }
    return kp.wide ? launch_bgk_contracted<S, SL, size_t>(kp, odd, f, phi, save, st)
                   : launch_bgk_contracted<S, SL, unsigned>(kp, odd, f, phi, save, st);
}

template <int SL>
static cudaError_t launch_bgk_sl(const KParams& kp, int storage, bool odd, const Views& v,
                                 float* save, bool trajectory, cudaStream_t st) {
    switch (storage) {
        case LBM_FP32: return launch_bgk_typed<float, SL>(kp, odd, v, save, trajectory, st);
        case LBM_FP16S: return launch_bgk_typed<__half, SL>(kp, odd, v, save, trajectory, st);
        case LBM_BF16S: return launch_bgk_typed<__nv_bfloat16, SL>(kp, odd, v, save, trajectory, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_bgk_step(const KParams& kp, int storage, int scalar, bool odd, const Views& v,
                            float* save, bool trajectory, cudaStream_t st) {
    if (scalar == LBM_SCALAR_Q7) return launch_bgk_sl<7>(kp, storage, odd, v, save, trajectory, st);
    if (scalar == LBM_SCALAR_Q6) return launch_bgk_sl<6>(kp, storage, odd, v, save, trajectory, st);
    return cudaErrorInvalidValue;
}

}  // namespace lbmgpu
