// lbm_aux.cuh -- initial state and diagnostics kernels, generic over the precision
// policy (lbm_prec.cuh).  The diagnostics evaluate in FP64, the initial state in FP64 or
// double words; both (de)quantise at the load / store.
#pragma once

#include "lbm_device.cuh"
#include "lbm_prec.cuh"
#include "lbm_step.cuh"

namespace lbm {

// Arithmetic type of the initial state's equilibria: FP64 for the FP64 policy, double words
// (48 bits, on the FP32 pipes) for every other one.
template <class R>
using init_t = typename std::conditional<std::is_same<R, double>::value, double, df64>::type;

// An FP64 input of the initial state as the arithmetic type.  For double words: the pair of
// df64(double) (x rounded to FP32, and the rest rounded to FP32; of two equally near x the one
// further from zero), put together with integer instructions.  The four FP64 instructions of
// the conversion occupy a scheduler's share of the FP64 unit for 64 cycles each: the N + 3
// inputs held that unit for 43 of the kernel's 78 us at 1024^2, N = 3, FP16 storage; now 64 us.  Only
// values so small or so large that a part would leave FP32's normal range are converted there.
template <class I>
__device__ __forceinline__ I init_input(double x)
{
    if constexpr (std::is_same<I, df64>::value) {
        constexpr int ONE = 0x00100000;                     // one of a double's exponent, in its upper word
        const int h = __double2hiint(x), l = __double2loint(x);
        if ((unsigned)((h & 0x7ff00000) - (1023 - 70) * ONE) < 196u * ONE) {
            const unsigned bl = (unsigned)l + 0x10000000u;  // half of the last bit that hi keeps
            const int bh = h + (bl < 0x10000000u);
            const unsigned hi = ((unsigned)((bh & 0x7fffffff) - 896 * ONE) << 3) | (bl >> 29);
            const unsigned unit = (unsigned)((h & 0x7ff00000) - 948 * ONE) << 3;   // 2^(exponent - 52)
            const float lo = (float)((int)(bl & 0x1fffffffu) - 0x10000000);
            const unsigned sign = (unsigned)h & 0x80000000u;
            return df64(__uint_as_float(hi | sign), lo * __uint_as_float(unit | sign));
        }
        if (((h << 1) | l) == 0) return df64(__int_as_float(h), 0.0f);   // 0 and -0
    }
    return I(x);
}

// A value of the initial state as the policy's arithmetic type (rounded once).
template <class R, class I>
__device__ __forceinline__ R init_value(I v)
{
    if constexpr (std::is_same<I, df64>::value && std::is_same<R, float>::value) return __fadd_rn(v.hi, v.lo);
    else return (R)v;
}

// eq. H inverted for one cell (the map, and what follows from it), FP64: rho H, T, rho, c_p, psi.
template <int N>
__device__ __forceinline__ void init_macro(const KParams& P, const double (&phi)[N], double T_in, double& rhoH, double& T,
                                           double& rho, double& cp, double& psi)
{
    const Mix<N> m = mixture_core<N>(P, phi);
    rhoH = inverse_map<N>(P, m, T_in);
    double fl;
    enthalpy_map<N, true>(P, m, rhoH, fl, T);
    const double fs = 1.0 - fl;
    rho = fma(fs, m.rs, fl * m.rl);
    cp = fma(fs, m.cs, fl * m.cl);
    psi = fs * m.dr;
}

// The same in double words, for a cell whose phase the input temperature decides with margin
// (returns false for any other: the FP64 form is then asked).  Above the liquidus the cell is
// liquid whatever its latent heat; below the solidus it is solid where it holds
// phase-changing material.  Either way the map returns the temperature it was given.  The
// screen runs on FP32 values of the inputs; its margin of 1e-5 of the magnitudes is 25
// times their rounding.
template <int N>
__device__ __forceinline__ bool init_macro_decided(const KParams& P, const df64 (&phi)[N], df64 T, df64& rhoH, df64& rho,
                                                   df64& cp, df64& psi)
{
    const Coef<float>& C = P.f;
    float rs = 0.0f, rl = 0.0f, cs = 0.0f, cl = 0.0f, Lv = 0.0f, La = 0.0f;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        rs = fmaf(phi[p].hi, C.rho_s[p], rs);
        rl = fmaf(phi[p].hi, C.rho_l[p], rl);
        cs = fmaf(phi[p].hi, C.cp_s[p], cs);
        cl = fmaf(phi[p].hi, C.cp_l[p], cl);
        Lv = fmaf(phi[p].hi, C.rhoL[p], Lv);
        La = fmaf(fabsf(phi[p].hi), C.rhoL[p], La);
    }
    const float t = T.hi, tolT = 1e-5f * (fabsf(t) + fabsf(C.T_sol) + fabsf(C.T_liq)) + 1e-30f;
    const Coef<df64>& X = P.x;
    if (t > C.T_liq + tolT) {
        const float rcl = rl * cl, As = rs * cs * C.T_sol, Al = fmaf(rcl, C.T_liq, Lv);
        const float h = fmaf(rcl, t - C.T_liq, Al);
        const float tol = 1e-5f * (fabsf(As) + fabsf(rcl * C.T_liq) + fabsf(rcl * t) + La) + 1e-30f;
        if (!(rl > 1e-20f && cl > 1e-20f && h > As + tol)) return false;
        rho = mix_sum<N, df64>(phi, X.rho_l);
        cp = mix_sum<N, df64>(phi, X.cp_l);
        rhoH = rfma(rho * cp, T, mix_sum<N, df64>(phi, X.rhoL));
        psi = df64(0);
        return true;
    }
    if (t < C.T_sol - tolT && Lv > 1e-5f * La + 1e-30f && rs > 1e-20f && cs > 1e-20f) {
        rho = mix_sum<N, df64>(phi, X.rho_s);
        cp = mix_sum<N, df64>(phi, X.cp_s);
        rhoH = rho * cp * T;
        psi = mix_sum<N, df64>(phi, X.drho);
        return true;
    }
    return false;
}

// t = 0 (Section 3 equilibria, Section 2 eq. H inverted): from phi_p, T, u build
// rho H, then f_l, T, rho, c_p by eq. H / eq. 2; populations at equilibrium with
// p = 0; mdot' = Q' = 0, psi' = psi, (phi_p u)' = phi_p u.
//
// The inputs are FP64 fields.  With everything in FP64 (and each of the 9 (N + 2) values
// converted on the same unit) the kernel was bound by the 2-lane FP64 pipe for every policy:
// 1676 us at 2048^2, N = 2, FP16 storage, against 95 us for its bytes.  The policies that
// store FP32 or less, and double words, now work in double words (an FP32 result is the
// double word rounded once): 196 us there.  FP64 decides the cells that eq. H does not decide
// by a margin.  What bounds it now is the number of its instructions (1720 per 32 cells at N = 3,
// 64 % of the issue slots).  Three blocks to an SM where 16-bit values are stored (a pass over 2048^2
// with 20 steps: 4619 us with two, 4578 with three); two for the wider types, whose three-phase kernel
// spills at 80 registers (1024^2, N = 3, FP32: 2284 us with two, 2316 with three).
// Populations come in opposite pairs, whose even and odd parts in c_i . u are shared.
template <int N, class Pr>
__global__ void __launch_bounds__(256, sizeof(typename Pr::TM) == 2 ? 3 : 2) init_kernel(const KParams P, const double* __restrict__ phi_in, const double* __restrict__ T_in,
                            const double* __restrict__ ux_in, const double* __restrict__ uy_in,
                            void* __restrict__ pop_base, typename Pr::TA* __restrict__ aux)
{
    using R = typename Pr::R;
    using TA = typename Pr::TA;
    using I = init_t<R>;
    using K = exact_t<I>;
    const long long S = P.S;
    const PopView<Pr> pop = pop_view<Pr>(P, pop_base);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < S; c += (long long)gridDim.x * blockDim.x) {
        double phd[N];
#pragma unroll
        for (int p = 0; p < N; ++p) phd[p] = LBM_LD(P, phi_in, p * S + c, N * S, 40);
        const double T0 = LBM_LD(P, T_in, c, S, 43);
        const I ux = ux_in ? init_input<I>(LBM_LD(P, ux_in, c, S, 41)) : I(0.0),
                uy = uy_in ? init_input<I>(LBM_LD(P, uy_in, c, S, 42)) : I(0.0);
        I phi[N], rhoH, T = init_input<I>(T0), rho, cp, psi;
#pragma unroll
        for (int p = 0; p < N; ++p) phi[p] = init_input<I>(phd[p]);
        bool decided = false;
        if constexpr (!std::is_same<I, double>::value) decided = init_macro_decided<N>(P, phi, T, rhoH, rho, cp, psi);
        if (!decided) {
            double rH, Tm, r, cpd, ps;
            init_macro<N>(P, phd, T0, rH, Tm, r, cpd, ps);
            rhoH = I(rH);
            T = I(Tm);
            rho = I(r);
            cp = I(cpd);
            psi = I(ps);
        }
        const I E = coef<I>(P).E_ref * T, Z = rho * cp * T;
        const I uu15 = K(1.5) * rfma(ux, ux, uy * uy);
        auto put = [&](auto kind, int s, int i, I v) {
            st_pop<Pr, decltype(kind)::value>(P, pop, s, i, c, init_value<R>(v), 44);
        };
        using F = std::integral_constant<int, KIND_F>;
        using G = std::integral_constant<int, KIND_G>;
        using H = std::integral_constant<int, KIND_H>;
        const I w0 = wgt_r<I>(0);
        put(F{}, 0, 0, -(w0 * rho * uu15));
        put(H{}, N + 1, 0, (rhoH - E) + w0 * (E - Z * uu15));
#pragma unroll
        for (int p = 0; p < N; ++p) put(G{}, 1 + p, 0, w0 * phi[p]);
        // opposite pairs (1, 3), (2, 4), (5, 7), (6, 8)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = k < 2 ? 1 + k : 3 + k, j = opp(i);
            const I w = wgt_r<I>(i);
            const I cu = i == 1 ? ux : i == 2 ? uy : i == 5 ? ux + uy : uy - ux;
            const I odd = K(3) * cu, even = rfma(K(4.5) * cu, cu, -uu15);
            const I sp = even + odd, sm = even - odd;
            const I wr = w * rho, wE = w * E, wZ = w * Z;
            put(F{}, 0, i, wr * sp);
            put(F{}, 0, j, wr * sm);
            put(H{}, N + 1, i, rfma(wZ, sp, wE));
            put(H{}, N + 1, j, rfma(wZ, sm, wE));
#pragma unroll
            for (int p = 0; p < N; ++p) {
                const I wp = w * phi[p];
                if constexpr (std::is_same<I, double>::value) {
                    put(G{}, 1 + p, i, rfma(wp, odd, wp));
                    put(G{}, 1 + p, j, rfma(-wp, odd, wp));
                } else {   // the product once: the same values
                    const I t = wp * odd;
                    put(G{}, 1 + p, i, t + wp);
                    put(G{}, 1 + p, j, wp - t);
                }
            }
        }
        LBM_ST(P, aux, aux_mdot() * S + c, P.aux_elems, 47, (TA)0.0);
        LBM_ST(P, aux, aux_Q() * S + c, P.aux_elems, 47, (TA)0.0);
        LBM_ST(P, aux, aux_psi() * S + c, P.aux_elems, 47, (TA)init_value<R>(psi));
#pragma unroll
        for (int p = 0; p < N; ++p) {
            LBM_ST(P, aux, aux_phiux(p) * S + c, P.aux_elems, 48, (TA)init_value<R>(phi[p] * ux));
            LBM_ST(P, aux, aux_phiuy(N, p) * S + c, P.aux_elems, 48, (TA)init_value<R>(phi[p] * uy));
        }
    }
}

// Diagnostics, pass 1: per-block partial sums (fixed order inside the block) in FP64
// of sum phi_p, sum f_s phi_p, max |sum_p phi_p - 1| and the count of non-finite cells,
// over the cells c0 .. c0 + cells - 1 (the whole lattice, or the own rows of a slab).
// partial[b * (2N + 2) + k]; pass 2 adds the blocks in index order.
template <int N, int NT, class Pr>
__global__ void __launch_bounds__(NT) diag_partial_kernel(const KParams P, const void* __restrict__ pop_base,
                                                          const typename Pr::TA* __restrict__ aux,
                                                          double* __restrict__ partial, long long c0,
                                                          long long cells)
{
    constexpr int K = 2 * N + 2;
    __shared__ double red[K][NT];
    const long long S = P.S;
    const PopView<Pr> pop = pop_view<Pr>(P, pop_base);
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    for (long long k = blockIdx.x * (long long)NT + threadIdx.x; k < cells; k += (long long)gridDim.x * NT) {
        const long long c = c0 + k;
        const double den = 1.0 - 0.5 * (double)LBM_LD(P, aux, aux_mdot() * S + c, P.aux_elems, 50);
        double phi[N], sum = 0.0;
#pragma unroll
        for (int p = 0; p < N; ++p) {
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < 9; ++i) s += (double)ld_pop<Pr, KIND_G>(P, pop, 1 + p, i, c, 51);
            phi[p] = s / den;
            sum += phi[p];
        }
        double sh = 0.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) sh += (double)ld_pop<Pr, KIND_H>(P, pop, N + 1, i, c, 52);
        double f0 = 0.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) f0 += (double)ld_pop<Pr, KIND_F>(P, pop, 0, i, c, 53);
        const double rhoH = fma(0.5, (double)LBM_LD(P, aux, aux_Q() * S + c, P.aux_elems, 54), sh);
        const Mix<N> m = mixture_core<N>(P, phi);
        double fl, T;
        enthalpy_map<N, false>(P, m, rhoH, fl, T);
        const double fs = 1.0 - fl;
        const bool bad = !isfinite(sum) || !isfinite(rhoH) || !isfinite(f0);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            acc[p] += phi[p];
            acc[N + p] += fs * phi[p];
        }
        acc[2 * N] = fmax(acc[2 * N], fabs(sum - 1.0));
        acc[2 * N + 1] += bad ? 1.0 : 0.0;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) red[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = NT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (k == 2 * N) red[k][threadIdx.x] = fmax(red[k][threadIdx.x], red[k][threadIdx.x + s]);
                else red[k][threadIdx.x] += red[k][threadIdx.x + s];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) partial[blockIdx.x * K + k] = red[k][0];
}

// Diagnostics, pass 2: one warp adds the block partials in a fixed order
// (lane-strided, then a shuffle tree), so the result does not depend on timing.
template <int N>
__global__ void diag_final_kernel(const double* __restrict__ partial, int nblocks, double* __restrict__ out)
{
    constexpr int K = 2 * N + 2;
    const int lane = threadIdx.x;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double v = 0.0;
        for (int b = lane; b < nblocks; b += 32) {
            const double w = partial[b * K + k];
            v = (k == 2 * N) ? fmax(v, w) : v + w;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double o = __shfl_down_sync(0xffffffffu, v, off);
            v = (k == 2 * N) ? fmax(v, o) : v + o;
        }
        if (lane == 0) out[k] = v;
    }
}

}  // namespace lbm
