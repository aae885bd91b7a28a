// lbm_aux.cuh -- initial state and diagnostics kernels, generic over the precision
// policy (lbm_prec.cuh).  The diagnostics evaluate in FP64, the initial state in FP64 or in
// double words that round as FP64 does; both (de)quantise at the load / store.
#pragma once

#include "lbm_device.cuh"
#include "lbm_prec.cuh"
#include "lbm_step.cuh"

namespace lbm {

// Arithmetic type of the initial state's equilibria: FP64 (d1: rounded as written, so that every kernel
// forms the same bits) for the FP64 policy and for double words,
// whose 48 bits would show the rounding of a double-word chain (measured against FP64 over the film,
// the drops and the pools: 1e-14 of the largest value, 1e-15 with FP64 and one rounding).  Policies that store
// FP32 or less form it in double words on the FP32 pipes where that gives what FP64 gives.
template <class R>
using init_t = typename std::conditional<std::is_same<R, float>::value, df64, d1>::type;

// An FP64 input of the initial state as the arithmetic type.  For double words: the pair of
// df64(double) (x rounded to FP32, and the rest rounded to FP32; of two equally near x the one
// further from zero), put together with integer instructions.  The four FP64 instructions of
// the conversion occupy a scheduler's share of the FP64 unit for 64 cycles each: the N + 3
// inputs held that unit for 43 of the kernel's 78 us at 1024^2, N = 3, FP16 storage, 64 us with
// integers (89 since init_cell tests the roundings).  Only values so small or so large that a part
// would leave FP32's normal range are converted there.
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

// Whether an input is so small (and not 0) that a product with it could leave the range in which a
// double word keeps all its bits.
__device__ __forceinline__ bool init_tiny(df64 x, float limit) { return fabsf(x.hi) < limit && x.hi != 0.0f; }

// The leading part of a value's magnitude, for the error bounds below.
__device__ __forceinline__ float init_mag(df64 v) { return fabsf(v.hi); }
__device__ __forceinline__ float init_mag(d1) { return 0.0f; }

// eq. H inverted for one cell (the map, and what follows from it), FP64: rho H, T, rho, c_p, psi.
template <int N>
__device__ __forceinline__ void init_macro(const KParams& P, const double (&phi)[N], double T_in, double& rhoH, double& T,
                                           double& rho, double& cp, double& psi)
{
    const Mix<N> m = mixture_core<N>(P, phi);
    rhoH = inverse_map<N>(P, m, T_in);
    double fl;
    enthalpy_map<N, true>(P, m, rhoH, fl, T);
    const double fs = __dsub_rn(1.0, fl);
    rho = __fma_rn(fs, m.rs, __dmul_rn(fl, m.rl));
    cp = __fma_rn(fs, m.cs, __dmul_rn(fl, m.cl));
    psi = __dmul_rn(fs, m.dr);
}

// The same in double words, for a cell whose phase the input temperature decides with margin
// (returns false for any other: the FP64 form is then asked).  Above the liquidus the cell is
// liquid whatever its latent heat; below the solidus it is solid where it holds
// phase-changing material.  Either way the map returns the temperature it was given.  The
// screen runs on FP32 values of the inputs; its margin of 1e-5 of the magnitudes is 25
// times their rounding.  A cell with negative fractions beyond 1/16 of a sum is not decided, so
// rho and c_p keep the relative error of a sum of positive terms.  La, pa: sum |phi_p| rho_l^p L_p,
// sum |phi_p (rho_s^p - rho_l^p)|.
template <int N>
__device__ __forceinline__ bool init_macro_decided(const KParams& P, const df64 (&phi)[N], df64 T, df64& rhoH, df64& rho,
                                                   df64& cp, df64& psi, float& La, float& pa)
{
    const Coef<float>& C = P.f;
    const Coef<df64>& X = P.x;
    const float t = T.hi, tolT = 1e-5f * (fabsf(t) + fabsf(C.T_sol) + fabsf(C.T_liq)) + 1e-30f;
    const bool warm = t > C.T_liq + tolT;
    if (!warm && !(t < C.T_sol - tolT)) return false;
    float rs = 0.0f, rl = 0.0f, cs = 0.0f, cl = 0.0f, Lv = 0.0f, ra = 0.0f, ca = 0.0f;
    La = pa = 0.0f;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const float ph = phi[p].hi, ap = fabsf(ph);
        rs = fmaf(ph, C.rho_s[p], rs);
        rl = fmaf(ph, C.rho_l[p], rl);
        cs = fmaf(ph, C.cp_s[p], cs);
        cl = fmaf(ph, C.cp_l[p], cl);
        Lv = fmaf(ph, C.rhoL[p], Lv);
        La = fmaf(ap, C.rhoL[p], La);
        ra = fmaf(ap, warm ? C.rho_l[p] : C.rho_s[p], ra);
        ca = fmaf(ap, warm ? C.cp_l[p] : C.cp_s[p], ca);
        if (!warm) pa = fmaf(ap, fabsf(C.drho[p]), pa);
    }
    if (warm) {
        if (!(rl > 1e-20f && cl > 1e-20f && ra <= 1.0625f * rl && ca <= 1.0625f * cl)) return false;
        const float rcl = rl * cl, As = rs * cs * C.T_sol, Al = fmaf(rcl, C.T_liq, Lv);
        const float h = fmaf(rcl, t - C.T_liq, Al);
        const float tol = 1e-5f * (fabsf(As) + fabsf(rcl * C.T_liq) + fabsf(rcl * t) + La) + 1e-30f;
        if (!(h > As + tol)) return false;
        rho = mix_sum<N, df64>(phi, X.rho_l);
        cp = mix_sum<N, df64>(phi, X.cp_l);
        rhoH = rfma(rho * cp, T, mix_sum<N, df64>(phi, X.rhoL));
        psi = df64(0);
        return true;
    }
    if (!(Lv > 1e-5f * La + 1e-30f && rs > 1e-20f && cs > 1e-20f && ra <= 1.0625f * rs && ca <= 1.0625f * cs)) return false;
    rho = mix_sum<N, df64>(phi, X.rho_s);
    cp = mix_sum<N, df64>(phi, X.cp_s);
    rhoH = rho * cp * T;
    psi = mix_sum<N, df64>(phi, X.drho);
    return true;
}

// Index of a value of the initial state in a cell's mask: population i of species s, then psi', then
// (phi_p u)' x and y.
__host__ __device__ constexpr int init_pop(int s, int i) { return 9 * s + i; }
__host__ __device__ constexpr int init_psi(int N) { return 9 * (N + 2); }
__host__ __device__ constexpr int init_lag(int N, int q) { return 9 * (N + 2) + 1 + q; }
constexpr unsigned long long INIT_ALL = ~0ull;   // (N = 4 has 63 values)

// The initial state of cell c in arithmetic of type I.  Where I is df64, returns the values that might
// round to another FP32 number than FP64's would, as a mask: what was stored for them is to be overwritten.
//
// Of a value v = hi + lo that is within d of the exact one, both v - d and v + d are rounded: where
// they give the same FP32 number, so does anything between, FP64's value (which is closer) among it.
// d is a sum of the error bounds of the operations: in units of u2 = 2^-48, a product of normalised
// pairs 5, of pairs with an unnormalised factor 11, a sum 9 (|x| + |y|), inputs and coefficients 1/2.
// So rho and c_p 42 (four phases), Z = rho c_p T 100, E 6, c_i . u 9 U with U = |u_x| + |u_y|, and
//   s = even +- odd of a direction      62 U + 278 U^2
//   f_i = w rho s                       |w rho| (239 U + 632 U^2)
//   h_i = w Z s + w E                   |w Z| (458 U + 1070 U^2) + 27 |w E|
//   h_0                                 128 (|Z| + |E| + |rho H|) + 64 sum |phi_p| rho_l^p L_p
//   g_i = w phi_p (1 + odd)             |w phi_p| (15 + 113 U)
//   f_0 80, phi_p w_0 and phi_p u 6, psi 42 of their magnitudes
// (the bounds below are these, rounded up to powers of two).  About one value in 10^5 fails the test.
template <int N, class Pr, class I>
__device__ __forceinline__ unsigned long long init_cell(const KParams& P, const PopView<Pr>& pop, typename Pr::TA* __restrict__ aux,
                                                        long long c, const double* __restrict__ phi_in,
                                                        const double* __restrict__ T_in, const double* __restrict__ ux_in,
                                                        const double* __restrict__ uy_in)
{
    using R = typename Pr::R;
    using TA = typename Pr::TA;
    using K = exact_t<I>;
    constexpr bool DW = std::is_same<I, df64>::value;
    const long long S = P.S;
    double phd[N];
#pragma unroll
    for (int p = 0; p < N; ++p) phd[p] = LBM_LD(P, phi_in, p * S + c, N * S, 40);
    const double T0 = LBM_LD(P, T_in, c, S, 43);
    const I ux = ux_in ? init_input<I>(LBM_LD(P, ux_in, c, S, 41)) : I(0.0),
            uy = uy_in ? init_input<I>(LBM_LD(P, uy_in, c, S, 42)) : I(0.0);
    using KW = const_t<I>;   // type of the weights and coefficients
    I phi[N], rhoH, T = init_input<I>(T0), rho, cp, psi;
    float La = 0.0f, pa = 0.0f;
#pragma unroll
    for (int p = 0; p < N; ++p) phi[p] = init_input<I>(phd[p]);
    unsigned long long mask = 0;
    bool decided = false;
    if constexpr (DW) {
        if (init_tiny(ux, 0x1p-40f) || init_tiny(uy, 0x1p-40f) || init_tiny(T, 0x1p-60f)) return INIT_ALL;
        // a tiny fraction is nothing to the sums over the phases, but its own values take FP64
#pragma unroll
        for (int p = 0; p < N; ++p)
            if (init_tiny(phi[p], 0x1p-60f))
                mask |= 0x1ffull << init_pop(1 + p, 0) | 1ull << init_lag(N, p) | 1ull << init_lag(N, N + p);
        decided = init_macro_decided<N>(P, phi, T, rhoH, rho, cp, psi, La, pa);
    }
    if (!decided) {
        double rH, Tm, r, cpd, ps;
        init_macro<N>(P, phd, T0, rH, Tm, r, cpd, ps);
        rhoH = I(rH);
        T = I(Tm);
        rho = I(r);
        cp = I(cpd);
        psi = I(ps);
        pa = init_mag(psi);
    }
    // value k of the cell as the policy's arithmetic type, rounded once
    auto value = [&](int k, I v, float d) {
        if constexpr (DW) {
            const float a = __fadd_rn(v.hi, __fadd_rn(v.lo, d)), b = __fadd_rn(v.hi, __fsub_rn(v.lo, d));
            if (!(a == b)) mask |= 1ull << k;
            return a;
        } else if constexpr (std::is_same<R, df64>::value) {
            return init_input<df64>(v.v);
        } else {
            return (R)v.v;
        }
    };
    const I E = T * coef<KW>(P).E_ref, Z = rho * cp * T;
    const I uu15 = rfma(ux, ux, uy * uy) * K(1.5);
    const float U = init_mag(ux) + init_mag(uy), UU = fmaf(2.5f * U, U, U);
    auto put = [&](auto kind, int s, int i, I v, float d) {
        st_pop<Pr, decltype(kind)::value>(P, pop, s, i, c, value(init_pop(s, i), v, d), 44);
    };
    using F = std::integral_constant<int, KIND_F>;
    using G = std::integral_constant<int, KIND_G>;
    using H = std::integral_constant<int, KIND_H>;
    const I w0 = I(wgt_r<KW>(0)), f0 = -(w0 * rho * uu15);
    put(F{}, 0, 0, f0, init_mag(f0) * 0x1p-41f);
    put(H{}, N + 1, 0, rfma(w0, rfma(-Z, uu15, E), rhoH - E), (init_mag(Z) + init_mag(E) + init_mag(rhoH) + La) * 0x1p-41f);
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const I g0 = w0 * phi[p];
        put(G{}, 1 + p, 0, g0, init_mag(g0) * 0x1p-45f);
    }
    // opposite pairs (1, 3), (2, 4), (5, 7), (6, 8)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = k < 2 ? 1 + k : 3 + k, j = opp(i);
        const I w = I(wgt_r<KW>(i));
        const I cu = i == 1 ? ux : i == 2 ? uy : i == 5 ? ux + uy : uy - ux;
        const I odd = cu * K(3), even = rfma(cu * K(4.5), cu, -uu15);
        const I sp = even + odd, sm = even - odd;
        const I wr = w * rho, wE = w * E, wZ = w * Z;
        const float df = init_mag(wr) * (UU * 0x1p-40f), dh = fmaf(init_mag(wZ), UU * 0x1p-39f, init_mag(wE) * 0x1p-43f);
        put(F{}, 0, i, wr * sp, df);
        put(F{}, 0, j, wr * sm, df);
        put(H{}, N + 1, i, rfma(wZ, sp, wE), dh);
        put(H{}, N + 1, j, rfma(wZ, sm, wE), dh);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            const I wp = w * phi[p];
            const float dg = init_mag(wp) * fmaf(U, 0x1p-41f, 0x1p-44f);
            if constexpr (DW) {   // the product once: the same values
                const I t = wp * odd;
                put(G{}, 1 + p, i, t + wp, dg);
                put(G{}, 1 + p, j, wp - t, dg);
            } else {
                put(G{}, 1 + p, i, rfma(wp, odd, wp), dg);
                put(G{}, 1 + p, j, rfma(-wp, odd, wp), dg);
            }
        }
    }
    LBM_ST(P, aux, aux_mdot() * S + c, P.aux_elems, 47, (TA)0.0);
    LBM_ST(P, aux, aux_Q() * S + c, P.aux_elems, 47, (TA)0.0);
    LBM_ST(P, aux, aux_psi() * S + c, P.aux_elems, 47, (TA)value(init_psi(N), psi, pa * 0x1p-42f));
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const I a = phi[p] * ux, b = phi[p] * uy;
        LBM_ST(P, aux, aux_phiux(p) * S + c, P.aux_elems, 48, (TA)value(init_lag(N, p), a, init_mag(a) * 0x1p-45f));
        LBM_ST(P, aux, aux_phiuy(N, p) * S + c, P.aux_elems, 48, (TA)value(init_lag(N, N + p), b, init_mag(b) * 0x1p-45f));
    }
    return mask;
}

// The values of a mask in FP64, one after another: a warp with a cell that needs any waits for the FP64
// unit, 64 cycles an instruction, so a value's own operations count (512^2, FP16 storage: 23 us, and 27 when
// the whole cell, some 350 operations, was formed again).  Out of line: its registers do not weigh on the
// cells that do without.
template <int N, class Pr>
__device__ __noinline__ void init_redo(const KParams& P, PopView<Pr> pop, typename Pr::TA* aux, long long c, const double* phi_in,
                                       const double* T_in, const double* ux_in, const double* uy_in, unsigned long long mask)
{
    if (mask == INIT_ALL) {
        init_cell<N, Pr, d1>(P, pop, aux, c, phi_in, T_in, ux_in, uy_in);
        return;
    }
    using TA = typename Pr::TA;
    const long long S = P.S;
    const d1 ux = ux_in ? LBM_LD(P, ux_in, c, S, 41) : 0.0, uy = uy_in ? LBM_LD(P, uy_in, c, S, 42) : 0.0;
    auto phi_of = [&](int p) { return d1(LBM_LD(P, phi_in, p * S + c, N * S, 40)); };
    double rhoH = 0.0, T = 0.0, rho = 0.0, cp = 0.0, psi = 0.0;
    const unsigned long long macro = 0x1ffull << init_pop(0, 0) | 0x1ffull << init_pop(N + 1, 0) | 1ull << init_psi(N);
    if (mask & macro) {
        double phi[N];
        for (int p = 0; p < N; ++p) phi[p] = phi_of(p).v;
        init_macro<N>(P, phi, LBM_LD(P, T_in, c, S, 43), rhoH, T, rho, cp, psi);
    }
    const d1 uu15 = rfma(ux, ux, uy * uy) * 1.5;
    const d1 E = d1(T) * P.d.E_ref, Z = d1(rho) * d1(cp) * d1(T);
    for (; mask; mask &= mask - 1) {
        const int k = __ffsll((long long)mask) - 1;
        if (k == init_psi(N)) {
            LBM_ST(P, aux, aux_psi() * S + c, P.aux_elems, 47, (TA)psi);
            continue;
        }
        if (k > init_psi(N)) {
            const int q = k - init_lag(N, 0);
            const d1 v = q < N ? phi_of(q) * ux : phi_of(q - N) * uy;
            LBM_ST(P, aux, (q < N ? aux_phiux(q) : aux_phiuy(N, q - N)) * S + c, P.aux_elems, 48, (TA)v.v);
            continue;
        }
        // as init_cell forms them: cu of the first direction of a pair, the second with the other sign of the odd part
        const int s = k / 9, i = k - 9 * s, j = i == 3 || i == 4 || i == 7 || i == 8 ? opp(i) : i;
        const d1 w = d1(wgt(i)), cu = j == 1 ? ux : j == 2 ? uy : j == 5 ? ux + uy : uy - ux;
        const d1 odd = cu * 3.0, even = rfma(cu * 4.5, cu, -uu15), sij = i == j ? even + odd : even - odd;
        if (s == 0) {
            st_pop<Pr, KIND_F>(P, pop, s, i, c, (float)(i == 0 ? -(w * d1(rho) * uu15) : w * d1(rho) * sij).v, 44);
        } else if (s == N + 1) {
            st_pop<Pr, KIND_H>(P, pop, s, i, c,
                               (float)(i == 0 ? rfma(w, rfma(-Z, uu15, E), d1(rhoH) - E) : rfma(w * Z, sij, w * E)).v, 44);
        } else {
            const d1 wp = w * phi_of(s - 1);
            st_pop<Pr, KIND_G>(P, pop, s, i, c, (float)(i == 0 ? wp : rfma(i == j ? wp : -wp, odd, wp)).v, 44);
        }
    }
}

// t = 0 (Section 3 equilibria, Section 2 eq. H inverted): from phi_p, T, u build
// rho H, then f_l, T, rho, c_p by eq. H / eq. 2; populations at equilibrium with
// p = 0; mdot' = Q' = 0, psi' = psi, (phi_p u)' = phi_p u.
//
// The inputs are FP64 fields.  With everything in FP64 (and each of the 9 (N + 2) values
// converted on the same unit) the kernel was bound by the 2-lane FP64 pipe for every policy:
// 1676 us at 2048^2, N = 2, FP16 storage, against 95 us for its bytes.  The policies that
// store FP32 or less work in double words (251 us there): their stored values are FP64's rounded to
// FP32 all the same, since the values whose rounding double words do not settle are formed again in
// FP64, as are macroscopic values that eq. H does not decide by a margin.  What bounds it is the
// number of its instructions, the test of the roundings among them (197 us without it).  Double
// words themselves take FP64: 1315 us there, the FP64 policy 945.  Three blocks to an SM where
// 16-bit values are stored (2048^2 251 us, with two 291; 1024^2, N = 3 89 and 95); two for the wider
// types, whose three-phase kernel spills at 80 registers.
// Populations come in opposite pairs, whose even and odd parts in c_i . u are shared.
template <int N, class Pr>
__global__ void __launch_bounds__(256, sizeof(typename Pr::TM) == 2 ? 3 : 2)
init_kernel(const __grid_constant__ KParams P, const double* __restrict__ phi_in, const double* __restrict__ T_in,
            const double* __restrict__ ux_in, const double* __restrict__ uy_in, void* __restrict__ pop_base,
            typename Pr::TA* __restrict__ aux)
{
    using I = init_t<typename Pr::R>;
    const long long S = P.S;
    const PopView<Pr> pop = pop_view<Pr>(P, pop_base);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < S; c += (long long)gridDim.x * blockDim.x) {
        const unsigned long long mask = init_cell<N, Pr, I>(P, pop, aux, c, phi_in, T_in, ux_in, uy_in);
        if constexpr (std::is_same<I, df64>::value)
            if (mask) init_redo<N, Pr>(P, pop, aux, c, phi_in, T_in, ux_in, uy_in, mask);
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
