// lbm_cell.cuh -- the arithmetic of one lattice update (arXiv 2603.22902, Sections 2 and 3),
// from the moments of the cell to its post-collision populations and lagged values, written
// once for FP64, double words and FP32 (lbm_vals.cuh); 16-bit storage has a form of its own
// (lbm_cell16.cuh).  The kernels supply the inputs and take the outputs through an Io object.
//
// What bounds it: the FP64 policy the number of its FP64 instructions (a warp instruction holds
// the SM's 2-lane unit for 16 cycles), double words and the FP32-arithmetic policies the number
// of instructions issued.  So the algebra is arranged for few operations:
//   * a cell that eq. H calls liquid or solid uses that state's sums of eq. 2 alone, and
//     rho c_p T = rho H - Lv or rho H, without the map's division;
//   * 1/rho, 1/tau_f, 1/tau_h and 1/(rho c_p) come from one reciprocal (three in double words);
//   * stencils are left as 12 grad and 6 lap (their differences along the diagonals are shared);
//     the factors go into coefficients;
//   * S - 3/2 tr Lambda = -3 u.F, since Lambda = uF + Fu + (S/3) I: S drops out of F_0 and of
//     the isotropic part of the flow source;
//   * opposite directions share their even and odd parts in c_i, which carry the weight of the
//     axis directions (1/9) from the start.
// Measured at N = 2, 512 x 512 (ncu, one step): FP64 487 -> 365 FP64 instructions per cell and
// 254 -> 193 us; double words 5600 -> 4740 instructions per cell, 69 -> 62 us.  Against the scheme in long double the FP64 fields
// are 2 to 15 times closer than with one product per weight and direction (the rest direction now
// takes what the others leave, so that sum_i g_i and sum_i h_i do not drift with the rounding of
// the weights).  Double words are as close as with the plain form: after 20 000 steps of the drop
// (64 x 48) and the film (16 x 64), against the scheme in 80 bits, phi 3.1e-11 and 1.5e-11 (plain form
// 4.8e-11 and 1.8e-11), T 1.6e-10 and 7.8e-13 (4.2e-10, 7.5e-13), the front 3.7e-10 and 6.1e-10 lattice units
// (5.3e-10, 7.8e-10).  On the 512 x 512 drop rounding alone spreads the front: over 48 runs from initial phi that
// differ by 1e-14 it is off by 9.2e-10 in the median and by more than 1e-8 in 7 (plain form 1.0e-9, 6 of 48).
#pragma once

#include "lbm_device.cuh"
#include "lbm_prec.cuh"

namespace lbm {

// A D2Q9 weight as a constant of arithmetic of type V.
template <class V>
__device__ __forceinline__ const_t<V> wgt_v(int i)
{
    return wgt_r<const_t<V>>(i);
}

template <class V>
__device__ __forceinline__ constexpr const_t<V> cst(double c)
{
    return const_t<V>(c);
}

template <class V>
__device__ __forceinline__ bool any_nonzero(V a)
{
    return !(a == V(0.0f));
}
template <class V>
__device__ __forceinline__ bool all_equal(V a, float b)
{
    return a == V(b);
}

// Post-collision populations q_i = (1 - omega) f_i + even_i +- odd_i of the eight moving
// directions.  ex, ey: even parts of the axis directions; e5, e6: of the diagonals (1, 1) and
// (-1, 1); odd parts along x and y: ca tx, ca ty.  All parts carry the axis weight 1/9, and the
// diagonals take a quarter of it.
template <class V, class CA>
__device__ __forceinline__ void collide_pairs(V om1, const V (&f)[9], V ex, V ey, V e5, V e6, V tx, V ty, CA ca, V (&q)[9])
{
    const auto quarter = exact_t<V>(0.25);
    if constexpr (std::is_same<V, df64>::value) {
        // a shared product and a sum are fewer instructions than two multiply-adds
        const V ax = tx * ca, ay = ty * ca, o5 = (ax + ay) * quarter, o6 = (ay - ax) * quarter;
        e5 = e5 * quarter;
        e6 = e6 * quarter;
        q[1] = rfma(om1, f[1], ex + ax);
        q[3] = rfma(om1, f[3], ex - ax);
        q[2] = rfma(om1, f[2], ey + ay);
        q[4] = rfma(om1, f[4], ey - ay);
        q[5] = rfma(om1, f[5], e5 + o5);
        q[7] = rfma(om1, f[7], e5 - o5);
        q[6] = rfma(om1, f[6], e6 + o6);
        q[8] = rfma(om1, f[8], e6 - o6);
        return;
    }
    const V mx = -tx, my = -ty;
    q[1] = rfma(om1, f[1], rfma(tx, ca, ex));
    q[3] = rfma(om1, f[3], rfma(mx, ca, ex));
    q[2] = rfma(om1, f[2], rfma(ty, ca, ey));
    q[4] = rfma(om1, f[4], rfma(my, ca, ey));
    const V o5 = (tx + ty) * (ca * quarter), o6 = (ty - tx) * (ca * quarter);
    q[5] = rfma(om1, f[5], rfma(e5, quarter, o5));
    q[7] = rfma(om1, f[7], rfma(e5, quarter, -o5));
    q[6] = rfma(om1, f[6], rfma(e6, quarter, o6));
    q[8] = rfma(om1, f[8], rfma(e6, quarter, -o6));
}
// The same with ca = 1 and one even part e for all directions.
template <class V>
__device__ __forceinline__ void collide_pairs(V om1, const V (&f)[9], V e, V ax, V ay, V (&q)[9])
{
    q[1] = rfma(om1, f[1], e + ax);
    q[3] = rfma(om1, f[3], e - ax);
    q[2] = rfma(om1, f[2], e + ay);
    q[4] = rfma(om1, f[4], e - ay);
    const auto quarter = exact_t<V>(0.25);
    const V o5 = (ax + ay) * quarter, o6 = (ay - ax) * quarter;
    if constexpr (std::is_same<V, df64>::value) {
        e = e * quarter;
        q[5] = rfma(om1, f[5], e + o5);
        q[7] = rfma(om1, f[7], e - o5);
        q[6] = rfma(om1, f[6], e + o6);
        q[8] = rfma(om1, f[8], e - o6);
    } else {
        q[5] = rfma(om1, f[5], rfma(e, quarter, o5));
        q[7] = rfma(om1, f[7], rfma(e, quarter, -o5));
        q[6] = rfma(om1, f[6], rfma(e, quarter, o6));
        q[8] = rfma(om1, f[8], rfma(e, quarter, -o6));
    }
}

// sum_p phi_p a_p.
template <int N, class V, class C>
__device__ __forceinline__ V phi_sum(const V (&phi)[N], const C (&a)[MAXN])
{
    V v = phi[0] * a[0];
#pragma unroll
    for (int p = 1; p < N; ++p) v = rfma(phi[p], a[p], v);
    return v;
}

// The FP32 screen of eq. H for one cell: 1 (liquid) where rho H lies above the liquidus value Al (and
// the solidus value As), 0 (solid) where phase-changing material is present (Lv > 0) and rho H lies
// below As, -1 where it does not decide (the mushy band, values near a threshold, phase-changing
// material below FP32 range or whose fractions cancel, values that are not finite).  Al, As and Lv are
// sums over the phases, and the tails of absent phases have either sign: the margin is 1e-5 of the
// sums of magnitudes, which is at least ten times the rounding of Al and As from leading parts, and Lv
// counts as positive or negative only beyond 1e-5 of its own.  With T_sol = T_liq = 0 Al is Lv and As is 0.
template <int N, class V>
__device__ __forceinline__ int eqh_screen(const KParams& P, const V (&phi)[N], V rhoH)
{
    const Coef<float>& C = P.f;
    float ph[N];
#pragma unroll
    for (int p = 0; p < N; ++p) ph[p] = lead(phi[p]);
    const float h = lead(rhoH);
    float Lv = __fmul_rn(ph[0], C.rhoL[0]), La = fabsf(Lv);
#pragma unroll
    for (int p = 1; p < N; ++p) {
        Lv = __fmaf_rn(ph[p], C.rhoL[p], Lv);
        La = __fmaf_rn(fabsf(ph[p]), C.rhoL[p], La);
    }
    float Al = Lv, As = 0.0f, mag = __fadd_rn(La, fabsf(h));
    const bool shifted = C.T_liq != 0.0f || C.T_sol != 0.0f;
    if (shifted) {
        float rl = 0.0f, cl = 0.0f, rs = 0.0f, cs = 0.0f, rla = 0.0f, cla = 0.0f, rsa = 0.0f, csa = 0.0f;
#pragma unroll
        for (int p = 0; p < N; ++p) {
            const float a = fabsf(ph[p]);
            rl = __fmaf_rn(ph[p], C.rho_l[p], rl);
            cl = __fmaf_rn(ph[p], C.cp_l[p], cl);
            rs = __fmaf_rn(ph[p], C.rho_s[p], rs);
            cs = __fmaf_rn(ph[p], C.cp_s[p], cs);
            rla = __fmaf_rn(a, C.rho_l[p], rla);
            cla = __fmaf_rn(a, C.cp_l[p], cla);
            rsa = __fmaf_rn(a, C.rho_s[p], rsa);
            csa = __fmaf_rn(a, C.cp_s[p], csa);
        }
        Al = __fmaf_rn(__fmul_rn(rl, cl), C.T_liq, Lv);
        As = __fmul_rn(__fmul_rn(rs, cs), C.T_sol);
        mag = __fmaf_rn(__fmul_rn(rla, cla), fabsf(C.T_liq), mag);
        mag = __fmaf_rn(__fmul_rn(rsa, csa), fabsf(C.T_sol), mag);
    }
    const float tol = __fmaf_rn(1e-5f, mag, 1e-30f);
    // without phase-changing material a cell is liquid whatever As; with it and As = 0 (not shifted), above Al is above As
    if (h > __fadd_rn(Al, tol) && (!shifted || h > __fadd_rn(As, tol) || Lv < __fmul_rn(-1e-5f, La))) return 1;
    // a double's leading part is 0 below 2^-126
    const float none = std::is_same<V, d1>::value ? 1e-30f : 0.0f;
    if (Lv > __fmaf_rn(1e-5f, La, none) && h < __fsub_rn(As, tol)) return 0;
    return -1;
}

// eq. H for one cell: the liquid fraction, as the FP64 map gives it (the map itself runs only where
// the screen does not decide).
template <int N, class V>
__device__ __forceinline__ V liquid_fraction(const KParams& P, const V (&phi)[N], V rhoH)
{
    const int sure = eqh_screen<N>(P, phi, rhoH);
    if (sure > 0) return V(1.0f);
    if (sure == 0) return V(0.0f);
    double phd[N], fl, T;
#pragma unroll
    for (int p = 0; p < N; ++p) phd[p] = (double)phi[p];
    const Mix<N> m = mixture_map<N>(P, phd);
    enthalpy_map<N, false>(P, m, (double)rhoH, fl, T);
    return V(const_t<V>(fl));
}

// phi_p and rho H of a cell from its populations and lagged mdot', Q' (Section 3, recovery of
// phi_p and H).  1 - mdot'/2 divides nothing where mdot' = 0 (away from the front).
template <int N, class V, class G, class H>
__device__ __forceinline__ void moments(const KParams& P, V mdm, V Qm, G&& g, H&& h, V (&phi)[N], V& rhoH)
{
    using K = exact_t<V>;
    auto sum = [](auto&& q) {
        const V a = (q(1) + q(3)) + (q(2) + q(4)), d = (q(5) + q(7)) + (q(6) + q(8));
        return q(0) + (a + d);
    };
#pragma unroll
    for (int p = 0; p < N; ++p) phi[p] = sum([&](int i) { return g(p, i); });
    if (any_nonzero(mdm)) {
        const V iden = rinv(rfma(mdm, K(-0.5), V(K(1))));
#pragma unroll
        for (int p = 0; p < N; ++p) phi[p] = phi[p] * iden;
    }
    rhoH = rfma(Qm, K(0.5), sum([&](int i) { return h(i); }));
}

// The mixture of eq. 2 in one cell.
template <class V>
struct Mixture {
    V rho, mu, lam, cp, psi, chi;
    V Zn, T0;   // T = Zn / (rho c_p) + T0
};

// rho and psi of a cell (all that its neighbours need besides phi_p).
template <int N, class V>
__device__ __forceinline__ void mix_rho_psi(const KParams& P, const V (&phi)[N], V fl, V& rho, V& psi)
{
    const auto& C = coef<const_t<V>>(P);
    if (all_equal(fl, 1.0f)) {
        rho = phi_sum<N>(phi, C.rho_l);
        psi = V(0.0f);
    } else {
        const V fs = V(1.0f) - fl;
        rho = rfma(fs, phi_sum<N>(phi, C.rho_s), fl * phi_sum<N>(phi, C.rho_l));
        psi = fs * phi_sum<N>(phi, C.drho);
    }
}

// rho H - sum_p phi_p rho_l^p L_p.
template <int N, class V, class C>
__device__ __forceinline__ V liquid_sensible(const V (&phi)[N], V rhoH, const C (&rhoL)[MAXN])
{
    V z = rhoH;
#pragma unroll
    for (int p = 0; p < N; ++p) z = rfma(-phi[p], rhoL[p], z);
    return z;
}

template <int N, class V>
__device__ __forceinline__ Mixture<V> mixture_of(const KParams& P, const V (&phi)[N], V rhoH, V fl)
{
    const auto& C = coef<const_t<V>>(P);
    Mixture<V> m;
    const V zero = V(0.0f);
    if (all_equal(fl, 1.0f)) {
        m.rho = phi_sum<N>(phi, C.rho_l);
        m.mu = phi_sum<N>(phi, C.mu_l);
        m.lam = phi_sum<N>(phi, C.lam_l);
        m.cp = phi_sum<N>(phi, C.cp_l);
        m.psi = m.chi = m.T0 = zero;
        m.Zn = liquid_sensible<N>(phi, rhoH, C.rhoL);
    } else if (all_equal(fl, 0.0f)) {
        m.rho = phi_sum<N>(phi, C.rho_s);
        m.mu = phi_sum<N>(phi, C.mu_s);
        m.lam = phi_sum<N>(phi, C.lam_s);
        m.cp = phi_sum<N>(phi, C.cp_s);
        m.psi = phi_sum<N>(phi, C.drho);
        m.chi = phi_sum<N>(phi, C.pcm);
        m.T0 = zero;
        m.Zn = rhoH;
    } else {
        const V fs = V(1.0f) - fl;
        m.rho = rfma(fs, phi_sum<N>(phi, C.rho_s), fl * phi_sum<N>(phi, C.rho_l));
        m.mu = rfma(fs, phi_sum<N>(phi, C.mu_s), fl * phi_sum<N>(phi, C.mu_l));
        m.lam = rfma(fs, phi_sum<N>(phi, C.lam_s), fl * phi_sum<N>(phi, C.lam_l));
        m.cp = rfma(fs, phi_sum<N>(phi, C.cp_s), fl * phi_sum<N>(phi, C.cp_l));
        m.psi = fs * phi_sum<N>(phi, C.drho);
        m.chi = fs * phi_sum<N>(phi, C.pcm);
        m.Zn = zero;
        m.T0 = rfma(fl, C.T_liq - C.T_sol, V(C.T_sol));
    }
    return m;
}

// 12 grad a and 6 lap a (isotropic 9-point stencils) from the nine values around a cell.
template <class V>
__device__ __forceinline__ void grad12(V e, V w, V n, V s, V ne, V nw, V se, V sw, V& gx, V& gy)
{
    using K = exact_t<V>;
    const V d1 = ne - sw, d2 = nw - se;
    gx = rfma(e - w, K(4), d1 - d2);
    gy = rfma(n - s, K(4), d1 + d2);
}
template <class V>
__device__ __forceinline__ V lap6(V c, V e, V w, V n, V s, V ne, V nw, V se, V sw)
{
    using K = exact_t<V>;
    return rfma(c, K(-20), rfma((e + w) + (n + s), K(4), (ne + sw) + (nw + se)));
}

// a / |G| for the pairwise normal n_pq = G / |G| weighted by a, or 0 where the guards hold:
// phi_p + phi_q <= 1e-12, |grad phi_pq| below the policy's absolute threshold (|grad phi_pq| =
// |G| / s^2; G is 12 times itself here), or below NGUARD times its own scale (ref).
template <class Pr, class V>
__device__ __forceinline__ V normal_weight(V s, V G2, V ref, V a)
{
    bool ok = s > V(const_t<V>(1e-12));
    if (ok) {
        const V s2 = s * s;
        ok = G2 > (s2 * s2) * const_t<V>(144.0 * Pr::NABS2);
        if constexpr (Pr::NGUARD > 0.0f) ok = ok && G2 > ref * const_t<V>(Pr::NGUARD * Pr::NGUARD);
    }
    V r = V(0.0f);
    if (ok) r = a * rrsqrt(G2);
    return r;
}

// The update of one cell, stages C to G.  phi, rhoH, fl: its moments and liquid
// fraction.  Io supplies
//   stencil(fi, gx, gy, lap): 12 grad of field fi (phi_p: fi = p, rho: N, psi: N + 1), and
//     6 lap for fi < N;   f(i), g(p, i), h(i): its populations;   lag(a): lagged plane a (see
//     aux_psi ...);
// and takes
//   push<KIND>(s, q): the post-collision populations of species s;
//   dirichlet(...): the boundary row's incoming enthalpy populations;
//   put_lag(a, v): the lagged values;   put_fields(...): the macroscopic fields (!COLLIDE).
template <int N, bool COLLIDE, class Pr, class V, class Io>
__device__ __forceinline__ void cell_update(const KParams& P, Io& io, const V (&phi)[N], V rhoH, V fl)
{
    using K = exact_t<V>;
    const auto& C = coef<const_t<V>>(P);
    const Mixture<V> m = mixture_of<N>(P, phi, rhoH, fl);
    const V rho = m.rho;

    // ---- stage C: isotropic stencils (12 grad, 6 lap) ------------------------
    V gpx[N + 2], gpy[N + 2], lap[N];
#pragma unroll(Pr::COMPACT ? 1 : N + 2)
    for (int fi = 0; fi < N + 2; ++fi) {
        V l;
        io.stencil(fi, gpx[fi], gpy[fi], l);
        if (fi < N) lap[fi] = l;
    }
    const V grx = gpx[N], gry = gpy[N], gsx = gpx[N + 1], gsy = gpy[N + 1];

    // ---- stage D: pairwise normals, R_p, chemical potentials, F_s -----------
    V Rx[N], Ry[N], mup[N], gpv[N], n2[N];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        // g'(phi) / 2, g = phi^2 (1 - phi)^2
        gpv[p] = (phi[p] * (V(K(1)) - phi[p])) * rfma(phi[p], K(-2), V(K(1)));
        if constexpr (Pr::NGUARD > 0.0f) n2[p] = rfma(gpx[p], gpx[p], gpy[p] * gpy[p]);
    }
#pragma unroll
    for (int p = 0; p < N; ++p)
#pragma unroll
        for (int q = p + 1; q < N; ++q) {
            // n_pq = grad(phi_p / s) / |grad(phi_p / s)|, s = phi_p + phi_q; the quotient rule
            // gives grad(phi_p / s) = G / s^2 with G below, so n_pq = G / |G|
            const V s = phi[p] + phi[q];
            const V mp = -phi[p];
            const V Gx = rfma(phi[q], gpx[p], mp * gpx[q]);
            const V Gy = rfma(phi[q], gpy[p], mp * gpy[q]);
            const V G2 = rfma(Gx, Gx, Gy * Gy);
            V ref = V(0.0f);
            if constexpr (Pr::NGUARD > 0.0f) ref = rfma(phi[q] * phi[q], n2[p], (phi[p] * phi[p]) * n2[q]);
            const V ar = normal_weight<Pr>(s, G2, ref, (phi[p] * phi[q]) * C.four_eps);
            Rx[p] = q == 1 ? ar * Gx : rfma(ar, Gx, Rx[p]);
            Ry[p] = q == 1 ? ar * Gy : rfma(ar, Gy, Ry[p]);
            Rx[q] = p == 0 ? -(ar * Gx) : rfma(-ar, Gx, Rx[q]);
            Ry[q] = p == 0 ? -(ar * Gy) : rfma(-ar, Gy, Ry[q]);
            const V gs = (s * (V(K(1)) - s)) * rfma(s, K(-2), V(K(1)));
            const V lp = q == 1 ? lap[q] * C.kk6[p][q] : rfma(lap[q], C.kk6[p][q], mup[p]);
            const V lq = p == 0 ? lap[p] * C.kk6[q][p] : rfma(lap[p], C.kk6[q][p], mup[q]);
            mup[p] = rfma(gpv[p] - gs, C.b4[p][q], lp);
            mup[q] = rfma(gpv[q] - gs, C.b4[q][p], lq);
        }
    V Fx = mup[0] * gpx[0], Fy = mup[0] * gpy[0];
#pragma unroll
    for (int p = 1; p < N; ++p) {
        Fx = rfma(mup[p], gpx[p], Fx);
        Fy = rfma(mup[p], gpy[p], Fy);
    }
    const auto c12 = cst<V>(1.0 / 12.0);
    Fx = rfma(Fx, c12, rho * C.accel[0]);
    Fy = rfma(Fy, c12, rho * C.accel[1]);

    // ---- stage E: flow macroscopics ----------------------------------------
    V f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = io.f(i);
    const V fa = f[5] - f[7], fb = f[8] - f[6];
    const V jx = (f[1] - f[3]) + (fa + fb);
    const V jy = (f[2] - f[4]) + (fa - fb);
    const V sum_f = ((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]));
    // 1 / rho, omega_f = 1 / tau_f = rho / A, omega_h = 1 / tau_h = 1 / B and T = Zn / (rho c_p) + T0;
    // tau_f = A / rho, A = 3 mu + rho / 2 (tau_f = mu / (rho c_s^2) + 1/2), and
    // tau_h = B = lambda / (rho_ref c_p,ref c_s^2) + 1/2
    const V Af = rfma(m.mu, K(3), rho * K(0.5));
    const V Bh = rfma(m.lam, C.tau_h_scale, V(K(0.5)));
    const V rc = rho * m.cp;
    V irho, om, oh, T;
    if constexpr (std::is_same<V, df64>::value) {
        // a chain of unnormalised products would show in 1/rho (the error of rho (1/rho) moves the
        // momentum step after step) and in T; a quotient costs little more than two products
        irho = rinv(rho);
        const V r = rinv(Af * Bh);
        om = rho * (Bh * r);
        oh = Af * r;
        T = m.Zn / rc + m.T0;
    } else {
        // one reciprocal for all four
        const V RA = rho * Af, BC = Bh * m.cp;
        const V r = rinv(RA * BC);
        const V rRA = BC * r, rBC = RA * r;
        irho = Af * rRA;
        om = (rho * rho) * rRA;
        oh = m.cp * rBC;
        T = rfma(m.Zn, irho * (Bh * rBC), m.T0);
    }
    const V usx = rfma(Fx, K(0.5), jx) * irho, usy = rfma(Fy, K(0.5), jy) * irho;
    const V fpx = m.chi * (V(C.us[0]) - usx), fpy = m.chi * (V(C.us[1]) - usy);
    const V ux = rfma(fpx, K(0.5), usx), uy = rfma(fpy, K(0.5), usy);
    // mdot = M / rho, M = -D psi / Dt; S = rho mdot + u . grad rho = M + u . grad rho
    const V M = rfma(rfma(ux, gsx, uy * gsy), cst<V>(-1.0 / 12.0), io.lag(aux_psi()) - m.psi);
    const V mdot = M * irho;
    const V S = rfma(rfma(ux, grx, uy * gry), c12, M);
    const V uF = rfma(ux, Fx, uy * Fy), uu = rfma(ux, ux, uy * uy);
    // p = 3/5 (sum f_i + S/2 + (tau_f - 1/2) F_0 - (2/3) rho u.u), F_0 = -(4/3) u.F
    const V tF = (m.mu * irho) * uF;
    const V p = rfma(tF, K(-4), rfma(S, K(0.5), rfma(rho * uu, cst<V>(-2.0 / 3.0), sum_f))) * cst<V>(0.6);

    if constexpr (!COLLIDE) {
        io.put_fields(phi, T, rhoH * irho, fl, ux, uy, p);
        return;
    }

    // ---- stage F: flow collision -------------------------------------------
    // even and odd parts of the equilibrium and source terms over w_i, times 1/9
    {
        const V ks = rfma(om, K(-0.5), V(K(1))), om1 = V(K(1)) - om;
        const V rom = om * rho, krho = ks * rho;
        const V hrom = rom * K(0.5), kFx = ks * Fx, kFy = ks * Fy;
        const V X = rfma(hrom, ux, kFx), Y = rfma(hrom, uy, kFy);
        const V axy = rfma(ux, Y, uy * X);
        const V kS = ks * S;
        const auto sixth = cst<V>(1.0 / 6.0), third = cst<V>(1.0 / 3.0);
        const V omp = om * p;
        const V iso = rfma(ux, X, uy * Y) * cst<V>(-1.0 / 3.0);
        const V a0 = rfma(omp, third, iso);
        const V x0 = rfma(omp, cst<V>(-3.75 / 9.0), iso);
        const V tx = rfma(krho, fpx, rfma(rom, ux, kFx)), ty = rfma(krho, fpy, rfma(rom, uy, kFy));
        const V as = rfma(kS, sixth, a0), bx = rfma(ux, X, as), by = rfma(uy, Y, as), bd = rfma(kS, sixth, rfma(uy, Y, bx));
        V q[9];
        q[0] = rfma(x0, K(4), om1 * f[0]);
        collide_pairs(om1, f, bx, by, bd + axy, bd - axy, tx, ty, third, q);
        io.template push<KIND_F>(0, q);
    }

    // ---- stage F: phase-field collisions -------------------------------------
    {
        const V gm = rfma(mdot, C.kg, V(C.omega_g));
#pragma unroll(Pr::COMPACT ? 1 : N)
        for (int pp = 0; pp < N; ++pp) {
            V gq[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) gq[i] = io.g(pp, i);
            const V pu = phi[pp] * ux, pv = phi[pp] * uy;
            const V bx = rfma(pu, C.g_pl[0], rfma(io.lag(aux_phiux(pp)), C.g_pl[1], Rx[pp] * C.g_pl[2]));
            const V by = rfma(pv, C.g_pl[0], rfma(io.lag(aux_phiuy(N, pp)), C.g_pl[1], Ry[pp] * C.g_pl[2]));
            const V og1 = V(C.omega_g1);
            // the rest direction takes what the others leave of phi_p (omega_g + k_g mdot), so
            // that the rounding of 1/9 does not change sum_i g_i, step after step
            const V all = phi[pp] * gm, b0 = all * cst<V>(1.0 / 9.0);
            V q[9];
            q[0] = rfma(b0, K(-5), rfma(gq[0], C.omega_g1, all));
            collide_pairs(og1, gq, b0, bx, by, q);
            io.template push<KIND_G>(1 + pp, q);
            io.put_lag(aux_phiux(pp), pu);
            io.put_lag(aux_phiuy(N, pp), pv);
        }
    }

    // ---- stage F: enthalpy collision + Dirichlet ghosts ---------------------
    {
        V h[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = io.h(i);
        // Z = rho c_p T, E = rho_ref c_p,ref T
        const V Z = rfma(rc, m.T0, m.Zn), E = T * C.E_ref;
        const V kh = rfma(oh, K(-0.5), V(K(1))), oh1 = V(K(1)) - oh;
        const V Zm = Z * mdot, src = kh * Zm;
        const V base = rfma(oh, E, src) * cst<V>(1.0 / 9.0);
        const V ohZ = oh * Z, vx = ohZ * ux, vy = ohZ * uy;
        const V vxx = vx * ux, vyy = vy * uy, vs = vxx + vyy;
        const V c0 = rfma(vs, cst<V>(-1.0 / 6.0), base);
        const V bx = rfma(vxx, K(0.5), c0), by = rfma(vyy, K(0.5), c0), bd = rfma(vs, K(0.5), c0);
        V q[9];
        // the rest direction takes what the others leave of omega_h rho H + k_h Z mdot
        q[0] = rfma(c0, K(-5), rfma(vs, K(-1.5), rfma(oh1, h[0], rfma(oh, rhoH, src))));
        collide_pairs(oh1, h, bx, by, rfma(vx, uy, bd), rfma(-vx, uy, bd), vx, vy, cst<V>(1.0 / 3.0), q);
        // outflow rows are copied inside push; Dirichlet rows get their incoming populations
        // from the ghost rule
        io.template push<KIND_H>(N + 1, q);
        io.dirichlet(h, oh1, Z, E, T, ux, uy, uu);
        io.put_lag(aux_mdot(), mdot);
        io.put_lag(aux_Q(), Zm);
        io.put_lag(aux_psi(), m.psi);
    }
}

}  // namespace lbm
