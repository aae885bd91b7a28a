// lbm_cell16.cuh -- the update of one cell for the policies with 16-bit moving populations: the
// algebra of lbm_cell.cuh in plain populations and in the order in which the scheme is written
// (arXiv 2603.22902, Sections 2 and 3), in FP32.
//
// Why it is not lbm_cell.cuh's form: a stored value keeps 8 (BF16) or 11 (FP16) bits, so another
// order of the FP32 roundings sends values near a tie to the other neighbour, and f_1 - f_3 and
// its like cancel all but that difference.  Two orders that are equally close to the unrounded
// scheme differ by 1 to 10 % in the velocities of a BF16 run (film 16 x 64, 20 steps) and by 0.2 %
// in those of an FP16 run (drop 512 x 512, 100 steps).  The results of these policies are
// therefore tied to this order.  The shared form needs fewer instructions (FP16 storage, N = 2,
// 512 x 512: 1236 against 1440 per cell).
#pragma once

#include "lbm_cell.cuh"

namespace lbm {

// The moments of a cell (phi_p, rho H), its state by eq. H and its mixture by eq. 2.
template <int N>
struct Cell16 {
    float phi[N], rhoH, fl, T, rho, psi, mu, lam, cp, chi;
};

// eq. H for one cell: f_l as the FP64 map gives it and, with WANT_T, T: of a cell that the FP32 screen
// decides by the formula of its branch, of the others by the map.
template <int N, bool WANT_T>
__device__ __forceinline__ void map_cell16(const KParams& P, Cell16<N>& m)
{
    const Coef<float>& C = P.f;
    const int sure = eqh_screen<N>(P, m.phi, m.rhoH);
    if (sure > 0) {
        m.fl = 1.0f;
        if (WANT_T) {
            const float rcl = mix_sum<N, float>(m.phi, C.rho_l) * mix_sum<N, float>(m.phi, C.cp_l);
            const float Al = fmaf(rcl, C.T_liq, mix_sum<N, float>(m.phi, C.rhoL));
            m.T = C.T_liq + (m.rhoH - Al) / rcl;
        }
        return;
    }
    if (sure == 0) {
        m.fl = 0.0f;
        if (WANT_T) m.T = m.rhoH / (mix_sum<N, float>(m.phi, C.rho_s) * mix_sum<N, float>(m.phi, C.cp_s));
        return;
    }
    double phd[N];
#pragma unroll
    for (int p = 0; p < N; ++p) phd[p] = (double)m.phi[p];
    const Mix<N> mix = mixture_map<N>(P, phd);
    double fld, Td = 0.0;
    enthalpy_map<N, WANT_T>(P, mix, (double)m.rhoH, fld, Td);
    m.fl = (float)fld;
    if (WANT_T) m.T = (float)Td;
}

// Stages A + B of one cell of the tile (OWN) or of its ring, which needs phi_p, rho and psi alone.
template <int N, bool OWN, class L>
__device__ __forceinline__ void moments16(const KParams& P, const L& ld, typename L::Cell c, Cell16<N>& m)
{
    const Coef<float>& C = P.f;
    const float mdm = ld.aux(aux_mdot(), c, 1);
    const float Qm = ld.aux(aux_Q(), c, 2);
    const float iden = 1.0f / (1.0f - 0.5f * mdm);
#pragma unroll
    for (int p = 0; p < N; ++p) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 9; ++i) s += ld.template pop<KIND_G>(1 + p, i, c, 3);
        m.phi[p] = s * iden;
    }
    float sh = 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) sh += ld.template pop<KIND_H>(N + 1, i, c, 4);
    m.rhoH = rfma(0.5f, Qm, sh);
    map_cell16<N, OWN>(P, m);
    const float fs = 1.0f - m.fl, fl = m.fl;
    m.rho = rfma(fs, mix_sum<N, float>(m.phi, C.rho_s), fl * mix_sum<N, float>(m.phi, C.rho_l));
    m.psi = fs * mix_sum<N, float>(m.phi, C.drho);
    if (OWN) {
        m.mu = rfma(fs, mix_sum<N, float>(m.phi, C.mu_s), fl * mix_sum<N, float>(m.phi, C.mu_l));
        m.lam = rfma(fs, mix_sum<N, float>(m.phi, C.lam_s), fl * mix_sum<N, float>(m.phi, C.lam_l));
        m.cp = rfma(fs, mix_sum<N, float>(m.phi, C.cp_s), fl * mix_sum<N, float>(m.phi, C.cp_l));
        m.chi = fs * mix_sum<N, float>(m.phi, C.pcm);
    }
}

// g'(x) - g'(s) of the chemical potentials, g'(x) = A(x) B(x) with A = 2 x (1 - x), B = 1 - 2 x.  The
// difference can be fused with either product or with none, which rounds in three ways, and a unit in
// the last place of mu_p is one of u.  The results of these policies were made with the choices below, for
// term 2 k (phase p) and 2 k + 1 (phase q) of the k-th pair, which the compiler made for each kernel when
// they were left to it; they are written out so that it makes no others.
constexpr int FUSE_X = 0, FUSE_S = 1, FUSE_NONE = 2;
enum Caller16 { CALLER_STEP, CALLER_STAGED, CALLER_BATCH, CALLER_FIELDS };
template <int N, int CALLER>
__device__ __forceinline__ constexpr int gdiff_form(int term)
{
    if (CALLER == CALLER_STAGED && N == 3) return FUSE_S;
    if (CALLER == CALLER_FIELDS && N == 4) return FUSE_S;
    if (CALLER == CALLER_STEP && N == 3 && term < 2) return FUSE_S;
    if (CALLER == CALLER_STEP && N == 4 && term == 0) return FUSE_NONE;
    return FUSE_X;
}
__device__ __forceinline__ float gdiff(int form, float x, float s)
{
    auto A = [](float a) { return __fmul_rn(__fmul_rn(2.0f, a), __fsub_rn(1.0f, a)); };
    auto B = [](float a) { return __fmaf_rn(-2.0f, a, 1.0f); };
    if (form == FUSE_X) return __fmaf_rn(A(x), B(x), -__fmul_rn(A(s), B(s)));
    const float gx = __fmul_rn(A(x), B(x));
    return form == FUSE_S ? __fmaf_rn(-A(s), B(s), gx) : __fsub_rn(gx, __fmul_rn(A(s), B(s)));
}

// Stages C to G (see cell_update in lbm_cell.cuh for what io supplies and takes).
template <int N, bool COLLIDE, class Pr, class Io>
__device__ __forceinline__ void cell_update16(const KParams& P, Io& io, const Cell16<N>& m)
{
    const Coef<float>& C = P.f;
    const float rho = m.rho, rhoH = m.rhoH, T = m.T;

    // ---- stage C: isotropic stencils ---------------------------------------
    float gpx[N + 2], gpy[N + 2], lap[N];
#pragma unroll
    for (int fi = 0; fi < N + 2; ++fi) {
        const float e = io.at(fi, 1, 0), w = io.at(fi, -1, 0), n = io.at(fi, 0, 1), s = io.at(fi, 0, -1);
        const float ne = io.at(fi, 1, 1), nw = io.at(fi, -1, 1), se = io.at(fi, 1, -1), sw = io.at(fi, -1, -1);
        gpx[fi] = (e - w) * float(1.0 / 3.0) + ((ne - nw) + (se - sw)) * float(1.0 / 12.0);
        gpy[fi] = (n - s) * float(1.0 / 3.0) + ((ne - se) + (nw - sw)) * float(1.0 / 12.0);
        if (fi < N) {
            const float v0 = io.at(fi, 0, 0);
            const float ax = (e + w) + (n + s);
            const float dg = (ne + nw) + (se + sw);
            lap[fi] = ax * float(2.0 / 3.0) + dg * float(1.0 / 6.0) - v0 * float(10.0 / 3.0);
        }
    }
    const float grx = gpx[N], gry = gpy[N], gsx = gpx[N + 1], gsy = gpy[N + 1];

    // ---- stage D: pairwise normals, R_p, chemical potentials, F_s -----------
    const float (&phi)[N] = m.phi;
    constexpr int CALLER = COLLIDE ? Io::CALLER : CALLER_FIELDS;
    float Rx[N], Ry[N], mup[N];
    int term = 0;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        Rx[p] = 0.0f;
        Ry[p] = 0.0f;
        mup[p] = 0.0f;
    }
#pragma unroll
    for (int p = 0; p < N; ++p)
#pragma unroll
        for (int q = p + 1; q < N; ++q) {
            const float s = phi[p] + phi[q];
            float nxv = 0.0f, nyv = 0.0f;
            if (s > 1e-12f) {
                // the guards of normal_weight (lbm_cell.cuh)
                const float Gx = phi[q] * gpx[p] - phi[p] * gpx[q];
                const float Gy = phi[q] * gpy[p] - phi[p] * gpy[q];
                const float G2 = Gx * Gx + Gy * Gy;
                const float s2 = s * s;
                const float ref = phi[q] * phi[q] * (gpx[p] * gpx[p] + gpy[p] * gpy[p]) +
                                  phi[p] * phi[p] * (gpx[q] * gpx[q] + gpy[q] * gpy[q]);
                if (G2 > float(Pr::NABS2) * (s2 * s2) && G2 > float(Pr::NGUARD * Pr::NGUARD) * ref) {
                    const float r = rrsqrt(G2);
                    nxv = Gx * r;
                    nyv = Gy * r;
                }
            }
            const float a = C.four_eps * phi[p] * phi[q];
            Rx[p] = rfma(a, nxv, Rx[p]);
            Ry[p] = rfma(a, nyv, Ry[p]);
            Rx[q] = rfma(-a, nxv, Rx[q]);
            Ry[q] = rfma(-a, nyv, Ry[q]);
            mup[p] += rfma(C.b2[p][q], gdiff(gdiff_form<N, CALLER>(term++), phi[p], s), C.kk[p][q] * lap[q]);
            mup[q] += rfma(C.b2[q][p], gdiff(gdiff_form<N, CALLER>(term++), phi[q], s), C.kk[q][p] * lap[p]);
        }
    float Fx = rho * C.accel[0], Fy = rho * C.accel[1];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        Fx = rfma(mup[p], gpx[p], Fx);
        Fy = rfma(mup[p], gpy[p], Fy);
    }

    // ---- stage E: flow macroscopics ----------------------------------------
    float f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = io.f(i);
    const float jx = ((f[1] - f[3]) + (f[5] - f[7])) + (f[8] - f[6]);
    const float jy = ((f[2] - f[4]) + (f[5] - f[7])) + (f[6] - f[8]);
    const float sum_f = ((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]));
    // 1 / rho, omega_f = 1 / tau_f = rho / A and omega_h = 1 / tau_h = 1 / B from one division (A, B: lbm_cell.cuh)
    const float Af = rfma(3.0f, m.mu, 0.5f * rho);
    const float Bh = rfma(m.lam, C.tau_h_scale, 0.5f);
    const float rAB = 1.0f / (rho * Af * Bh);
    const float irho = (Af * Bh) * rAB;
    const float om = (rho * rho) * (Bh * rAB);
    const float oh = (rho * Af) * rAB;
    const float usx = rfma(0.5f, Fx, jx) * irho, usy = rfma(0.5f, Fy, jy) * irho;
    const float fpx = m.chi * (C.us[0] - usx), fpy = m.chi * (C.us[1] - usy);
    const float ux = rfma(0.5f, fpx, usx), uy = rfma(0.5f, fpy, usy);
    const float psim = io.lag(aux_psi());
    const float mdot = -((m.psi - psim) + (ux * gsx + uy * gsy)) * irho;
    const float Ssrc = rfma(rho, mdot, ux * grx + uy * gry);
    const float Lxx = rfma(2.0f * ux, Fx, Ssrc * float(1.0 / 3.0));
    const float Lyy = rfma(2.0f * uy, Fy, Ssrc * float(1.0 / 3.0));
    const float Lxy = rfma(ux, Fy, uy * Fx);
    const float tmh = 3.0f * m.mu * irho;  // tau_f - 1/2
    const float F0 = wgt_r<float>(0) * rfma(-1.5f, Lxx + Lyy, Ssrc);
    const float uu = rfma(ux, ux, uy * uy);
    const float p = 0.6f * (((sum_f + 0.5f * Ssrc) + tmh * F0) - rho * wgt_r<float>(0) * 1.5f * uu);

    if constexpr (!COLLIDE) {
        io.put_fields(phi, T, rhoH * irho, m.fl, ux, uy, p);
        return;
    }

    // ---- stage F: flow collision -------------------------------------------
    {
        const float k = rfma(-0.5f, om, 1.0f), om1 = 1.0f - om;
        const float Fex = rfma(rho, fpx, Fx), Fey = rfma(rho, fpy, Fy);
        const float rom = om * rho;
        const float a0 = om * rfma(-1.5f * rho, uu, 3.0f * p) + k * rfma(-1.5f, Lxx + Lyy, Ssrc);
        const float ax = 3.0f * rfma(rom, ux, k * Fex);
        const float ay = 3.0f * rfma(rom, uy, k * Fey);
        const float axx = 4.5f * rfma(rom * ux, ux, k * Lxx);
        const float ayy = 4.5f * rfma(rom * uy, uy, k * Lyy);
        const float axy = 9.0f * rfma(rom * ux, uy, k * Lxy);
        const float bx = a0 + axx, by = a0 + ayy, bd = a0 + axx + ayy;
        float X[9];
        X[0] = rfma(-6.75f * om, p, a0);
        X[1] = bx + ax;
        X[3] = bx - ax;
        X[2] = by + ay;
        X[4] = by - ay;
        X[5] = (bd + axy) + (ax + ay);
        X[7] = (bd + axy) - (ax + ay);
        X[6] = (bd - axy) + (ay - ax);
        X[8] = (bd - axy) - (ay - ax);
        float q[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) q[i] = rfma(wgt_r<float>(i), X[i], om1 * f[i]);
        io.template push<KIND_F>(0, q);
    }

    // ---- stage F: phase-field collisions -------------------------------------
    {
        const float og = C.omega_g, kg = C.kg, og1 = 1.0f - og;
#pragma unroll
        for (int pp = 0; pp < N; ++pp) {
            float gq[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) gq[i] = io.g(pp, i);
            const float Dx = phi[pp] * ux - io.lag(aux_phiux(pp));
            const float Dy = phi[pp] * uy - io.lag(aux_phiuy(N, pp));
            const float b0 = og * phi[pp] + kg * phi[pp] * mdot;
            const float bxv = 3.0f * og * phi[pp] * ux + kg * rfma(3.0f, Dx, Rx[pp]);
            const float byv = 3.0f * og * phi[pp] * uy + kg * rfma(3.0f, Dy, Ry[pp]);
            float q[9];
            q[0] = rfma(wgt_r<float>(0), b0, og1 * gq[0]);
            q[1] = rfma(wgt_r<float>(1), b0 + bxv, og1 * gq[1]);
            q[3] = rfma(wgt_r<float>(3), b0 - bxv, og1 * gq[3]);
            q[2] = rfma(wgt_r<float>(2), b0 + byv, og1 * gq[2]);
            q[4] = rfma(wgt_r<float>(4), b0 - byv, og1 * gq[4]);
            q[5] = rfma(wgt_r<float>(5), b0 + (bxv + byv), og1 * gq[5]);
            q[7] = rfma(wgt_r<float>(7), b0 - (bxv + byv), og1 * gq[7]);
            q[6] = rfma(wgt_r<float>(6), b0 + (byv - bxv), og1 * gq[6]);
            q[8] = rfma(wgt_r<float>(8), b0 - (byv - bxv), og1 * gq[8]);
            io.template push<KIND_G>(1 + pp, q);
            io.put_lag(aux_phiux(pp), phi[pp] * ux);
            io.put_lag(aux_phiuy(N, pp), phi[pp] * uy);
        }
    }

    // ---- stage F: enthalpy collision + Dirichlet ghosts ---------------------
    {
        float h[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = io.h(i);
        const float Z = rho * m.cp * T, E = C.E_ref * T;
        const float kh = rfma(-0.5f, oh, 1.0f), oh1 = 1.0f - oh;
        const float Zm = Z * mdot;
        const float c0 = oh * rfma(-1.5f * Z, uu, E) + kh * Zm;
        const float ohZ = oh * Z;
        const float cxv = 3.0f * ohZ * ux, cyv = 3.0f * ohZ * uy;
        const float cxx = 4.5f * ohZ * ux * ux, cyy = 4.5f * ohZ * uy * uy, cxy = 9.0f * ohZ * ux * uy;
        const float heq0 = (rhoH - E) + wgt_r<float>(0) * rfma(-1.5f * Z, uu, E);
        const float bx = c0 + cxx, by = c0 + cyy, bd = c0 + cxx + cyy;
        float q[9];
        q[0] = rfma(oh, heq0, rfma(kh * wgt_r<float>(0), Zm, oh1 * h[0]));
        q[1] = rfma(wgt_r<float>(1), bx + cxv, oh1 * h[1]);
        q[3] = rfma(wgt_r<float>(3), bx - cxv, oh1 * h[3]);
        q[2] = rfma(wgt_r<float>(2), by + cyv, oh1 * h[2]);
        q[4] = rfma(wgt_r<float>(4), by - cyv, oh1 * h[4]);
        q[5] = rfma(wgt_r<float>(5), (bd + cxy) + (cxv + cyv), oh1 * h[5]);
        q[7] = rfma(wgt_r<float>(7), (bd + cxy) - (cxv + cyv), oh1 * h[7]);
        q[6] = rfma(wgt_r<float>(6), (bd - cxy) + (cyv - cxv), oh1 * h[6]);
        q[8] = rfma(wgt_r<float>(8), (bd - cxy) - (cyv - cxv), oh1 * h[8]);
        io.template push<KIND_H>(N + 1, q);
        io.dirichlet16(h, oh1, Z, E, T, ux, uy, uu);
        io.put_lag(aux_mdot(), mdot);
        io.put_lag(aux_Q(), Zm);
        io.put_lag(aux_psi(), m.psi);
    }
}

}  // namespace lbm
