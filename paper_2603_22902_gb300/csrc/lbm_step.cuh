// lbm_step.cuh -- the fused time step of the coupled LB scheme (arXiv 2603.22902,
// Section 3), one kernel launch per step, generic over the storage / arithmetic
// precision policy (lbm_prec.cuh).
//
// State between launches: pre-collision (post-streaming) populations f, g_p (p < N),
// h as structure-of-arrays planes (rest block + moving block), and the lagged planes
// mdot', Q' = rho c_p T mdot, psi', (phi_p u)'.  One launch reads set A and writes
// set B (ping-pong), so it is race-free across blocks.
//
// Per block (a TX x TY tile, one thread per cell):
//   1. the moments of every cell of the tile and of its 1-cell ring (phi_p = sum g /
//      (1 - mdot'/2), rho H = sum h + Q'/2) and the liquid fraction of eq. H: the ring
//      cells recompute phi_p, rho, psi from their own populations (no second kernel, no
//      extra HBM field).  FP64 / FP32 / 16-bit policies evaluate the own cell in registers and
//      share the ring out; the compact (double-word) policy runs one loop over all positions
//      so that this code exists once.  f_l is always the FP64 map's; an FP32 screen decides
//      the cells that are clearly liquid or solid (liquid_fraction, lbm_cell.cuh);
//   2. ghost values beyond walls/outflows are filled (zero gradient; wetting for phi_p),
//      skipped by tiles that have none;
//   3. the rest of the cell's update (lbm_cell.cuh, for 16-bit storage lbm_cell16.cuh): stencils from shared
//      memory, interface terms, flow macroscopics and the three BGK collisions;
//   4. post-collision populations are pushed to the neighbours' slots of set B with
//      the boundary rules (bounce-back, outflow copy, non-equilibrium extrapolation
//      of the Dirichlet temperature; rows that are neither the lattice's first nor its
//      last skip the checks, see push_species), and the lagged planes are written.
// No address outside the planes is ever formed, not even for a value that is then
// not used: the compiler may issue loads ahead of the branch that guards them.
#pragma once

#include "lbm_cell.cuh"
#include "lbm_cell16.cuh"
#include "lbm_device.cuh"
#include "lbm_prec.cuh"

namespace lbm {

struct ExportPtrs {
    double *phi, *T, *H, *fl, *ux, *uy, *p;
};

// v mod n in [0, n) for any int v (n > 0).
__device__ __forceinline__ int wrap_index(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// Views of one population set: rest block (N + 2 planes) and moving block (8 (N + 2)).
template <class Pr>
struct PopView {
    typename Pr::TR* rest;
    typename Pr::TM* move;
};
template <class Pr>
__device__ __forceinline__ PopView<Pr> pop_view(const KParams& P, const void* base)
{
    char* b = (char*)base;
    return PopView<Pr>{(typename Pr::TR*)b, (typename Pr::TM*)(b + P.rest_elems * (long long)sizeof(typename Pr::TR))};
}

// A stored moving population (direction i >= 1) as a plain value of the arithmetic type R.
template <class Pr, int KIND>
__device__ __forceinline__ typename Pr::R dequant(const KParams& P, typename Pr::TM q, int i)
{
    using R = typename Pr::R;
    if constexpr (!Pr::QUANT) {
        return (R)q;
    } else {
        const float w = (float)wgt(i);
        const float qf = to_f(q);
        if (KIND == KIND_F) return qf * (w * F_SCALE);
        if (KIND == KIND_G) return qf * w;
        return qf * (w * P.f.E_ref);
    }
}

// Load population i of species s at cell c as a plain value (dequantised to R).
template <class Pr, int KIND>
__device__ __forceinline__ typename Pr::R ld_pop(const KParams& P, const PopView<Pr>& v, int s, int i, long long c, int site)
{
    using R = typename Pr::R;
    if (i == 0) return (R)LBM_LDX(Pr::COH, P, v.rest, (long long)s * P.S + c, P.rest_elems, site);
    const auto q = LBM_LDX(Pr::COH, P, v.move, (long long)(s * 8 + i - 1) * P.S + c, P.move_elems, site);
    return dequant<Pr, KIND>(P, q, i);
}

// The value type of a policy's step: 16-bit storage computes in float (lbm_cell16.cuh).
template <class Pr>
using step_val = typename std::conditional<Pr::QUANT, float, val_t<typename Pr::R>>::type;

// Population i of species s at cell c as the step's arithmetic takes it.
template <class Pr, int KIND>
__device__ __forceinline__ step_val<Pr> ld_val(const KParams& P, const PopView<Pr>& v, int s, int i, unsigned c, int site)
{
    using R = typename Pr::R;
    if (i == 0) return step_val<Pr>((R)ld_plane<Pr::COH>(P, v.rest, s, c, P.rest_elems, site));
    return step_val<Pr>(dequant<Pr, KIND>(P, ld_plane<Pr::COH>(P, v.move, s * 8 + i - 1, c, P.move_elems, site), i));
}

// The same load for a second read of a population in one step: through the cached
// (L1) path instead of the read-only one, so that the compiler does not merge it with
// the first read and keep the value in a register meanwhile.
template <class Pr, int KIND>
__device__ __forceinline__ step_val<Pr> ld_val_late(const KParams& P, const PopView<Pr>& v, int s, int i, unsigned c, int site)
{
    using R = typename Pr::R;
#ifdef LBM_CHECK_BOUNDS
    const long long idx = i == 0 ? (long long)s * P.S + c : (long long)(s * 8 + i - 1) * P.S + c;
    if (!lbm_in_bounds(P.dbg, idx, i == 0 ? P.rest_elems : P.move_elems, site))
        return step_val<Pr>((R)0.0f);
#else
    (void)site;
#endif
    if (i == 0) return step_val<Pr>((R)lbm_ld_l1<Pr::COH>(plane_elem(v.rest, P, s, c)));
    return step_val<Pr>(dequant<Pr, KIND>(P, lbm_ld_l1<Pr::COH>(plane_elem(v.move, P, s * 8 + i - 1, c)), i));
}

// The plain value val of a moving population (direction i >= 1) in its stored form.
template <class Pr, int KIND>
__device__ __forceinline__ typename Pr::TM quant(const KParams& P, typename Pr::R val, int i)
{
    using TM = typename Pr::TM;
    if constexpr (!Pr::QUANT) {
        return (TM)val;
    } else {
        const float w = (float)wgt(i);
        float q;
        if (KIND == KIND_F) q = (float)val * (1.0f / (w * F_SCALE));
        else if (KIND == KIND_G) q = (float)val * (1.0f / w);
        else q = (float)val * (1.0f / w) * P.f.inv_E_ref;
        return from_f<TM>(q);
    }
}

// Store the plain value val of population i of species s at cell c (quantised from R).
template <class Pr, int KIND>
__device__ __forceinline__ void st_pop(const KParams& P, const PopView<Pr>& v, int s, int i, long long c,
                                       typename Pr::R val, int site)
{
    if (i == 0) LBM_ST(P, v.rest, (long long)s * P.S + c, P.rest_elems, site, (typename Pr::TR)val);
    else LBM_ST(P, v.move, (long long)(s * 8 + i - 1) * P.S + c, P.move_elems, site, (quant<Pr, KIND>(P, val, i)));
}

// The same at cell c + shift, from the step's value type; shift is the same for all threads.
template <class Pr, int KIND>
__device__ __forceinline__ void st_val(const KParams& P, const PopView<Pr>& v, int s, int i, int shift, unsigned c,
                                       step_val<Pr> val, int site)
{
    using R = typename Pr::R;
    using TR = typename Pr::TR;
    using TM = typename Pr::TM;
    if (i == 0) st_plane<TR>(P, v.rest, s, shift, c, P.rest_elems, site, (TR)(R)val);
    else st_plane<TM>(P, v.move, s * 8 + i - 1, shift, c, P.move_elems, site, quant<Pr, KIND>(P, (R)val, i));
}

// Where a step reads its inputs.  A loader addresses a cell of the tile-with-ring by a
// Cell value and gives its populations (dequantised) and lagged values.
//   GlobalLoader: the population and lagged sets in global memory, cells by their index in
//     the lattice (step_tile_l maps a position of the tile-with-ring to it).
//   StagedLoader: the same inputs of one tile copied into shared memory by the
//     tensor-memory accelerator (lbm_staged.cuh); cells by their position in the tile.
template <class Pr>
struct GlobalLoader {
    using V = step_val<Pr>;
    using Cell = unsigned;
    static constexpr bool GLOBAL = true;   // step_tile_l locates the cells itself
    const KParams& P;
    PopView<Pr> pin;
    const typename Pr::TA* __restrict__ ain;
    __device__ __forceinline__ Cell own(int x, int y, int, int) const { return (unsigned)y * (unsigned)P.nx + (unsigned)x; }
    template <int KIND>
    __device__ __forceinline__ V pop(int s, int i, Cell c, int site) const
    {
        return ld_val<Pr, KIND>(P, pin, s, i, c, site);
    }
    template <int KIND>
    __device__ __forceinline__ V pop_late(int s, int i, Cell c, int site) const
    {
        return ld_val_late<Pr, KIND>(P, pin, s, i, c, site);
    }
    __device__ __forceinline__ V aux(int a, Cell c, int site) const
    {
        return V((typename Pr::R)ld_plane<Pr::COH>(P, ain, a, c, P.aux_elems, site));
    }
};

// Stage A + B of one cell of the tile or its ring: phi_p, rho H and f_l.
template <int N, class Pr, class L, class V>
__device__ __forceinline__ void cell_moments(const KParams& P, const L& ld, typename L::Cell c, V (&phi)[N], V& rhoH, V& fl)
{
    moments<N>(P, ld.aux(aux_mdot(), c, 1), ld.aux(aux_Q(), c, 2),
               [&](int p, int i) { return ld.template pop<KIND_G>(1 + p, i, c, 3); },
               [&](int i) { return ld.template pop<KIND_H>(N + 1, i, c, 4); }, phi, rhoH);
    fl = liquid_fraction<N>(P, phi, rhoH);
}

// phi_p, rho and psi of a cell (what its neighbours' stencils read), and rho H.
template <int N, class Pr>
__device__ __forceinline__ void halo_moments(const KParams& P, const PopView<Pr>& pin,
                                             const typename Pr::TA* __restrict__ ain, unsigned c,
                                             val_t<typename Pr::R> (&phi)[N], val_t<typename Pr::R>& rho,
                                             val_t<typename Pr::R>& psi, val_t<typename Pr::R>& rhoH)
{
    const GlobalLoader<Pr> ld{P, pin, ain};
    val_t<typename Pr::R> fl;
    cell_moments<N, Pr>(P, ld, c, phi, rhoH, fl);
    mix_rho_psi<N>(P, phi, fl, rho, psi);
}

// Push one post-collision population q_j of species s at node (x, y) into set B.
// Periodic sides wrap; a population leaving through an x wall is reflected into the
// node's own opposite slot (half-way bounce-back); through a y wall likewise, except
// the enthalpy populations at a Dirichlet wall (their incoming slots are filled by the
// ghost rule); through an outflow side it is dropped.
template <int J, int KIND, class Pr>
__device__ __forceinline__ void push(const KParams& P, const PopView<Pr>& out, int s, int x, int y, step_val<Pr> q)
{
    int tx = x + cx(J), ty = y + cy(J);
    bool xo = false, yo = false;
    if (cx(J) != 0 && (unsigned)tx >= (unsigned)P.nx) {
        if (P.bc[0] == PERIODIC) tx = tx < 0 ? tx + P.nx : tx - P.nx;
        else xo = true;
    }
    if (cy(J) != 0 && (unsigned)ty >= (unsigned)P.ny) {
        if (P.bc[2] == PERIODIC) ty = ty < 0 ? ty + P.ny : ty - P.ny;
        else yo = true;
    }
    const unsigned own = (unsigned)y * (unsigned)P.nx + (unsigned)x;
    if (!xo && !yo) {
        st_val<Pr, KIND>(P, out, s, J, 0, (unsigned)ty * (unsigned)P.nx + (unsigned)tx, q, 10);
    } else if (xo) {
        st_val<Pr, KIND>(P, out, s, opp(J), 0, own, q, 11);
    } else {
        const int side = ty < 0 ? 2 : 3;
        if (P.bc[side] == WALL && !(KIND == KIND_H && P.tbc[side] == DIRICHLET))
            st_val<Pr, KIND>(P, out, s, opp(J), 0, own, q, 12);
    }
}

// Extra write of a boundary-row rule: value v into slot J of node (x + c_J, y),
// same row; skipped when that node is beyond an x wall.
template <int J, int KIND, class Pr>
__device__ __forceinline__ void push_row(const KParams& P, const PopView<Pr>& out, int s, int x, int y,
                                         step_val<Pr> v)
{
    int tx = x + cx(J);
    if (cx(J) != 0 && (unsigned)tx >= (unsigned)P.nx) {
        if (P.bc[0] != PERIODIC) return;
        tx = tx < 0 ? tx + P.nx : tx - P.nx;
    }
    st_val<Pr, KIND>(P, out, s, J, 0, (unsigned)y * (unsigned)P.nx + (unsigned)tx, v, 13);
}

// push_row for a direction j known at run time, whose x component is dx.
template <int KIND, class Pr>
__device__ __forceinline__ void push_row_at(const KParams& P, const PopView<Pr>& out, int s, int j, int dx, int x,
                                            int y, step_val<Pr> v)
{
    int tx = x + dx;
    if (dx != 0 && (unsigned)tx >= (unsigned)P.nx) {
        if (P.bc[0] != PERIODIC) return;
        tx = tx < 0 ? tx + P.nx : tx - P.nx;
    }
    st_val<Pr, KIND>(P, out, s, j, 0, (unsigned)y * (unsigned)P.nx + (unsigned)tx, v, 13);
}

// All nine pushes of one species, plus the outflow copies of the boundary rows.  Two paths,
// chosen per cell by the caller:
//   inside: the cell's row is neither the lattice's first nor its last, and x is periodic or the
//     columns of its tile and their ring lie inside the lattice: every population lands in
//     the neighbour c + c_J with its x taken modulo nx, no boundary rule;
//   otherwise the checks of push() for every population.
template <int KIND, class Pr>
__device__ __forceinline__ void push_species(const KParams& P, const PopView<Pr>& out, int s, int x, int y,
                                             bool inside, const step_val<Pr> (&q)[9])
{
    if (inside) {
        const unsigned nx = (unsigned)P.nx, c = (unsigned)y * nx + (unsigned)x;
        const unsigned cm = x == 0 ? c + (nx - 1) : c - 1, cp = x == P.nx - 1 ? c - (nx - 1) : c + 1;
        st_val<Pr, KIND>(P, out, s, 0, 0, c, q[0], 10);
#pragma unroll
        for (int j = 1; j < 9; ++j)
            st_val<Pr, KIND>(P, out, s, j, cy(j) * P.nx, cx(j) < 0 ? cm : (cx(j) > 0 ? cp : c), q[j], 10);
        return;
    }
    push<0, KIND, Pr>(P, out, s, x, y, q[0]);
    push<1, KIND, Pr>(P, out, s, x, y, q[1]);
    push<2, KIND, Pr>(P, out, s, x, y, q[2]);
    push<3, KIND, Pr>(P, out, s, x, y, q[3]);
    push<4, KIND, Pr>(P, out, s, x, y, q[4]);
    push<5, KIND, Pr>(P, out, s, x, y, q[5]);
    push<6, KIND, Pr>(P, out, s, x, y, q[6]);
    push<7, KIND, Pr>(P, out, s, x, y, q[7]);
    push<8, KIND, Pr>(P, out, s, x, y, q[8]);
    if (y == 0 && P.bc[2] == OUTFLOW) {
        push_row<2, KIND, Pr>(P, out, s, x, y, q[2]);
        push_row<5, KIND, Pr>(P, out, s, x, y, q[5]);
        push_row<6, KIND, Pr>(P, out, s, x, y, q[6]);
    }
    if (y == P.ny - 1 && P.bc[3] == OUTFLOW) {
        push_row<4, KIND, Pr>(P, out, s, x, y, q[4]);
        push_row<7, KIND, Pr>(P, out, s, x, y, q[7]);
        push_row<8, KIND, Pr>(P, out, s, x, y, q[8]);
    }
}

// Resident threads per SM the register allocation must allow (launch bounds): the
// policy's choice, or LBM_OCC_THREADS when a build overrides it for tuning.
#ifdef LBM_OCC_THREADS
#define LBM_OCC(Pr) (LBM_OCC_THREADS)
#else
#define LBM_OCC(Pr) (Pr::OCC_THREADS)
#endif
// Shared-memory elements of type R that step_tile needs: phi_p, rho and psi on the
// tile and its one-cell ring, and (COMPACT policies) rho H and f_l of the tile's cells.
template <int N, int TX, int TY, class Pr>
__host__ __device__ constexpr int tile_smem_elems()
{
    return (N + 2) * (TX + 2) * (TY + 2) + (Pr::COMPACT ? 2 * TX * TY : 0);
}

// What cell_update and cell_update16 read and write of the cell (x, y) of a tile: its stencil
// windows from shared memory (fields of H x W values, the cell at (lx, ly)), its populations and
// lagged values through the loader, its outputs to set B.
template <int N, int H, int W, class Pr, class L, bool BATCH = false>
struct CellIo {
    static constexpr int CALLER = !L::GLOBAL ? CALLER_STAGED : BATCH ? CALLER_BATCH : CALLER_STEP;
    using V = step_val<Pr>;
    using TA = typename Pr::TA;
    const KParams& P;
    const L& ld;
    const V* fields;               // [N + 2][H][W]
    const PopView<Pr>& pout;
    TA* __restrict__ aout;
    const ExportPtrs& ex;
    int lx, ly, x, y;
    bool inside;                   // push_species
    unsigned c;
    typename L::Cell oc;
    // the values of field fi at offset (dx, dy) from the cell
    __device__ __forceinline__ V at(int fi, int dx, int dy) const
    {
        return reinterpret_cast<const V (*)[W]>(fields + fi * H * W)[ly + dy][lx + dx];
    }
    __device__ __forceinline__ void stencil(int fi, V& gx, V& gy, V& lap) const
    {
        const V (*a)[W] = reinterpret_cast<const V (*)[W]>(fields + fi * H * W);
        const V e = a[ly][lx + 1], w = a[ly][lx - 1], n = a[ly + 1][lx], s = a[ly - 1][lx];
        const V ne = a[ly + 1][lx + 1], nw = a[ly + 1][lx - 1], se = a[ly - 1][lx + 1], sw = a[ly - 1][lx - 1];
        grad12(e, w, n, s, ne, nw, se, sw, gx, gy);
        if (fi < N) lap = lap6(a[ly][lx], e, w, n, s, ne, nw, se, sw);
    }
    __device__ __forceinline__ V f(int i) const { return ld.template pop_late<KIND_F>(0, i, oc, 5); }
    __device__ __forceinline__ V g(int p, int i) const { return ld.template pop_late<KIND_G>(1 + p, i, oc, 6); }
    __device__ __forceinline__ V h(int i) const { return ld.template pop_late<KIND_H>(N + 1, i, oc, 7); }
    __device__ __forceinline__ V lag(int a) const { return ld.aux(a, oc, 14); }
    template <int KIND>
    __device__ __forceinline__ void push(int s, const V (&q)[9])
    {
        push_species<KIND, Pr>(P, pout, s, x, y, inside, q);
    }
    __device__ __forceinline__ void put_lag(int a, V v)
    {
        st_plane<TA>(P, aout, a, 0, c, P.aux_elems, 30, (TA)(typename Pr::R)v);
    }
    // Dirichlet wall: ghost behind the half-way wall with T_g = 2 T_w - T, u = 0; its
    // post-collision population is h_eq(ghost) + (1 - 1/tau_h)(h_j - h_eq_j) for the
    // three directions j that enter the boundary row (one code path for both walls:
    // directions (0, sy), (1, sy), (-1, sy), sy = +1 at the bottom, -1 at the top).
    __device__ __forceinline__ int dirichlet_side() const
    {
        return (y == 0 && P.bc[2] == WALL && P.tbc[2] == DIRICHLET)          ? 2
               : (y == P.ny - 1 && P.bc[3] == WALL && P.tbc[3] == DIRICHLET) ? 3
                                                                             : -1;
    }
    __device__ __forceinline__ void dirichlet(const V (&h)[9], V oh1, V Z, V E, V T, V ux, V uy, V uu)
    {
        using K = exact_t<V>;
        const int side = dirichlet_side();
        if (side < 0) return;
        const auto& C = coef<const_t<V>>(P);
        const bool top = side == 3;
        const V vy = top ? -uy : uy;
        const V Eg = (V(C.Tw[side]) * K(2) - T) * C.E_ref;
        const V uu15 = uu * K(-1.5);
        // equilibrium (over w_j) of a moving direction with c_j . u = cu
        auto heq = [&](V cu) { return rfma(Z, rfma(cu * K(4.5), cu, rfma(cu, K(3), uu15)), E); };
        auto value = [&](V hj, V cu, int j) { return rfma(oh1, hj - heq(cu) * wgt_v<V>(j), Eg * wgt_v<V>(j)); };
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 4 : 2, 0, x, y, value(top ? h[4] : h[2], vy, 2));
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 8 : 5, 1, x, y, value(top ? h[8] : h[5], ux + vy, 5));
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 7 : 6, -1, x, y, value(top ? h[7] : h[6], vy - ux, 5));
    }
    // The same in the order of roundings that 16-bit storage keeps (lbm_cell16.cuh).
    __device__ __forceinline__ void dirichlet16(const float (&h)[9], float oh1, float Z, float E, float T, float ux, float uy,
                                                float uu)
    {
        const int side = dirichlet_side();
        if (side < 0) return;
        const Coef<float>& C = P.f;
        const bool top = side == 3;
        const float vy = top ? -uy : uy;
        const float Eg = C.E_ref * (2.0f * C.Tw[side] - T);
        auto heq = [&](float w, float cu) { return w * rfma(Z, rfma(4.5f * cu, cu, rfma(3.0f, cu, -1.5f * uu)), E); };
        const float wa = wgt_r<float>(2), wd = wgt_r<float>(5);
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 4 : 2, 0, x, y, rfma(oh1, (top ? h[4] : h[2]) - heq(wa, vy), wa * Eg));
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 8 : 5, 1, x, y,
                                rfma(oh1, (top ? h[8] : h[5]) - heq(wd, ux + vy), wd * Eg));
        push_row_at<KIND_H, Pr>(P, pout, N + 1, top ? 7 : 6, -1, x, y,
                                rfma(oh1, (top ? h[7] : h[6]) - heq(wd, vy - ux), wd * Eg));
    }
    __device__ __forceinline__ void put_fields(const V (&phi)[N], V T, V H_, V fl, V ux, V uy, V p)
    {
        const long long S = P.S;
#pragma unroll
        for (int q = 0; q < N; ++q)
            if (ex.phi) LBM_ST(P, ex.phi, q * S + c, N * S, 20, (double)phi[q]);
        if (ex.T) LBM_ST(P, ex.T, c, S, 21, (double)T);
        if (ex.H) LBM_ST(P, ex.H, c, S, 22, (double)H_);
        if (ex.fl) LBM_ST(P, ex.fl, c, S, 23, (double)fl);
        if (ex.ux) LBM_ST(P, ex.ux, c, S, 24, (double)ux);
        if (ex.uy) LBM_ST(P, ex.uy, c, S, 25, (double)uy);
        if (ex.p) LBM_ST(P, ex.p, c, S, 26, (double)p);
    }
};

// Ghost values of a tile's ring beyond walls / outflows, by a block of NT threads (all of them
// call it, after a block barrier; it ends with one when it did anything): zero gradient, plus
// the wall's wetting condition for phi_p.  fields: phi_p, rho, psi, each H x W values.  Tiles
// whose ring lies inside the lattice along every non-periodic axis have none.
template <int N, int TX, int TY, int NT, class V>
__device__ __forceinline__ void fill_ghosts(const KParams& P, V* fields, int x0, int y0)
{
    constexpr int W = TX + 2, H = TY + 2;
    V (*s_phi)[H][W] = reinterpret_cast<V (*)[H][W]>(fields);
    V (*s_rho)[W] = reinterpret_cast<V (*)[W]>(fields + N * H * W);
    V (*s_psi)[W] = reinterpret_cast<V (*)[W]>(fields + (N + 1) * H * W);
    const int nx = P.nx, ny = P.ny;
    const bool xper = P.bc[0] == PERIODIC, yper = P.bc[2] == PERIODIC;
    const bool ghosts = (!xper && (x0 < 1 || x0 + TX > nx - 1)) || (!yper && (y0 < 1 || y0 + TY > ny - 1));
    if (!ghosts) return;
    const auto& C = coef<const_t<V>>(P);
    for (int k = threadIdx.x; k < W * H; k += NT) {
        const int lx = k % W, ly = k / W;
        const int gx = x0 + lx - 1, gy = y0 + ly - 1;
        const bool xo = !xper && (gx < 0 || gx >= nx);
        const bool yo = !yper && (gy < 0 || gy >= ny);
        if (!xo && !yo) continue;
        const int sx = xo ? min(max(gx, 0), nx - 1) - x0 + 1 : lx;
        const int sy = yo ? min(max(gy, 0), ny - 1) - y0 + 1 : ly;
        const int wx = xo ? (gx < 0 ? 0 : 1) : -1;
        const int wy = yo ? (gy < 0 ? 2 : 3) : -1;
        V ph[N];
#pragma unroll
        for (int p = 0; p < N; ++p) ph[p] = s_phi[p][sy][sx];
#pragma unroll
        for (int p = 0; p < N; ++p) {
            V corr = V(0.0f);
#pragma unroll
            for (int q = 0; q < N; ++q) {
                if (q == p) continue;
                V cw = V(0.0f);
                if (wx >= 0) cw = cw + V(C.wet[wx][p][q]);
                if (wy >= 0) cw = cw + V(C.wet[wy][p][q]);
                corr = rfma(cw * ph[p], ph[q], corr);
            }
            s_phi[p][ly][lx] = ph[p] + corr;
        }
        s_rho[ly][lx] = s_rho[sy][sx];
        s_psi[ly][lx] = s_psi[sy][sx];
    }
    __syncthreads();
}

// One TX x TY tile (tile column bx, row by) of one time step, run by a block of
// TX * TY threads; smem holds tile_smem_elems<N, TX, TY, Pr>() elements of shared memory.
// Every thread of the block must call it (it holds two block barriers); the caller
// places a block barrier before smem is used again.  RING_TEAM: a block of 2 TX TY threads, whose
// second half evaluates the ring while the first evaluates the tile's cells (not for COMPACT policies).
// BATCH: the caller is a batch's kernel (gdiff_form, lbm_cell16.cuh).
template <int N, int TX, int TY, bool COLLIDE, class Pr, bool RING_TEAM = false, bool BATCH = false, class L>
__device__ __forceinline__ void step_tile_l(const KParams& P, const L& ld, void* __restrict__ pout_base,
                                            typename Pr::TA* __restrict__ aout, const ExportPtrs& ex, int bx, int by,
                                            typename Pr::R* smem)
{
    using V = step_val<Pr>;
    constexpr int W = TX + 2, H = TY + 2, CELLS = TX * TY, NT = RING_TEAM ? 2 * CELLS : CELLS;
    V* fields = reinterpret_cast<V*>(smem);
    V (*s_phi)[H][W] = reinterpret_cast<V (*)[H][W]>(fields);          // [N][H][W]
    V (*s_rho)[W] = reinterpret_cast<V (*)[W]>(fields + N * H * W);    // [H][W]
    V (*s_psi)[W] = reinterpret_cast<V (*)[W]>(fields + (N + 1) * H * W);
    V (*s_own)[NT] = reinterpret_cast<V (*)[NT]>(fields + (N + 2) * H * W);  // COMPACT: rho H, f_l of own cells

    const int nx = P.nx, ny = P.ny;
    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int x0 = bx * TX, y0 = by * TY;
    const int x = x0 + tx, y = y0 + ty;
    static_assert(!(RING_TEAM && Pr::COMPACT), "the one loop over all positions has no ring of its own");
    const bool own_team = !RING_TEAM || tid < CELLS;
    const bool owned = own_team && x < nx && y < ny;
    const bool xper = P.bc[0] == PERIODIC, yper = P.bc[2] == PERIODIC;
    using Cell = typename L::Cell;

    // Position (lx, ly) of the tile-with-ring as a cell of the loader.  In global memory the
    // coordinates are brought into range before anything else (periodic: full modulo, since
    // a tile may be wider / taller than the domain; otherwise clamped, and the position is
    // reported as beyond the domain, to be filled by the ghost rule), so no address outside
    // the planes is ever formed; a staged tile has its ring inside the lattice.
    auto locate = [&](int lx, int ly, Cell& cell) {
        if constexpr (L::GLOBAL) {
            int gx = x0 + lx - 1, gy = y0 + ly - 1;
            bool beyond = false;
            if (gx < 0 || gx >= nx) {
                if (xper) gx = wrap_index(gx, nx);
                else { beyond = true; gx = min(max(gx, 0), nx - 1); }
            }
            if (gy < 0 || gy >= ny) {
                if (yper) gy = wrap_index(gy, ny);
                else { beyond = true; gy = min(max(gy, 0), ny - 1); }
            }
            cell = (unsigned)gy * (unsigned)nx + (unsigned)gx;
            return !beyond;
        } else {
            return ld.locate(lx, ly, cell);
        }
    };
    // phi_p, rho and psi of a position to shared memory
    auto put = [&](int lx, int ly, const V (&ph)[N], V r, V ps) {
#pragma unroll
        for (int p = 0; p < N; ++p) s_phi[p][ly][lx] = ph[p];
        s_rho[ly][lx] = r;
        s_psi[ly][lx] = ps;
    };
    auto share = [&](int lx, int ly, const V (&ph)[N], V fl) {
        V r, ps;
        mix_rho_psi<N>(P, ph, fl, r, ps);
        put(lx, ly, ph, r, ps);
    };
    V phi[N], rhoH, fl;
    Cell16<N> m;   // 16-bit storage
    if constexpr (Pr::COMPACT) {
        // ---- stages A + B: one code path for all (TX + 2)(TY + 2) positions, so that
        // the moments are compiled once; the own cells' rho H and f_l go to shared memory
#pragma unroll 1
        for (int k = tid; k < W * H; k += NT) {
            const int lx = k % W, ly = k / W;
            Cell cell;
            if (!locate(lx, ly, cell)) continue;
            V ph[N], rH, flv;
            cell_moments<N, Pr>(P, ld, cell, ph, rH, flv);
            share(lx, ly, ph, flv);
            const int ox = lx - 1, oy = ly - 1;
            if ((unsigned)ox < (unsigned)TX && (unsigned)oy < (unsigned)TY) {
                const int o = oy * TX + ox;
                s_own[0][o] = rH;
                s_own[1][o] = flv;
            }
        }
    } else {
        // ---- stages A + B: the own cell in registers, then the ring -----------------
        auto halo_at = [&](int lx, int ly) {
            Cell cell;
            if (!locate(lx, ly, cell)) return;
            if constexpr (Pr::QUANT) {
                Cell16<N> r;
                moments16<N, false>(P, ld, cell, r);
                put(lx, ly, r.phi, r.rho, r.psi);
            } else {
                V ph[N], rH, flv;
                cell_moments<N, Pr>(P, ld, cell, ph, rH, flv);
                share(lx, ly, ph, flv);
            }
        };
        if (owned) {
            if constexpr (Pr::QUANT) {
                moments16<N, true>(P, ld, ld.own(x, y, tx, ty), m);
                put(tx + 1, ty + 1, m.phi, m.rho, m.psi);
            } else {
                cell_moments<N, Pr>(P, ld, ld.own(x, y, tx, ty), phi, rhoH, fl);
                share(tx + 1, ty + 1, phi, fl);
            }
        } else if (own_team) {
            halo_at(tx + 1, ty + 1);
        }
        constexpr int NRING = 2 * W + 2 * TY;
        for (int k = RING_TEAM ? tid - CELLS : tid; k < NRING; k += CELLS) {
            if (RING_TEAM && own_team) break;
            int lx, ly;
            if (k < W) { lx = k; ly = 0; }
            else if (k < 2 * W) { lx = k - W; ly = H - 1; }
            else if (k < 2 * W + TY) { lx = 0; ly = k - 2 * W + 1; }
            else { lx = W - 1; ly = k - 2 * W - TY + 1; }
            halo_at(lx, ly);
        }
    }
    __syncthreads();
    fill_ghosts<N, TX, TY, NT>(P, fields, x0, y0);
    if constexpr (!Pr::COH) step_launch_next();
    if (!owned) return;
    if constexpr (Pr::COMPACT) {
#pragma unroll
        for (int p = 0; p < N; ++p) phi[p] = s_phi[p][ty + 1][tx + 1];
        rhoH = s_own[0][tid];
        fl = s_own[1][tid];
    }

    // ---- stages C to G of the own cell ---------------------------------------
    // the push path of this cell (push_species): the same for a row of the tile, so for a
    // warp of a 32-wide tile; only the lattice's first and last rows, and columns at a
    // side that is not periodic, take the general path
    const bool inside = y >= 1 && y <= ny - 2 && (xper || (x0 >= 1 && x0 + TX <= nx - 1));
    const PopView<Pr> pout = pop_view<Pr>(P, pout_base);
    CellIo<N, H, W, Pr, L, BATCH> io{P, ld, fields, pout, aout, ex, tx + 1, ty + 1, x, y, inside, (unsigned)y * (unsigned)nx + (unsigned)x,
                              ld.own(x, y, tx, ty)};
    if constexpr (Pr::QUANT) cell_update16<N, COLLIDE, Pr>(P, io, m);
    else cell_update<N, COLLIDE, Pr>(P, io, phi, rhoH, fl);
}

// One TX x TY tile read from global memory (the loader of the one-cell step).
template <int N, int TX, int TY, bool COLLIDE, class Pr, bool RING_TEAM = false, bool BATCH = false>
__device__ __forceinline__ void step_tile(const KParams& P, const void* __restrict__ pin_base,
                                          void* __restrict__ pout_base, const typename Pr::TA* __restrict__ ain,
                                          typename Pr::TA* __restrict__ aout, const ExportPtrs& ex, int bx, int by,
                                          typename Pr::R* smem)
{
    const GlobalLoader<Pr> ld{P, pop_view<Pr>(P, pin_base), ain};
    step_tile_l<N, TX, TY, COLLIDE, Pr, RING_TEAM, BATCH>(P, ld, pout_base, aout, ex, bx, by, smem);
}

// Tile (bx, by) of block b of a one-dimensional grid of tx * ty tiles.  The tiles on the
// outer ring of the tile grid (those at a side of the lattice: ghost pass, pushes with
// the boundary rules, wrapped reads; about twice the time of an interior tile) take the
// lowest block indices, so that they start in the first wave and overlap the interior
// tiles of later waves instead of finishing last.  Grids of fewer than three tiles along
// an axis are taken in order.
__device__ __forceinline__ void ring_first_tile(int b, int tx, int ty, int& bx, int& by)
{
    if (tx < 3 || ty < 3) {
        bx = b % tx;
        by = b / tx;
        return;
    }
    if (b < 2 * tx) {                       // bottom row, then top row
        bx = b % tx;
        by = b < tx ? 0 : ty - 1;
        return;
    }
    const int k = b - 2 * tx;
    if (k < 2 * (ty - 2)) {                 // left and right columns
        bx = (k & 1) ? tx - 1 : 0;
        by = 1 + (k >> 1);
        return;
    }
    const int m = k - 2 * (ty - 2);         // interior tiles, row by row
    bx = 1 + m % (tx - 2);
    by = 1 + m / (tx - 2);
}

// Tile (bx, by) of block b of a launch over the tile rows `rows` of a tx x ty tile grid:
// all rows in the order of ring_first_tile, or the inner / edge rows in row order.
__device__ __forceinline__ void tile_of_block(int b, int tx, int ty, const TileRows& rows, int& bx, int& by)
{
    if (rows.part == ROWS_ALL) {
        ring_first_tile(b, tx, ty, bx, by);
        return;
    }
    bx = b % tx;
    const int k = b / tx;
    by = rows.part == ROWS_INNER ? rows.lo + k : (k < rows.lo ? k : rows.hi + (k - rows.lo));
}

// One launch = one time step of one lattice (or of some of its tile rows, `rows`), one
// block per tile (a one-dimensional grid, the tiles at the sides first).
template <int N, int TX, int TY, bool COLLIDE, class Pr, bool RING_TEAM = false>
__global__ void __launch_bounds__(TX * TY * (RING_TEAM ? 2 : 1), (LBM_OCC(Pr) + TX * TY - 1) / (TX * TY * (RING_TEAM ? 2 : 1)))
fused_step_kernel(const KParams P, const void* __restrict__ pin_base, void* __restrict__ pout_base,
                  const typename Pr::TA* __restrict__ ain, typename Pr::TA* __restrict__ aout, ExportPtrs ex,
                  TileRows rows)
{
    __shared__ typename Pr::R smem[tile_smem_elems<N, TX, TY, Pr>()];
    int bx, by;
    tile_of_block(blockIdx.x, (P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY, rows, bx, by);
    step_wait_previous();
    step_tile<N, TX, TY, COLLIDE, Pr, RING_TEAM>(P, pin_base, pout_base, ain, aout, ex, bx, by, smem);
}

}  // namespace lbm
