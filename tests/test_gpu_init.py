"""The initial state (lbm_set_fields) of the policies that form it in double words, against
the FP64 policy's, value by value: every branch of eq. H (liquid, solid, mushy, exactly at
the thresholds, cells without phase-changing material, tails of either sign, and a parameter
set whose solidus value of rho H lies above the liquidus value)."""
import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _case(kind, nx, ny):
    c = W.lateral_pool(n=max(nx, ny, 8))
    c.nx, c.ny = nx, ny
    r = W.uniform(11, 8 * nx * ny).reshape(8, ny, nx)
    c.phi = r[:3] / r[:3].sum(0)
    c.phi[0][r[3] < 0.2] = 0.0            # no phase 0 ...
    c.phi[1][r[3] < 0.1] = 0.0            # ... and none that changes phase at all
    c.phi[1][(r[3] > 0.1) & (r[3] < 0.15)] = -1e-17
    c.phi[0][(r[3] > 0.95)] = 1e-300
    c.ux, c.uy = 0.1 * (r[4] - 0.5), 0.1 * (r[5] - 0.5)
    c.phases[0].update(rho_s=0.9, cp_s=0.7, latent=3.0)
    c.phases[1].update(rho_l=0.01, rho_s=0.012, cp_l=100.0, cp_s=90.0, latent=5.0)
    if kind == "mushy":
        c.T_sol, c.T_liq = -0.1, 0.1
    elif kind == "above":                 # As = rho_s c_s T_sol > Al: large temperatures, c_s > c_l
        c.T_sol, c.T_liq = 300.0, 300.5
        for ph in c.phases[:2]:
            ph.update(cp_s=2.0 * ph["cp_l"], latent=0.5)
    c.T = c.T_liq + (r[6] - 0.5)
    c.T[r[7] < 0.05] = c.T_liq
    c.T[r[7] > 0.95] = c.T_sol
    return c


def _state(L, case, prec):
    s = L.Solver(case, precision=prec).set_fields()
    raw = np.frombuffer(s.save_state(), dtype=np.uint8)[8:]
    s.close()
    N, S = case.N, case.nx * case.ny
    tr, tm, ta = {"fp64": (8, 8, 8), "df64": (8, 8, 8), "fp32": (4, 4, 4), "fp16s": (4, 2, 4)}[prec]

    def val(b, size):
        if prec == "df64":
            v = b.view(np.float32).reshape(-1, 2).astype(np.float64)
            return v[:, 0] + v[:, 1]
        return b.view({8: np.float64, 4: np.float32, 2: np.float16}[size]).astype(np.float64)

    a, b = (N + 2) * S * tr, 8 * (N + 2) * S * tm
    rest = val(raw[:a], tr).reshape(N + 2, 1, S)
    move = val(raw[a:a + b], tm).reshape(N + 2, 8, S)
    if prec == "fp16s":
        w = np.array([1 / 9] * 4 + [1 / 36] * 4)[:, None]
        E = case.rho_ref * case.cp_ref
        move = move * np.stack([w / 4096.0] + [w] * N + [w * E])
    return np.concatenate([rest, move], 1), val(raw[a + b:], ta).reshape(3 + 2 * N, S)


@pytest.mark.parametrize("prec", ["df64", "fp32", "fp16s"])
@pytest.mark.parametrize("kind", ["sharp", "mushy", "above"])
@pytest.mark.parametrize("size", [(3, 3), (40, 33)])
def test_initial_state_is_the_fp64_one(prec, kind, size):
    from paper_2603_22902_gb300 import lbm as L
    case = _case(kind, *size)
    ref, got = _state(L, case, "fp64"), _state(L, case, prec)
    # one rounding to the stored type, and a chain of at most 16 double-word operations, each
    # within 4 2^-48 of the largest value of the species
    unit = {"df64": 2.0 ** -48, "fp32": 2.0 ** -24, "fp16s": 2.0 ** -11}[prec] * (1.0 + 2.0 ** -9)
    for k, (a, b) in enumerate(zip(ref, got)):
        scale = np.abs(a).max(axis=tuple(range(1, a.ndim)), keepdims=True)
        floor = 2.0 ** -24 * np.array([1 / 4096.0] + [1.0] * (case.N + 1))[:, None, None] if prec == "fp16s" and k == 0 else 0.0
        assert np.all(np.abs(a - b) <= unit * np.abs(a) + 64 * 2.0 ** -48 * scale + floor), (k, np.abs(a - b).max())


@pytest.mark.parametrize("prec", ["df64", "fp32"])
def test_inputs_of_every_magnitude_and_at_rounding_ties(prec):
    """(phi_0 u)' with phi_0 = 1 is the input u: zeros of either sign, the powers of two around the range that
    integer instructions convert (2^-70 ... 2^126 is beyond any velocity; up to 2^-4 here), values half-way between
    two FP32 numbers, one bit beside them, and values whose rounding carries into the exponent."""
    case = _case("sharp", 40, 33)
    S = case.nx * case.ny
    case.phi = np.zeros_like(case.phi)
    case.phi[0] = 1.0
    e = np.arange(S) % 140 - 143                             # 2^-143 ... 2^-4
    one = np.float64(1.0).view(np.int64)
    low = np.array([0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff, 0x30000000, 0xfffffffffffff, 0xffffff0000000])
    m = (one + low[np.arange(S) % len(low)]).view(np.float64)
    u = np.ldexp(m, e) * np.where(np.arange(S) % 2, -1.0, 1.0)
    u[::50] = 0.0
    u[1::50] = -0.0
    case.ux, case.uy = u.reshape(case.ny, case.nx), u[::-1].reshape(case.ny, case.nx).copy()
    from paper_2603_22902_gb300 import lbm as L
    _, aux = _state(L, case, prec)
    # the pair of words holds the input to 2^-48, the product with 1 adds 4 2^-48; FP32 rounds once; words below
    # 2^-126 are multiples of 2^-149
    unit = {"df64": 5 * 2.0 ** -48, "fp32": 2.0 ** -24 * (1.0 + 2.0 ** -9)}[prec]
    for got, want in ((aux[3], case.ux), (aux[3 + case.N], case.uy)):
        want = want.reshape(-1)
        assert np.all(np.abs(got - want) <= unit * np.abs(want) + 2.0 ** -147), np.abs(got - want).max()
