"""f_l of eq. H against the map's own branches, cell by cell, where an FP32 look at the cell can mislead:
two materials that change phase, present only as tails of opposite sign whose latent heats cancel to
between 1e-14 and 1e-6 of themselves.  Lv = sum phi_p rho_l^p L_p > 0 is then decided by digits that FP32
does not hold, and a cold cell is solid where it holds and liquid where it does not."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _case(T_sol, T_liq):
    nx, ny = 40, 33
    c = W.lateral_pool(n=40)
    c.nx, c.ny = nx, ny
    c.phases[0].update(rho_s=0.9, latent=3.0)
    c.phases[1].update(rho_l=0.9, rho_s=0.8, latent=5.0)
    c.T_sol, c.T_liq = T_sol, T_liq
    r = W.uniform(23, 4 * nx * ny).reshape(4, ny, nx)
    a = 10.0 ** (-9.0 + 7.0 * r[0]) * np.where(r[3] < 0.5, 1.0, -1.0)
    delta = 10.0 ** (-14.0 + 8.0 * r[1]) * np.where(r[2] < 0.5, 1.0, -1.0)
    b = -a * (3.0 / (0.9 * 5.0)) * (1.0 + delta)
    c.phi = np.stack([a, b, 1.0 - a - b])
    c.T = np.full((ny, nx), -0.5)
    c.ux = c.uy = np.zeros((ny, nx))
    return c


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32", "fp16s", "bf16s"])
@pytest.mark.parametrize("T_sol,T_liq", [(0.0, 0.0), (-0.1, 0.2)])
def test_cancelling_tails_take_the_branch_of_the_map(prec, T_sol, T_liq):
    from paper_2603_22902_gb300 import lbm as L
    case = _case(T_sol, T_liq)
    s = L.Solver(case, precision=prec).set_fields()
    F = s.fields_numpy()
    s.close()
    rhoL = [Fraction(ph["rho_l"] * ph["latent"]) for ph in case.phases]
    seen = {0.0: 0, 1.0: 0}
    for y in range(case.ny):
        for x in range(case.nx):
            terms = [Fraction(float(F["phi"][p, y, x])) * rhoL[p] for p in range(case.N)]
            Lv, La = sum(terms), sum(abs(t) for t in terms)
            # the map adds up in FP64: N roundings of 2^-53 of the magnitudes
            if abs(Lv) <= La * Fraction(4, 2 ** 53):
                continue
            want = 0.0 if Lv > 0 else 1.0
            assert F["fl"][y, x] == want, (x, y, float(Lv), float(La))
            seen[want] += 1
    assert min(seen.values()) > 100, seen
