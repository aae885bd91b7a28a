"""The contract of lbm_set_tile where the FP64 map of eq. H runs: with T_sol < T_liq, neither of them 0,
cells freeze through a mushy band whose f_l comes from differences of products.  Every operation is
rounded as written, so the fields after many steps do not depend on the tile shape or on whether a lattice
is stepped alone or in a batch."""
import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _case(N):
    c = W.perturbed(W.film(nx=24, ny=70, h0=40.0), seed=3, amp_u=1e-3) if N == 2 else W.lateral_pool(n=36)
    c.T_sol, c.T_liq = -0.35, 0.15
    c.T = c.T + 0.3
    return c


def _fields(case, prec, **kw):
    from paper_2603_22902_gb300 import lbm as L
    s = L.Solver(case, precision=prec, **kw).set_fields()
    s.step(300)
    F = s.fields_numpy()
    s.close()
    return F


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [2, 3])
def test_shapes_and_batches_give_the_same_bits(N, prec):
    from paper_2603_22902_gb300 import lbm as L
    A = _fields(_case(N), prec)
    assert ((A["fl"] > 0.01) & (A["fl"] < 0.99)).sum() > 20
    others = {str(t): _fields(_case(N), prec, tile=t) for t in ((32, 8), (32, 4), (64, 4), (16, 16))}
    for mode in ("per_step", "persistent"):
        s = L.Solver(_case(N), precision=prec).set_fields()
        b = L.Batch([s]).set_plan(mode=mode)
        b.step(300)
        b.sync()
        others[mode] = s.fields_numpy()
        b.close()
        s.close()
    for name, B in others.items():
        for k in A:
            assert np.array_equal(A[k], B[k], equal_nan=True), (name, k)
