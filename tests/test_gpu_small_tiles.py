"""FP64 steps of small lattices run on 8x4 tiles of one warp (one lattice, and the tiles of a batch
in its per-step form).  Every cell's arithmetic is rounded as written, so the fields must be
those of the 32x8 tiles bit for bit, at sizes around the edges of both shapes and for every kind
of side."""
import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "walls_3x3": lambda: _walls(W.lateral_pool(n=3)),
    "outflow_8x4": lambda: W.film(nx=8, ny=4, h0=2.0),
    "periodic_9x5": lambda: W.perturbed(W.periodic_drop(n=9, R=2.0, ny=5, rho_gas=0.5), seed=2),
    "cap_33x31": lambda: W.sessile_cap(33, 31, 9.0, theta=70.0, ste=0.2),
    "walls_40x40_N3": lambda: _walls(W.lateral_pool(n=40)),
    "cap_152x150": lambda: W.sessile_cap(152, 150, 40.0, theta=70.0, ste=0.2),   # more than four tiles to an SM
    "walls_65x65_N4": lambda: W.impurity_freeze(n=65, n_disks=2),
}


def _walls(c):
    c.wet_cos = np.array([[[0.0, 0.3, 0.1], [-0.3, 0.0, -0.2], [-0.1, 0.2, 0.0]]] * 4)
    return c


def _fields(s, steps):
    s.step(steps)
    return s.fields_numpy()


@pytest.mark.parametrize("name", list(CASES))
def test_small_tiles_equal_the_large_ones(name):
    from paper_2603_22902_gb300 import lbm as L
    a = L.Solver(CASES[name]()).set_fields()
    b = L.Solver(CASES[name](), tile=(32, 8)).set_fields()
    A, B = _fields(a, 25), _fields(b, 25)
    a.close()
    b.close()
    for k in A:
        assert np.array_equal(A[k], B[k], equal_nan=True), k


@pytest.mark.parametrize("tile", [(32, 8), (64, 4), (16, 16)])
def test_batch_of_small_cases_equals_single_runs(tile):
    from paper_2603_22902_gb300 import lbm as L
    cases = W.small_batch()
    solvers = [L.Solver(c).set_fields() for c in cases]
    b = L.Batch(solvers).set_plan(mode="per_step", tiles=[tile] * 4)
    b.step(25)
    b.sync()
    for c, s in zip(cases, solvers):
        F = s.fields_numpy()
        one = L.Solver(c, tile=(32, 8)).set_fields()
        G = _fields(one, 25)
        one.close()
        for k in F:
            assert np.array_equal(F[k], G[k], equal_nan=True), (c.name, k)
    b.close()
