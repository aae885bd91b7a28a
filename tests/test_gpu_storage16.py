"""Runs with 16-bit moving populations, value by value.  A stored value keeps 8 (BF16) or 11 (FP16)
bits, so FP32 roundings in another order send values near a tie to the other neighbour and move the
velocities by 1 to 10 % (BF16) or a few 1e-3 (FP16), no formula being wrong.  The order is part of these
policies' results: the recorded runs (golden/storage16_runs.npz, the fields after the steps below) have
to come back as they are, whatever the shape of the tiles, staged or not."""
import os

import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "storage16_runs.npz")
CASES = {   # case, steps
    "film": (lambda: W.perturbed(W.film(nx=16, ny=64, h0=32.0), seed=7, amp_u=1e-3), 60),
    "drop": (lambda: W.perturbed(W.sessile_drop(n=64, ny=48, R=14.0), seed=7, amp_u=1e-3, amp_T=0.02), 20),
    "odd": (lambda: W.perturbed(W.sessile_drop(n=61, ny=45, R=13.0), seed=7, amp_u=1e-3, amp_T=0.02), 20),
}
FORMS = {"default": {}, "one_launch": dict(staged=False), "64x4": dict(staged=False, tile=(64, 4)),
         "16x16": dict(staged=False, tile=(16, 16))}


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("prec", ["bf16s", "fp16s"])
def test_run_is_the_recorded_one(prec, name, form):
    from paper_2603_22902_gb300 import lbm as L
    case, steps = CASES[name]
    s = L.Solver(case(), precision=prec, **FORMS[form]).set_fields()
    s.step(steps)
    F = s.fields_numpy()
    s.close()
    with np.load(GOLDEN) as want:
        for k in ("phi", "T", "ux", "uy"):
            assert np.array_equal(F[k].astype(np.float32), want[f"{prec}.{name}.{k}"]), k


PHASES = os.path.join(os.path.dirname(__file__), "golden", "storage16_runs_phases.npz")
MORE = {   # three and four phases: case, options, 20 steps; the one-launch and the staged form have recordings of their own
    "janus": (lambda: W.perturbed(W.janus_drop(nx=60, ny=33, R=13.0, mobility=0.1), seed=7, amp_u=1e-3, amp_T=0.02), {}),
    "pool": (lambda: W.perturbed(W.lateral_pool(n=48), seed=7, amp_u=1e-3), dict(staged=False)),
    "pool_staged": (lambda: W.perturbed(W.lateral_pool(n=48), seed=7, amp_u=1e-3), dict(staged=True)),
    "impurity": (lambda: W.perturbed(W.impurity_freeze(n=65, n_disks=2), seed=7, amp_u=1e-3, amp_T=0.02), {}),
}


@pytest.mark.parametrize("name", list(MORE))
@pytest.mark.parametrize("prec", ["bf16s", "fp16s"])
def test_run_of_more_phases_is_the_recorded_one(prec, name):
    from paper_2603_22902_gb300 import lbm as L
    case, options = MORE[name]
    s = L.Solver(case(), precision=prec, **options).set_fields()
    s.step(20)
    F = s.fields_numpy()
    s.close()
    with np.load(PHASES) as want:
        for k in ("ux", "uy"):
            assert np.array_equal(F[k].astype(np.float32), want[f"{prec}.{name}.{k}"]), k
