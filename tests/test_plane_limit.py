"""lbm_create refuses a lattice whose planes the kernels' 32-bit byte offsets do not reach: more than 4 GB
to a plane, 2^29 cells of 8 bytes or 2^30 of 4 (validation runs before any CUDA call, so no memory is
asked for).  The largest lattice below each limit passes the check: what stops it here is the missing device."""
import pytest

from paper_2603_22902_gb300 import build as B
from paper_2603_22902_gb300 import lbm
from paper_2603_22902_gb300 import workloads as W


def _code(precision, nx, ny):
    case = W.film(nx=8, ny=16)
    grid, phases, th, bc, num = lbm.make_structs(case, precision)
    grid.nx, grid.ny = nx, ny
    with pytest.raises(lbm.LBMError) as e:
        lbm.lbm_create(grid, case.N, phases, th, bc, num)
    return e.value.code


@pytest.mark.parametrize("precision,log2", [("fp64", 29), ("df64", 29), ("fp32", 30), ("fp16s", 30), ("bf16s", 30)])
def test_planes_beyond_4_gb_are_refused(precision, log2):
    import torch
    B.build()
    assert _code(precision, 1 << 15, (1 << (log2 - 15)) + 1) == lbm.LBM_EINVAL
    if not torch.cuda.is_available():
        assert _code(precision, 1 << 15, 1 << (log2 - 15)) == lbm.LBM_ECUDA
