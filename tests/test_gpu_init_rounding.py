"""The initial state (lbm_set_fields) is FP64's, rounded once to the type that is stored, whatever
arithmetic formed it: FP32 values are those of the FP64 policy's state rounded to FP32, 16-bit values
are made from these as the format lays down, and double words hold the FP64 values to their 48 bits."""
import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W
from tests.test_gpu_init import _case

pytestmark = pytest.mark.gpu


def _noisy_drop():
    n = 512
    c = W.sessile_drop(n=n)
    r = W.uniform(5, 3 * n * n, -1.0, 1.0).reshape(3, n, n)
    c.T = c.T + 0.02 * r[0]
    c.ux, c.uy = 1e-3 * r[1], 1e-3 * r[2]
    return c


CASES = {"drop": _noisy_drop, "sharp": lambda: _case("sharp", 200, 133), "mushy": lambda: _case("mushy", 200, 133),
         "above": lambda: _case("above", 200, 133), "tiny": lambda: _tiny()}


def _tiny():
    """Fractions, velocities and temperatures over the magnitudes at which FP32 parts run out of range."""
    c = _case("sharp", 200, 133)
    S = c.nx * c.ny
    e = (np.arange(S) % 150 - 150).reshape(c.ny, c.nx)
    c.phi[0] = np.ldexp(1.0 + c.phi[0], e)
    c.phi[1] = np.ldexp(1.0 + c.phi[1], e[::-1])
    c.phi[2] = 1.0 - c.phi[0] - c.phi[1]
    c.ux, c.uy = np.ldexp(1.0 + 0.3 * c.ux, e - 4), -np.ldexp(1.0 + 0.3 * c.uy, e[:, ::-1] - 4)
    c.T = np.where(np.arange(S).reshape(c.ny, c.nx) % 3 == 0, np.ldexp(1.0 + 0.3 * c.T, e), c.T)
    return c


def _blocks(L, case, prec):
    """Rest block [N + 2, S], moving block [N + 2, 8, S] and lagged planes as they are stored."""
    s = L.Solver(case, precision=prec).set_fields()
    raw = np.frombuffer(s.save_state(), dtype=np.uint8)[8:]
    s.close()
    N, S = case.N, case.nx * case.ny
    tr, tm, ta = {"fp64": ("f8",) * 3, "df64": (np.dtype(("f4", 2)),) * 3, "fp32": ("f4",) * 3, "fp16s": ("f4", "f2", "f4"),
                  "bf16s": ("f4", "u2", "f4")}[prec]
    size = lambda t: np.dtype(t).itemsize
    val = lambda b, t: b.view("f4").reshape(-1, 2) if prec == "df64" else b.view(t)
    a = (N + 2) * S * size(tr)
    b = a + 8 * (N + 2) * S * size(tm)
    return [val(raw[:a], tr), val(raw[a:b], tm), val(raw[b:], ta)]


@pytest.mark.parametrize("name", list(CASES))
def test_fp32_state_is_the_fp64_state_rounded(name):
    from paper_2603_22902_gb300 import lbm as L
    case = CASES[name]()
    for ref, got in zip(_blocks(L, case, "fp64"), _blocks(L, case, "fp32")):
        assert np.array_equal(ref.astype(np.float32), got)


@pytest.mark.parametrize("prec", ["fp16s", "bf16s"])
@pytest.mark.parametrize("name", list(CASES))
def test_16_bit_state_is_made_from_the_fp32_state(name, prec):
    from paper_2603_22902_gb300 import lbm as L
    case = CASES[name]()
    N, S = case.N, case.nx * case.ny
    (r0, m0, a0), (r1, m1, a1) = _blocks(L, case, "fp32"), _blocks(L, case, prec)
    assert np.array_equal(r0, r1) and np.array_equal(a0, a1)
    one = np.float32(1.0)
    w = np.array([1 / 9] * 4 + [1 / 36] * 4, dtype=np.float32)[:, None]
    cp_ref = case.cp_ref if case.cp_ref > 0 else 2 * case.phases[0]["cp_s"] * case.phases[0]["cp_l"] / (
        case.phases[0]["cp_s"] + case.phases[0]["cp_l"])
    m0 = m0.reshape(N + 2, 8, S)
    q = np.concatenate([(m0[:1] * (one / (w * np.float32(1 / 4096)))), m0[1:-1] * (one / w),
                        m0[-1:] * (one / w) * np.float32(1.0 / (case.rho_ref * cp_ref))])
    with np.errstate(over="ignore"):
        if prec == "fp16s":
            want = q.astype(np.float16).reshape(-1)
            assert np.array_equal(want, m1)
        else:
            import torch
            want = torch.from_numpy(q.reshape(-1).copy()).to(torch.bfloat16).float().numpy()
            assert np.array_equal(want, torch.from_numpy(m1.view(np.int16).copy()).view(torch.bfloat16).float().numpy())


@pytest.mark.parametrize("name", list(CASES))
def test_double_words_hold_the_fp64_state(name):
    from paper_2603_22902_gb300 import lbm as L
    case = CASES[name]()
    for ref, got in zip(_blocks(L, case, "fp64"), _blocks(L, case, "df64")):
        v = got[:, 0].astype(np.float64) + got[:, 1]
        # the two roundings of a double to hi + lo: 2^-49 of it, and 2^-150 where lo is below FP32's normal range
        assert np.all(np.abs(v - ref) <= 2.0 ** -49 * np.abs(ref) + 2.0 ** -149)
