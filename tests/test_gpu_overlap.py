"""Step launches overlap (programmatic stream serialization): queued without a wait between
them they must give what the same steps give when each is waited for, between other work of the
stream (initial state, fields, diagnostics) and replayed from a CUDA graph of the caller."""
import numpy as np
import pytest

from paper_2603_22902_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [("fp16s", lambda: W.sessile_drop(n=256, R=60.0, ny=64)),      # staged
         ("fp16s", lambda: W.sessile_drop(n=203, R=50.0, ny=61)),      # one launch per step, odd sides
         ("fp32", lambda: W.lateral_pool(n=48)),
         ("df64", lambda: W.film(nx=40, ny=33, h0=16.0)),
         ("fp64", lambda: W.film(nx=16, ny=64, h0=32.0)),              # one-warp tiles, a block to an SM
         ("fp64", lambda: W.sessile_drop(n=260, R=60.0, ny=130))]      # 32x8 tiles


@pytest.mark.parametrize("k", range(len(CASES)))
def test_queued_steps_equal_waited_ones(k):
    import torch
    from paper_2603_22902_gb300 import lbm as L
    prec, make = CASES[k]
    a, b = L.Solver(make(), precision=prec), L.Solver(make(), precision=prec)
    out = []
    for s, wait in ((a, False), (b, True)):
        for rep in range(3):
            s.set_fields()
            F = []
            for n in (1, 2, 30):
                for _ in range(n):
                    s.step(1)
                    if wait:
                        torch.cuda.synchronize()
                F.append(s.fields())
        torch.cuda.synchronize()
        out.append([{q: v.cpu().numpy() for q, v in f.items()} for f in F])
        s.close()
    for f, g in zip(*out):
        for q in f:
            assert np.array_equal(f[q], g[q], equal_nan=True), q


@pytest.mark.parametrize("k", range(len(CASES)))
def test_steps_captured_in_a_graph(k):
    import torch
    from paper_2603_22902_gb300 import lbm as L
    prec, make = CASES[k]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = L.Solver(make(), precision=prec, stream=st).set_fields()
        s.step(2)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.step(6)
        for _ in range(3):
            g.replay()
        F = {q: v.cpu().numpy() for q, v in s.fields().items()}
        s.close()
    r = L.Solver(make(), precision=prec).set_fields()
    r.step(20)
    G = r.fields_numpy()
    r.close()
    for q in F:
        assert np.array_equal(F[q], G[q], equal_nan=True), q
