"""The built-in tile depth (chosen from the boxes of a context) against explicit depths: the step's fields do
not depend on it beyond the order of the Krylov sums, and an FP64 context's solves not at all (their tiles
depend on the box alone, so a box iterates the same in any ensemble)."""
import numpy as np
import pytest

from paper_1404_0959_gb300.inputs import random_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fe():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    build.build()
    from paper_1404_0959_gb300 import fe as fe_mod
    return fe_mod


@pytest.mark.parametrize("sizes", [(8,), (21, 40), (96,), (24, 33, 64, 100)])
@pytest.mark.parametrize("fp64", [True, False])
def test_default_depth_matches_an_explicit_one(fe, sizes, fp64):
    """Bars: the per-step ones of the oracle tests (1e-11 FP64, 1e-5 mixed); FP64 iteration counts equal."""
    prec, tol, bar = (fe.FE_FP64, 1e-10, 1e-11) if fp64 else (fe.FE_FP32_MIXED, 1e-8, 1e-5)
    out = []
    for tz in (0, 4):
        s = fe.Solver([dict(N=N, nu=0.005, tau_p=[0.05], Y0=[0.01], seed=N) for N in sizes], precision=prec, p_tol=tol)
        for b, N in enumerate(sizes):
            rho, u, Y, _ = random_fields(N, 1, False, seed=N, mach=0.3, noise=0.02)
            s.set_state(b, rho, u, Y)
        if tz:
            s.set_tiling(tz)
        code, info = s.step(1)
        assert code == fe.FE_OK
        out.append(([s.get_state(b) for b in range(len(sizes))], info))
        s.close()
    for b in range(len(sizes)):
        x, y = out[0][0][b], out[1][0][b]
        for p, q in [(x["rho"], y["rho"]), (x["p"], y["p"])] + list(zip(x["u"] + x["phi"] + x["Y"],
                                                                       y["u"] + y["phi"] + y["Y"])):
            q = q.astype(np.float64)
            assert np.linalg.norm(p - q) <= bar * np.linalg.norm(q)
        if fp64:
            assert out[0][1][b]["iters"] == out[1][1][b]["iters"]
