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


@pytest.mark.parametrize("transonic", [False, True])
@pytest.mark.parametrize("N", [8, 9, 24, 45, 53, 67, 84, 86])
def test_one_launch_solves(fe, N, transonic):
    """The FP64 solves of small boxes in one launch (up to 8 units of 256 cells per block, 4 for BiCGStab; larger
    boxes run kernel by kernel) against the oracle's: ragged last units, one to many units per block, both sides of
    the limits.  A solution to residual 1e-12 of a system of condition number below 10 is within 1e-11; iteration
    counts agree up to the rounding of the stopping test."""
    import torch
    from oracle import krylov, piso
    from paper_1404_0959_gb300.inputs import random_vector
    rho, u, Y, _ = random_fields(N, 1, False, seed=N, mach=0.3, noise=0.01)
    s = fe.Solver([dict(N=N, nu=0.005, tau_p=[0.05], Y0=[0.01])], transonic=transonic,
                  solver=fe.FE_BICGSTAB_JACOBI if transonic else fe.FE_PCG_JACOBI)
    s.set_state(0, rho, u, Y)
    prm = piso.Params(N=N, nu=0.005, transonic=transonic, p_tol=1e-12)
    st = piso.make_state(prm, rho, u, Y)
    psi = piso.compressibility(prm, st["rho"], st["p"])
    dt = piso.time_step(prm, st["u"], float("inf"))
    M, diag = piso.helmholtz(prm, psi, dt, st["u"] if transonic else None)
    b = random_vector(N, 100 + N)
    xr, itr, _, _ = (krylov.bicgstab if transonic else krylov.pcg)(M, b, diag, 1e-12, 500)
    bd = torch.as_tensor(b, device="cuda")
    for _ in range(2):  # the second call finds the first one's packets and vectors
        code, x, info = s.solve_pressure(0, bd, dt, 1e-12, 500)
        assert code == fe.FE_OK and abs(info.iters - itr) <= 1 and info.rel_res_true <= 2e-12
        x = x.cpu().numpy()
        assert np.linalg.norm(x - xr) <= 1e-11 * np.linalg.norm(xr)
    code, x, info = s.solve_pressure(0, bd, dt, 1e-12, 2)  # the cap is a verdict, not a hang
    assert code == fe.FE_ERR_NOT_CONVERGED and info.iters == 2
    code, x, info = s.solve_pressure(0, torch.zeros_like(bd), dt, 1e-12, 50)
    assert code == fe.FE_OK and info.iters == 0 and not x.any()
    s.close()


@pytest.mark.parametrize("N", [10, 22, 30, 34, 66])
@pytest.mark.parametrize("kind", ["barotropic", "fourier", "two-way", "two-fluid"])
def test_rings_on_grids_of_8_byte_chunks(fe, N, kind):
    """FP32 steps on even N that are no multiple of four (ring kernels with 8-byte copies: tiles narrower than
    the box, ragged, wrapping more than once) against the oracle at the mixed-precision bar."""
    from oracle import piso
    nd = 2
    rho, u, Y, T = random_fields(N, nd, kind == "fourier", seed=N, mach=0.2, noise=0.01)
    f32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)  # noqa: E731
    rho, u, Y = f32(rho), [f32(c) for c in u], [f32(y) for y in Y]
    T = f32(T) if T is not None else None
    kw = dict(closure=1 if kind == "fourier" else 0, coupling=1 if kind == "two-way" else 0,
              dust_model=1 if kind == "two-fluid" else 0)
    prm = piso.Params(N=N, nu=0.005, tau_p=[0.05, 0.1], Y0=[0.01, 0.02], p_tol=1e-10, **kw)
    ref, _ = piso.step(prm, piso.make_state(prm, rho, u, Y, T))
    s = fe.Solver([dict(N=N, nu=0.005, tau_p=[0.05, 0.1], Y0=[0.01, 0.02])], precision=fe.FE_FP32_MIXED, p_tol=1e-8,
                  solver=fe.FE_PCG_POLY, **kw)
    s.set_state(0, rho, u, Y, T)
    code, _ = s.step(1)
    assert code == fe.FE_OK
    got = s.get_state(0)
    pairs = [(got["rho"], ref["rho"]), (got["p"], ref["p"])] + list(zip(got["u"] + got["phi"] + got["Y"],
                                                                         ref["u"] + ref["phi"] + ref["Y"]))
    if kind == "fourier":
        pairs.append((got["T"], ref["T"]))
    if kind == "two-fluid":
        pairs += [(a, b) for j in range(nd) for a, b in zip(got["V"][j], ref["V"][j])]
    for a, b in pairs:
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
    s.close()
