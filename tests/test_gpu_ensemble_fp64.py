"""FP64 boxes of one context against the same boxes alone, bit for bit, where the context's boxes take different
solves (one launch or kernel by kernel), several one-launch groups, or chunks that its total would have set."""
import numpy as np
import pytest

from paper_1404_0959_gb300.inputs import random_fields

pytestmark = pytest.mark.gpu


def _solver(fe, sizes, transonic, graphs):
    s = fe.Solver([dict(N=N, nu=0.005, tau_p=[0.05], Y0=[0.01], seed=N) for N in sizes], p_tol=1e-10,
                  transonic=transonic, solver=fe.FE_BICGSTAB_JACOBI if transonic else fe.FE_PCG_JACOBI)
    for b, N in enumerate(sizes):
        rho, u, Y, _ = random_fields(N, 1, False, seed=N, mach=0.3, noise=0.02)
        s.set_state(b, rho, u, Y)
    if graphs:
        fe.fe_use_graphs(s.ctx, True)
    code, info = s.step(2)
    assert code == fe.FE_OK
    out = [s.get_state(b) for b in range(len(sizes))]
    s.close()
    return out, info


@pytest.mark.parametrize("sizes,transonic", [((64, 64, 84, 24), False), ((96, 64, 100, 40), False),
                                             ((100, 130), False), ((64, 66, 48), True), ((72, 32, 64, 80), True)])
def test_box_equals_its_solo_run(sizes, transonic):
    """One launch holds up to 4864 units of 128 cells in CG (85^3) and 2432 in BiCGStab (67^3): two groups; one-launch
    boxes beside larger ones; larger ones only, of 1 M to 2.2 M cells (chunks of 1024 and 2048 cells alone)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    build.build()
    from paper_1404_0959_gb300 import fe
    solo = [_solver(fe, (N,), transonic, False) for N in sizes]
    for graphs in (False, True):
        got, info = _solver(fe, sizes, transonic, graphs)
        for b in range(len(sizes)):
            a, (r, ri) = got[b], solo[b]
            for x, y in zip([a["rho"], a["p"]] + a["u"] + a["phi"] + a["Y"],
                            [r[0]["rho"], r[0]["p"]] + r[0]["u"] + r[0]["phi"] + r[0]["Y"]):
                assert np.array_equal(x, y), (b, graphs)
            assert info[b]["iters"] == ri[0]["iters"] and info[b]["dt"] == ri[0]["dt"]


@pytest.mark.parametrize("sizes", [(96, 100), (130,)])
def test_explicit_depths(sizes):
    """Kernel-by-kernel FP64 solves on tiles of 7 and 16 planes against the default's 4 (N < 128) and 8: only the order
    of the sums differs (the per-step bar of the oracle tests, 1e-11; the stopping test may turn by one iteration)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    build.build()
    from paper_1404_0959_gb300 import fe
    out = []
    for tz in (0, 7, 16):
        s = fe.Solver([dict(N=N, nu=0.005, tau_p=[0.05], Y0=[0.01], seed=N) for N in sizes], p_tol=1e-10)
        for b, N in enumerate(sizes):
            rho, u, Y, _ = random_fields(N, 1, False, seed=N, mach=0.3, noise=0.02)
            s.set_state(b, rho, u, Y)
        if tz:
            s.set_tiling(tz)
        code, info = s.step(1)
        assert code == fe.FE_OK
        out.append(([s.get_state(b) for b in range(len(sizes))], info))
        s.close()
    for got, info in out[1:]:
        for b in range(len(sizes)):
            for x, y in [(got[b][k], out[0][0][b][k]) for k in ("rho", "p")] + list(zip(got[b]["u"], out[0][0][b]["u"])):
                assert np.linalg.norm(x - y) <= 1e-11 * np.linalg.norm(y)
            assert all(abs(i - j) <= 1 for i, j in zip(info[b]["iters"], out[0][1][b]["iters"]))
