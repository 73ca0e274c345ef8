"""The Q field where strain and rotation cancel: FP64 arithmetic for either field type, rounded to it once."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-17, 1e17])
@pytest.mark.parametrize("N,fp64", [(9, False), (32, False), (50, False), (32, True)])
def test_cancelling_strain_and_rotation(N, fp64, scale):
    """u = (F(x + y), -F(x + y), 0) has Q = 0; with a perturbation of 1e-7 what is left lies 1e-7 below the terms.
    Bar: 10 x 2^-53 of the sum of magnitudes (three roundings per product, one per gradient and its own, as the
    differences of FP32 values are exact; four of the sum; two of the scale), for FP64 fields also three roundings
    of each gradient's own terms, and the rounding of the result to the field type."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    build.build()
    from paper_1404_0959_gb300 import fe
    rng = np.random.default_rng(N)
    k = np.arange(N)
    F = rng.standard_normal(N)[(k[:, None] + k[None, :]) % N][None]
    eps = lambda: 1e-7 * rng.standard_normal((N, N, N))  # noqa: E731
    dt = np.float64 if fp64 else np.float32
    u = [(scale * (f + eps())).astype(dt) for f in (F, -F, 0.0 * F)]
    s = fe.Solver([dict(N=N, tau_p=[], Y0=[])], precision=fe.FE_FP64 if fp64 else fe.FE_FP32_MIXED)
    one = np.ones((N, N, N), dtype=dt)
    s.set_state(0, one, u, [])
    q = s.q_criterion(0).cpu().numpy()
    s.close()
    ld = np.longdouble
    ih = ld(1) / (ld(2.0 * math.pi / N))

    def grad(a, axis):  # axis 0, 1, 2 = x, y, z; fields are [z][y][x]
        at = lambda o: np.roll(a.astype(ld), -o, 2 - axis)  # noqa: E731
        return (10 * (at(1) - at(-1)) - (at(2) - at(-2))) * ih / 16, \
            (10 * (abs(at(1)) + abs(at(-1))) + abs(at(2)) + abs(at(-2))) * ih / 16

    g, G = ([[grad(u[c], m)[i] for c in range(3)] for m in range(3)] for i in range(2))
    pairs = [((m, m), (m, m), 0.5) for m in range(3)] + [((a, b), (b, a), 1.0) for a, b in ((0, 1), (0, 2), (1, 2))]
    terms = [w * g[a][b] * g[c][d] for (a, b), (c, d), w in pairs]
    ref, mag = -sum(terms), sum(abs(t) for t in terms)
    rnd = (ld(2) ** -53, ld(2) ** -1075) if fp64 else (ld(2) ** -24, ld(2) ** -150)
    bar = (rnd[0] + ld(2) ** -50) * abs(ref) + rnd[1] + 10 * ld(2) ** -53 * mag
    if fp64:
        bar = bar + 3 * ld(2) ** -53 * sum(w * (abs(g[a][b]) * G[c][d] + G[a][b] * abs(g[c][d]))
                                           for (a, b), (c, d), w in pairs)
    assert np.median(abs(ref) / mag) < 1e-5  # the case is one of cancellation
    assert np.all(abs(q.astype(ld) - ref) <= bar)
