"""The analysis entry points on one context: their kept work memory and their kernels at the sizes
where tiles, line groups and radices end, against the oracle."""
import math

import numpy as np
import pytest

from oracle import diag as odiag
from oracle import isosurface as oiso
from paper_1404_0959_gb300.inputs import random_fields, smooth_field

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


def test_les_keeps_the_surface_memory(fe):
    """The a-priori LES call between two extractions of one context leaves the second one's work memory alone."""
    import torch
    N = 24
    f = smooth_field(N, 5, 1.0)
    T, _ = oiso.extract(f, 0.1, 2 * math.pi / N)
    s = fe.Solver([dict(N=N, tau_p=[], Y0=[])])
    s.init_state()
    fd = torch.as_tensor(f, device="cuda").contiguous()
    tri = torch.zeros((len(T), 9), dtype=torch.float64, device="cuda")
    n0, a0 = fe.fe_isosurface(s.ctx, 0, fd.data_ptr(), 0.1, tri.data_ptr(), len(T))
    fe.fe_les_apriori(s.ctx, 0, 2, 0.17)
    other = torch.full((64 * N ** 3,), 7.0, device="cuda")  # takes memory that was given back by mistake
    n1, a1 = fe.fe_isosurface(s.ctx, 0, fd.data_ptr(), 0.1, tri.data_ptr(), len(T))
    assert n0 == n1 == len(T) and a0 == a1
    assert float(other.min()) == 7.0 and float(other.max()) == 7.0
    assert np.array_equal(tri.cpu().numpy().reshape(-1, 3, 3), T)
    s.close()


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("N", [8, 9, 12, 21, 27, 32, 40, 48, 54, 64, 96, 128])
def test_diagnostics_at_every_radix_and_ragged_tiles(fe, N, fp64):
    """Sums, Q and the spectrum (N = 2^a 3^b) on grids that end tiles (32 x 8 x 16), groups of eight lines
    and every butterfly (16, 8, 4, 2, 3), fewer and more bins than shells.  The sums, the transform and the
    bins are FP64 for either field type: 1e-12 of the largest bin bounds log2(N) roundings of a transform
    and a sum; Q of FP32 fields is one FP32 rounding of a 46-bit value."""
    rho, u, Y, T = random_fields(N, 2, True, seed=N, noise=0.02)
    dt = np.float64 if fp64 else np.float32
    rho, T = rho.astype(dt), T.astype(dt)
    u, Y = [c.astype(dt) for c in u], [y.astype(dt) for y in Y]
    s = fe.Solver([dict(N=N, tau_p=[0.05, 0.1], Y0=[0.01, 0.02])], closure=fe.FE_FOURIER,
                  precision=fe.FE_FP64 if fp64 else fe.FE_FP32_MIXED)
    s.set_state(0, rho, u, Y, T)
    r8, u8, h = rho.astype(np.float64), [c.astype(np.float64) for c in u], 2 * math.pi / N
    smooth = N & (N - 1) == 0 or N in (9, 12, 27, 48, 54, 96)
    for nbins in ((N // 2, N + 3) if smooth else (0,)):
        ref, got = odiag.diagnostics(r8, u8, h, nbins), s.diagnostics(0, nbins)
        for k in ("ke", "ke_u", "enstrophy", "taylor", "rho_rms"):
            assert abs(got[k] - ref[k]) <= 1e-12 * abs(ref[k]), k
        usq = sum(c * c for c in u8)
        cv = 1.0 / 1.4 / 0.4
        assert abs(got["energy"] / (h ** 3 * np.sum(r8 * (cv * T.astype(np.float64) + 0.5 * usq))) - 1) < 1e-12
        for j in range(2):
            assert abs(got["dust_mass"][j] / (h ** 3 * np.sum(r8 * Y[j].astype(np.float64))) - 1) < 1e-12
        if nbins:
            assert np.max(np.abs(got["spectrum"] - ref["spectrum"])) <= 1e-12 * np.max(ref["spectrum"])
    q = s.q_criterion(0).cpu().numpy().astype(np.float64)
    qr = odiag.q_criterion(u8, h)
    assert np.all(np.abs(q - qr) <= (1e-15 if fp64 else 6e-8) * np.abs(qr) + 1e-12 * np.max(np.abs(qr)))
    s.close()


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("N", [8, 9, 13])
def test_surface_of_noise(fe, N, fp64):
    """White noise cuts cubes in every sign pattern: triangles bit for bit the oracle's, on grids that do and
    do not fill the blocks of 128 cubes, with a level that is no FP32 number and with values equal to it."""
    import torch
    rng = np.random.default_rng(N)
    f = rng.standard_normal((N, N, N))
    if not fp64:
        f = f.astype(np.float32).astype(np.float64)
    f.reshape(-1)[::17] = 0.25
    s = fe.Solver([dict(N=N, tau_p=[], Y0=[])], precision=fe.FE_FP64 if fp64 else fe.FE_FP32_MIXED)
    fd = torch.as_tensor(f, device="cuda", dtype=torch.float64 if fp64 else torch.float32).contiguous()
    for iso in (0.1, 0.25):
        T, area = oiso.extract(f, iso, 2 * math.pi / N)
        tri = torch.zeros((len(T) + 3, 9), dtype=torch.float64, device="cuda")
        n, a = fe.fe_isosurface(s.ctx, 0, fd.data_ptr(), iso, tri.data_ptr(), len(T) + 3)
        assert n == len(T) and abs(a - area) <= 1e-12 * area
        assert np.array_equal(tri[:n].cpu().numpy().reshape(-1, 3, 3), T)
        assert not tri[n:].any()
    s.close()


@pytest.mark.parametrize("W,share", [(1, 1.0), (37, 1.0), (250, 1.0), (700, 1.0), (257, 0.3)])
def test_depth_image_of_small_and_large_triangles(fe, W, share):
    """Depth images bit for bit the oracle's: triangles below a pixel, of a few pixels, of more rows than the
    kernel's row lists hold (24), partly and wholly outside the image."""
    import torch
    N = 9
    f = np.random.default_rng(3).standard_normal((N, N, N))
    h = 2 * math.pi / N
    T, _ = oiso.extract(f, 0.4, h)
    T = np.concatenate([T[:4000 if W < 100 else 70], [[[-1.0, -2.0, 0.5], [9.0, 1.0, 0.1], [2.0, 8.0, 0.3]],     # large, beyond all edges
                            [[50.0, 1.0, 0.1], [51.0, 2.0, 0.1], [50.0, 3.0, 0.1]],    # outside
                            [[1.0, 1.0, 0.1], [2.0, 2.0, 0.1], [3.0, 3.0, 0.1]]]])     # no area
    s = fe.Solver([dict(N=N, tau_p=[], Y0=[])])
    tri = torch.as_tensor(T.reshape(-1, 9), device="cuda").contiguous()
    L = share * (N + 1) * h
    depth = torch.empty((W, W), dtype=torch.float32, device="cuda")
    fe.fe_raster_depth(s.ctx, tri.data_ptr(), len(T), W, L, depth.data_ptr())
    assert np.array_equal(depth.cpu().numpy(), oiso.raster_depth(T, W, L))
    s.close()
