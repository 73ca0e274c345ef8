"""The staged convolution kernel on grids that are no multiple of its tiles (32 x 8 x 4, 16 x 8 x 4 and
16 x 4 x 4 voxels), with levels of odd size and levels smaller than a tile, forward and backward, at the bars of
test_gpu_unet.py (the BF16-matched oracle: 1e-2 per layer, 3e-2 per gradient)."""
import numpy as np
import pytest

from oracle import unet as ounet
from paper_1404_0959_gb300.inputs import smooth_field
from tests import test_gpu_unet as base
from tests.test_gpu_unet import fe  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def problem(fe, N):  # noqa: F811
    s, psi = base.make(fe, N, seed=2)
    P = ounet.init_params(2, seed=4)
    fe.fe_load_preconditioner(s.ctx, base.flat(P))
    r = smooth_field(N, 10, 1.0) + 0.1 * np.random.default_rng(9).standard_normal((N, N, N))
    return s, psi, P, r


@pytest.mark.parametrize("N", [8, 12, 20, 36, 68])
def test_layers_on_ragged_tiles(fe, N):  # noqa: F811
    import torch
    s, psi, P, r = problem(fe, N)
    z = torch.empty((N, N, N), dtype=torch.float32, device="cuda")
    rt = torch.tensor(r, device="cuda")
    fe.fe_precond_apply(s.ctx, 0, rt.data_ptr(), base.DT, z.data_ptr())
    Q = {k: (base.bf16(v) if k.endswith(".W") else v) for k, v in P.items()}
    conv, relu, up2 = ounet.conv, ounet.relu, ounet.up2
    acts, a = {}, base.bf16(base.oracle_input(r, psi, N))
    for name, stride in (("e1a", 1), ("e1b", 1), ("d1", 2), ("e2", 1), ("d2", 2), ("e3", 1)):
        a = acts[name] = base.bf16(relu(conv(a, Q[name + ".W"], Q[name + ".b"], stride)))
    for name, up, skip in (("u2", "e3", "e2"), ("u1", "u2", "e1b")):
        x = np.concatenate([up2(acts[up]), acts[skip]])
        acts[name] = base.bf16(relu(conv(x, Q[name + ".W"], Q[name + ".b"])))
    for l, name in enumerate(base.NAMES[:8]):
        lev, C = base.LEVEL_CH[l]
        n = N >> lev
        g = fe.fe_precond_activation(s.ctx, l, n ** 3 * C).reshape(n, n, n, C).transpose(3, 0, 1, 2)
        assert base.rel(g, acts[name]) < 1e-2, name
    y = fe.fe_precond_activation(s.ctx, 8, N ** 3).reshape(N, N, N)
    assert base.rel(y, conv(acts["u1"], Q["out.W"], Q["out.b"])[0]) < 1e-2
    s.close()


@pytest.mark.parametrize("N", [12, 20, 36])
def test_gradients_on_ragged_tiles(fe, N):  # noqa: F811
    import torch
    s, psi, P, r = problem(fe, N)
    h = 2 * np.pi / N
    rho_r, d0 = ounet.precond_scales(r, base.DT, h)
    e = r / ounet.jacobi_diag(psi, base.DT, h) + rho_r * d0 * smooth_field(N, 11, 1.0)
    rt, et = torch.tensor(r, device="cuda"), torch.tensor(e, device="cuda")
    fe.fe_precond_train_step(s.ctx, 0, rt.data_ptr(), et.data_ptr(), base.DT, 0.0)
    g = base.unflat(fe.fe_get_preconditioner(s.ctx, gradients=True), P)
    t = ounet.training_target(r, e, psi, base.DT, h)
    _, _, G = base.quantised_forward_backward(P, base.oracle_input(r, psi, N), t)
    errs = {n + k: base.rel(g[n + k], G[n + k]) for n in base.NAMES for k in (".W", ".b")}
    assert max(errs.values()) < 3e-2, errs
    s.close()


@pytest.mark.parametrize("N", [16, 28, 44, 52])
def test_weight_gradients_on_staged_tiles(fe, N):  # noqa: F811
    """The staged weight gradients where a grid is smaller than the 16 x 4 x 4 (stride 2: 16 x 4 x 2) voxel tile,
    of odd size (28: 14 and 7; 44: 22 and 11), or leaves remainders along every axis; accumulation in FP32 of the
    same BF16 products, so the bars of the gradients above hold."""
    test_gradients_on_ragged_tiles(fe, N)


def test_parameters_come_back_as_loaded(fe):  # noqa: F811
    """The parameters' way out (padding of the first and last layers left behind, biases between the weights) returns
    what was loaded, bit for bit; before a training step the gradients are zero."""
    s, _, P, _ = problem(fe, 8)
    w = np.random.default_rng(3).standard_normal(fe.fe_preconditioner_size()).astype(np.float32)
    fe.fe_load_preconditioner(s.ctx, w)
    assert np.array_equal(fe.fe_get_preconditioner(s.ctx), w)
    assert not fe.fe_get_preconditioner(s.ctx, gradients=True).any()
    s.close()
