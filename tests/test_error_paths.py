"""The library's host code when a call fails or a kernel gives up a bounded wait, on the CPU: its objects linked with
a stand-in for the CUDA runtime (fake_cudart.cpp) whose kernels do nothing but call a hook."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1404_0959_gb300 import build as fe_build
from paper_1404_0959_gb300 import fe

HERE = os.path.dirname(os.path.abspath(__file__))
HOOK = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.c_uint, ctypes.c_uint, ctypes.c_uint, ctypes.c_size_t,
                        ctypes.POINTER(ctypes.c_void_p))


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    fe_build.build()
    objs = [os.path.join(fe_build.BUILD, s.replace(".cu", ".o")) for s in fe_build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        fe_build.build(force=True)
    path = str(tmp_path_factory.mktemp("fake") / "libfe_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp")] + objs, check=True)
    lib = fe.load_library(path)
    lib.fake_find.restype = ctypes.c_void_p
    lib.fake_find.argtypes = [ctypes.c_size_t]
    lib.fake_room.restype = ctypes.c_size_t
    lib.fake_room.argtypes = [ctypes.c_void_p]
    lib.fake_allocations.restype = ctypes.c_size_t
    lib.fake_fail_alloc.argtypes = [ctypes.c_long]
    return lib


class Fake:
    """Control of the stand-in: kernels launched so far, and effects by a part of the kernel's name."""

    def __init__(self, lib):
        self.lib, self.kernels, self.effects = lib, [], {}
        self._hook = HOOK(self._call)
        lib.fake_hook(self._hook)

    def _call(self, name, gx, gy, gz, smem, args):
        name = name.decode()
        self.kernels.append(name)
        for part, effect in self.effects.items():
            if part in name:
                effect(name, gx, args)

    def ran(self, part):
        return any(part in k for k in self.kernels)

    def fail(self, call=""):
        self.lib.fake_fail_call(call.encode())


@pytest.fixture
def fake(library, monkeypatch):
    monkeypatch.setattr(fe, "_lib", library)
    f = Fake(library)
    yield f
    library.fake_hook(HOOK())
    library.fake_fail_alloc(-1)
    f.fail()
    library.cudaGetLastError()
    assert library.fake_allocations() == 0


def solver(sizes=(24,), **kw):
    return fe.Solver([dict(N=N, tau_p=[0.05], Y0=[0.01]) for N in sizes], stream=0, **kw)


def pointer(args, i):
    """Value of a kernel's pointer argument i."""
    return ctypes.cast(args[i], ctypes.POINTER(ctypes.c_void_p))[0]


def scalar_slot(name):
    """Index of a box scalar and the number of them, from the header's enumeration."""
    import re
    text = open(os.path.join(fe_build.CSRC, "fe_internal.cuh")).read()
    body = re.sub(r"//[^\n]*", "", re.search(r"enum[^{]*\{([^}]*SC_KERR[^}]*)\}", text).group(1))
    items, n = {"MAXD": fe.FE_MAX_DUST}, 0
    for it in filter(None, (t.strip() for t in body.split(","))):
        key, _, val = it.partition("=")
        n = eval(val, {}, dict(items)) if val else n
        items[key.strip()] = n
        n += 1
    return items[name], items["NSC"]


def solve(s, N, tol=1e-8, maxit=3):
    b, x = np.zeros(N ** 3), np.zeros(N ** 3)
    info = fe.fe_solve_info()
    return fe.lib().fe_solve_pressure(s.ctx, 0, b.ctypes.data, x.ctypes.data, 0.1, tol, maxit, ctypes.byref(info))


@pytest.mark.parametrize("transonic", [False, True])
def test_solve_reports_a_wait_that_ran_out(fake, transonic):
    """A block of the one-launch solve that gives up sets SC_KERR: fe_solve_pressure says FE_ERR_CUDA, not that the
    solve did not converge, and puts the step scalars back."""
    kerr, nsc = scalar_slot("SC_KERR")
    s = solver(transonic=transonic, solver=fe.FE_BICGSTAB_JACOBI if transonic else fe.FE_PCG_JACOBI)
    sc = ctypes.cast(fake.lib.fake_find(nsc * 8), ctypes.POINTER(ctypes.c_double))

    def give_up(*_):
        sc[kerr] = 1.0

    before = [sc[q] for q in range(nsc)]
    fake.effects = {"kc_bicg" if transonic else "kc_cg": give_up}
    assert solve(s, 24) == fe.FE_ERR_CUDA
    assert fake.ran("kc_")
    assert [sc[q] for q in range(nsc)] == before
    fake.effects = {}
    assert solve(s, 24) == fe.FE_ERR_NOT_CONVERGED  # kernels that do nothing converge to nothing
    s.close()


class TcConvArgs(ctypes.Structure):
    _fields_ = [("s0", ctypes.c_void_p), ("s1", ctypes.c_void_p), ("c0", ctypes.c_int), ("c1", ctypes.c_int),
                ("m0", ctypes.c_int), ("m1", ctypes.c_int), ("No", ctypes.c_int), ("W", ctypes.c_void_p),
                ("bias", ctypes.c_void_p), ("out", ctypes.c_void_p), ("out32", ctypes.c_void_p),
                ("relu", ctypes.c_int), ("err", ctypes.c_void_p)]


def learned(precision):
    s = fe.Solver([dict(N=128, tau_p=[], Y0=[])], stream=0, solver=fe.FE_FCG_LEARNED, precision=precision)
    w = np.zeros(fe.lib().fe_preconditioner_size(), dtype=np.float32)
    assert fe.lib().fe_load_preconditioner(s.ctx, w.ctypes.data, w.size) == fe.FE_OK
    return s


def give_up_convolution(name, gx, args):
    err = ctypes.cast(args[0], ctypes.POINTER(TcConvArgs))[0].err
    ctypes.cast(err, ctypes.POINTER(ctypes.c_int))[0] = 1


def train(s):
    r = np.zeros(128 ** 3, dtype=np.float32)
    loss = ctypes.c_double()
    return fe.lib().fe_precond_train_step(s.ctx, 0, r.ctypes.data, r.ctypes.data, 0.1, 1e-3, ctypes.byref(loss))


def one(i):
    def effect(name, gx, args):
        ctypes.cast(pointer(args, i), ctypes.POINTER(ctypes.c_double))[0] = 1.0
    return effect


def test_training_step_with_an_unfinished_convolution(fake):
    """No weight is updated from activations of a convolution that gave up; the step fails, the next does not."""
    s = learned(fe.FE_FP32_MIXED)
    sums = {"k_sumsq": one(2), "k_target": one(6)}  # the norms of the residual and of the target
    fake.effects = dict(sums, k_conv_ring=give_up_convolution)
    assert train(s) == fe.FE_ERR_CUDA
    assert fake.ran("k_conv_ring") and not fake.ran("k_adam")
    fake.effects = sums
    assert train(s) == fe.FE_OK and fake.ran("k_adam")
    s.close()


@pytest.mark.parametrize("what", ["solve", "step"])
def test_learned_solve_with_an_unfinished_convolution(fake, what):
    """The flag of a convolution that gave up fails the solve or step that ran it, and no later call."""
    s = learned(fe.FE_FP64)

    def running(name, gx, args):  # one box starts its solve
        ctypes.cast(pointer(args, 3), ctypes.POINTER(ctypes.c_int))[0] = 1

    call = (lambda: solve(s, 128, maxit=1)) if what == "solve" else (lambda: fe.lib().fe_step(s.ctx, 1, None))
    fake.effects = {"k_cg_init": running, "k_conv_ring": give_up_convolution}
    assert call() == fe.FE_ERR_CUDA and fake.ran("k_conv_ring")
    fake.effects = {}
    assert call() == (fe.FE_ERR_NOT_CONVERGED if what == "solve" else fe.FE_OK)
    r = np.zeros(128 ** 3)
    z = np.zeros(128 ** 3, dtype=np.float32)
    assert fe.lib().fe_precond_apply(s.ctx, 0, r.ctypes.data, 0.1, z.ctypes.data) == fe.FE_OK
    s.close()


def test_autotune_reports_a_wait_that_ran_out(fake):
    """A trial step whose solve gives up fails fe_autotune, which puts the scalars back; the next step runs."""
    kerr, nsc = scalar_slot("SC_KERR")
    s = solver()
    sc = ctypes.cast(fake.lib.fake_find(nsc * 8), ctypes.POINTER(ctypes.c_double))

    def give_up(*_):
        sc[kerr] = 1.0

    fake.effects = {"kc_cg": give_up}
    assert fe.lib().fe_autotune(s.ctx, 1, None) == fe.FE_ERR_CUDA and fake.ran("kc_cg")
    fake.effects = {}
    assert fe.lib().fe_step(s.ctx, 1, None) == fe.FE_OK
    assert fe.lib().fe_autotune(s.ctx, 1, None) == fe.FE_OK
    s.close()


def test_shared_memory_limits_do_not_follow_the_box(fake):
    """The limit of a kernel's dynamic shared memory is one value per device: a context of small boxes must not lower
    what a launch of a large one, on another thread, has just allowed."""
    def use(N):
        s = fe.Solver([dict(N=N, tau_p=[], Y0=[])], stream=0, solver=fe.FE_FCG_LEARNED, precision=fe.FE_FP32_MIXED)
        w = np.zeros(fe.lib().fe_preconditioner_size(), dtype=np.float32)
        assert fe.lib().fe_load_preconditioner(s.ctx, w.ctypes.data, w.size) == fe.FE_OK
        r, loss = np.zeros(N ** 3, dtype=np.float32), ctypes.c_double()
        assert fe.lib().fe_precond_train_step(s.ctx, 0, r.ctypes.data, r.ctypes.data, 0.1, 1e-3,
                                              ctypes.byref(loss)) == fe.FE_OK
        spec, d = np.zeros(8), fe.fe_diag()
        assert fe.lib().fe_diagnostics(s.ctx, 0, ctypes.byref(d), spec.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                                       8) == fe.FE_OK
        assert fe.lib().fe_init_state(s.ctx, 0, fe.FE_INIT_SPECTRAL) == fe.FE_OK
        s.close()
        return {k: fake.lib.fake_limit(k.encode()) for k in set(fake.kernels)}

    fake.effects = {"k_sumsq": one(2), "k_target": one(6)}
    for large, small in ((128, 24), (256, 128)):
        a = use(large)
        b = use(small)
        assert any(v > 48 * 1024 for v in a.values())
        assert all(b[k] >= v for k, v in a.items() if k in b), [(k, v, b[k]) for k, v in a.items() if b.get(k, v) < v]


def test_refused_launches_are_not_taken_for_done(fake):
    """A convolution whose launch is refused runs in the next form that serves the layer; a refused weight-gradient
    launch fails the step before any weight moves."""
    s = learned(fe.FE_FP32_MIXED)
    fake.effects = {"k_sumsq": one(2), "k_target": one(6)}
    assert train(s) == fe.FE_OK
    ring = next(k for k in fake.kernels if "k_conv_ringILi16" in k)
    staged = [sum("k_conv_st" in k for k in fake.kernels)]
    fake.kernels.clear()
    fake.fail(ring)
    assert train(s) == fe.FE_OK
    staged.append(sum("k_conv_st" in k for k in fake.kernels) + sum("k_conv_ringILi16" in k for k in fake.kernels))
    assert ring not in fake.kernels and staged[1] > staged[0]
    wgrad = next(k for k in fake.kernels if "k_wgrad" in k)
    fake.kernels.clear()
    fake.fail(wgrad)
    assert train(s) == fe.FE_ERR_CUDA and not fake.ran("k_adam")
    fake.fail("cudaFuncSetAttribute")
    fake.lib.fake_forget_limits()
    assert train(s) == fe.FE_ERR_CUDA and not fake.ran("k_adam")
    s.close()


@pytest.mark.parametrize("solver_id,N0", [(fe.FE_PCG_JACOBI, 256), (fe.FE_PCG_POLY, 128)])
def test_streamed_cg_beside_a_smaller_context(fake, solver_id, N0):
    """A context created for smaller boxes leaves the streamed CG kernels of a living one their shared memory."""
    def iterate(name, gx, args):  # a box starts its refined solve, and nothing ends it but the caps
        for q in (3, 4):
            ctypes.cast(pointer(args, q), ctypes.POINTER(ctypes.c_int))[0] = 1

    a = solver((N0,), precision=fe.FE_FP32_MIXED, solver=solver_id)
    b = solver((64,), precision=fe.FE_FP32_MIXED, solver=solver_id)
    fake.effects = {"k_refine_start": iterate}
    for s, N in ((a, N0), (b, 64), (a, N0)):
        fake.kernels.clear()
        x = np.zeros(N ** 3, dtype=np.float32)
        info = fe.fe_solve_info()
        rc = fe.lib().fe_solve_pressure(s.ctx, 0, x.ctypes.data, x.ctypes.data, 0.1, 1e-8, 2, ctypes.byref(info))
        assert fake.ran("kb_cg_") and fake.lib.fake_pending_error() == 0
        assert rc == fe.FE_ERR_NOT_CONVERGED
    a.close()
    b.close()


@pytest.mark.parametrize("solver_id", [fe.FE_PCG_JACOBI, fe.FE_BICGSTAB_JACOBI])
def test_without_one_launch_solves(fake, solver_id):
    """A failed occupancy query, or no memory for the one-launch solves, leaves no error behind and the kernels that
    solved such boxes without them; every other failed allocation refuses the context and gives all memory back."""
    kw = dict(transonic=solver_id == fe.FE_BICGSTAB_JACOBI, solver=solver_id)
    fake.fail("cudaOccupancy")
    s = solver(**kw)
    assert fake.lib.fake_pending_error() == 0
    fake.fail()
    assert solve(s, 24) == fe.FE_ERR_NOT_CONVERGED and not fake.ran("kc_")
    s.close()
    created = 0
    for n in range(64):
        fake.lib.fake_fail_alloc(n)
        try:
            s = solver(**kw)
        except fe.FeError as e:
            assert e.code == fe.FE_ERR_OOM and fake.lib.fake_allocations() == 0
            continue
        if fake.lib.fake_fail_alloc_left() >= 0:  # all allocations made
            s.close()
            break
        created += 1
        assert fake.lib.fake_pending_error() == 0
        fake.kernels.clear()
        assert solve(s, 24) == fe.FE_ERR_NOT_CONVERGED and not fake.ran("kc_")
        s.close()
    assert created == 1 and n > 8


@pytest.mark.parametrize("precision,sizes", [(fe.FE_FP64, (24, 100)), (fe.FE_FP32_MIXED, (64, 64)),
                                             (fe.FE_FP32_MIXED, (24, 40))])
def test_tiling_that_does_not_fit_in_memory(fake, precision, sizes):
    """When an allocation of new work lists fails the context keeps its old ones whole: a step launches no kernel on a
    list that is gone or shorter than its grid."""
    s = solver(sizes, precision=precision)
    lists, bad = [], []

    def check(name, gx, args):
        lists.append(name)
        if not fake.lib.fake_room(pointer(args, 0)) or fake.lib.fake_room(pointer(args, 1)) < gx * 8:
            bad.append(name)

    for n in range(16):
        fake.lib.fake_fail_alloc(n)
        rc = fe.lib().fe_set_tiling(s.ctx, 1 + n % 3)
        done = fake.lib.fake_fail_alloc_left() >= 0
        fake.lib.fake_fail_alloc(-1)
        assert rc == (fe.FE_OK if done else fe.FE_ERR_OOM)
        fake.effects = {"PKNS_6BoxDevEPK4int2": check}
        assert fe.lib().fe_step(s.ctx, 1, None) == fe.FE_OK
        solve(s, sizes[0])
        fake.effects = {}
        assert not bad, (n, bad)
        if done:
            break
    assert done and n >= 2 and len(lists) > 20
    s.close()


def test_refused_allocations_leave_no_error_behind(fake):
    """FE_ERR_OOM of one call is not reported again by the next check, of this context or of another."""
    s = fe.Solver([dict(N=24, tau_p=[], Y0=[])], stream=0, solver=fe.FE_FGMRES_LEARNED, precision=fe.FE_FP32_MIXED)
    w = np.zeros(fe.lib().fe_preconditioner_size(), dtype=np.float32)
    act = np.zeros(24 ** 3 * 16, dtype=np.float32)
    diag, stats, total, area = fe.fe_diag(), fe.fe_les_stats(), ctypes.c_longlong(), ctypes.c_double()
    f = np.zeros(24 ** 3, dtype=np.float32)
    lib, p = fe.lib(), f.ctypes.data

    def create():
        return solver((24,), precision=fe.FE_FP32_MIXED).close() or fe.FE_OK

    calls = [create, lambda: lib.fe_init_state(s.ctx, 0, fe.FE_INIT_SPECTRAL),
             lambda: lib.fe_load_preconditioner(s.ctx, w.ctypes.data, w.size),
             lambda: lib.fe_precond_activation(s.ctx, 0, act.ctypes.data, act.size),
             lambda: lib.fe_diagnostics(s.ctx, 0, ctypes.byref(diag), None, 0),
             lambda: lib.fe_les_apriori(s.ctx, 0, 2, 0.17, ctypes.byref(stats), None),
             lambda: lib.fe_isosurface(s.ctx, 0, p, 0.5, None, 0, ctypes.byref(total), ctypes.byref(area)),
             lambda: lib.fe_raster_depth(s.ctx, None, 0, 16, 1.0, p)]
    for call in calls:
        for n in range(64):
            lib.fake_fail_alloc(n)
            try:
                rc = call()
            except fe.FeError as e:
                rc = e.code
            done = lib.fake_fail_alloc_left() >= 0
            lib.fake_fail_alloc(-1)
            assert rc == (fe.FE_OK if done else fe.FE_ERR_OOM), (calls.index(call), n)
            assert lib.fake_pending_error() == 0, (calls.index(call), n)
            if done:
                break
        assert done and n >= 1
    s.close()


def test_refused_solve_leaves_the_step_scalars(fake):
    """fe_solve_pressure without a loaded network is refused; its tolerance, cap and dt do not stay for the steps."""
    _, nsc = scalar_slot("SC_KERR")
    s = fe.Solver([dict(N=24, tau_p=[], Y0=[])], stream=0, solver=fe.FE_FCG_LEARNED)
    sc = ctypes.cast(fake.lib.fake_find(nsc * 8), ctypes.POINTER(ctypes.c_double))
    before = [sc[q] for q in range(nsc)]
    assert solve(s, 24, tol=0.5) == fe.FE_ERR_UNSUPPORTED
    assert [sc[q] for q in range(nsc)] == before
    s.close()
