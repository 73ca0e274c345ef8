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
