"""The calls whose time is measured, over the range of sizes and options in which they are used.

Kinds of case (the key ``kind``):

``step``      a program restarts from a saved state, takes some PISO steps and reads the new state:
              ``fe_set_fields`` + ``fe_set_clock``, ``fe_step``, ``fe_get_fields`` on device buffers.  One box
              or an ensemble, FP64 or mixed precision, every closure, dust model and plain solver.
``solve``     one pressure solve with the learned preconditioner (``fe_solve_pressure``).
``train``     one training step of that preconditioner (``fe_precond_train_step``; weights and gradients read).
``analysis``  what a run evaluates every few steps: diagnostics with the spectrum, the Q field, the a-priori
              LES statistics and fields.
``surface``   the iso-surface of a Q field and its depth image.

``exact`` restates each of them in plain torch in 64 bits.
"""
import math

import torch

from paper_1404_0959_gb300 import fe

DEV = "cuda"
GAMMA, PRANDTL = 1.4, 0.7
TAU, LOAD = (0.05, 0.1, 0.3), (0.01, 0.02, 0.02)  # relaxation time and mean mass fraction per dust class
SOLVERS = {"jacobi": fe.FE_PCG_JACOBI, "poly": fe.FE_PCG_POLY, "bicgstab": fe.FE_BICGSTAB_JACOBI}
CS = 0.17  # Smagorinsky constant of the a-priori test


# ---- the cases --------------------------------------------------------------------------------
def _step(name, N, **kw):
    c = dict(kind="step", N=N, sizes="", boxes=1, precision="mixed", closure="barotropic", dust=1, model="equilibrium",
             coupling="one-way", solver="poly", mach=0.2, k0=4.0, nu=0.005, tol=1e-8, steps=1, graphs=True)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest workload: FP64, host-driven as a context starts out, a few steps between reads
        _step("step 32 fp64", 32, precision="fp64", solver="jacobi", tol=1e-10, steps=4, graphs=False),
        # transonic flow on a grid that no fast path asks for: non-symmetric operator, two classes
        _step("step 45 transonic fp64", 45, precision="fp64", solver="bicgstab", mach=0.5, dust=2, tol=1e-10,
              graphs=False),
        # the default precision and solver at an ordinary size
        _step("step 128 fp64", 128, precision="fp64", solver="jacobi", k0=8.0, nu=0.002, tol=1e-8),
        # the 128^3 Fourier-closure workload
        _step("step 128 fourier", 128, closure="fourier", mach=0.5, nu=0.002),
        # dust with its own momentum, an uneven grid
        _step("step 150 two-fluid", 150, model="two-fluid", dust=2, k0=6.0, nu=0.002),
        # the benchmark workload
        _step("step 256", 256, k0=8.0, nu=0.001),
        # the largest workload: 512^3, Fourier closure, three classes
        _step("step 512 fourier", 512, closure="fourier", mach=0.5, k0=8.0, nu=5e-4, dust=3),
        # the ensemble of 64 uneven boxes in one context
        _step("ensemble 64", 0, sizes="32,48,64,96", boxes=64, steps=4),
        # the analysis of a 256^3 state between steps
        dict(name="analysis 256", kind="analysis", N=256, precision="mixed", filter=2, mach=0.2, k0=8.0),
        # the Q iso-surface of the figures and its depth image
        dict(name="surface 192", kind="surface", N=192, precision="mixed", width=2048, level=0.5, mach=0.2, k0=8.0),
        # a solve whose every direction comes from the network
        dict(name="learned solve 128", kind="solve", N=128, precision="mixed", every=1, mach=0.2, k0=8.0, tol=1e-8),
        # one step of training it
        dict(name="train 64", kind="train", N=64, precision="mixed", mach=0.2, k0=4.0, rate=1e-3),
    ]


def draw(rng):
    """One more case: kinds by how often they are called, sizes over their ranges on a log scale."""
    def size(lo, hi, multiple=1):
        return max(multiple, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple)

    mach, k0 = rng.choice((0.2, 0.3, 0.5)), round(rng.uniform(3.0, 8.0), 2)
    what = rng.choice(("step",) * 6 + ("fp64",) * 4 + ("ensemble", "solve", "train", "analysis", "surface"))
    if what == "step":
        model = rng.choice(("equilibrium",) * 4 + ("two-fluid", "two-way"))
        fourier = model == "equilibrium" and rng.random() < 0.4
        N = size(24, 400)
        N = rng.choice((N, N - N % 4, 1 << max(5, N.bit_length() - 1)))
        return _step("", N, closure="fourier" if fourier else "barotropic", mach=mach, k0=k0,
                     model="two-fluid" if model == "two-fluid" else "equilibrium",
                     coupling="two-way" if model == "two-way" else "one-way", dust=rng.choice((1, 1, 2, 3)),
                     solver=rng.choice(("poly", "poly", "jacobi")), nu=rng.choice((0.005, 0.002)),
                     steps=4 if N < 64 else 1, graphs=rng.random() < 0.7)
    if what == "fp64":
        N = size(20, 160)
        transonic = rng.random() < 0.3
        return _step("", N, precision="fp64", mach=mach, k0=k0, dust=rng.choice((0, 1, 2, 3)),
                     closure=rng.choice(("barotropic", "barotropic", "fourier")),
                     solver="bicgstab" if transonic else "jacobi", nu=rng.choice((0.005, 0.002)), tol=1e-10,
                     steps=4 if N < 48 else 1, graphs=rng.random() < 0.4)
    if what == "ensemble":
        sizes = ",".join(str(size(24, 100, rng.choice((1, 4)))) for _ in range(rng.randint(2, 4)))
        return _step("", 0, sizes=sizes, boxes=rng.randint(4, 48), mach=mach, steps=2, graphs=rng.random() < 0.7)
    if what == "solve":
        return dict(kind="solve", N=size(32, 128, 4), precision="mixed", every=rng.choice((0, 1)), mach=mach, k0=k0,
                    tol=1e-8)
    if what == "train":
        return dict(kind="train", N=size(24, 96, 4), precision=rng.choice(("mixed", "fp64")), mach=mach, k0=k0,
                    rate=1e-3)
    if what == "analysis":
        N = rng.choice((36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324))
        return dict(kind="analysis", N=N, precision=rng.choice(("mixed", "mixed", "fp64")), filter=rng.randint(1, 4),
                    mach=mach, k0=k0)
    return dict(kind="surface", N=size(40, 224), precision=rng.choice(("mixed", "mixed", "fp64")),
                width=rng.choice((512, 1000, 1024, 2048)), level=rng.choice((0.25, 0.5, 1.0)), mach=mach,
                k0=k0)


# ---- operators on the periodic grid, [..., z, y, x], direction d = 0, 1, 2 is x, y, z -----------
def _at(f, d, s):
    return torch.roll(f, -s, dims=-1 - d)


def _I4(f, d):
    return (9.0 * (f + _at(f, d, 1)) - _at(f, d, -1) - _at(f, d, 2)) / 16.0


def _G4(f, d, h):
    return (27.0 * (_at(f, d, 1) - f) + _at(f, d, -1) - _at(f, d, 2)) / (24.0 * h)


def _G2(f, d, h):
    return (_at(f, d, 1) - f) / h


def _D1(F, d, h):
    return (F - _at(F, d, -1)) / h


def _D(F, h):
    return _D1(F[0], 0, h) + _D1(F[1], 1, h) + _D1(F[2], 2, h)


def _Gc(f, d, h):
    return _D1(_I4(f, d), d, h)


def _stress(u, mu, h, d, div):
    """tau[m] on the d-faces."""
    t = [mu * (_G4(u[m], d, h) + _I4(_Gc(u[d], m, h), d)) for m in range(3)]
    t[d] = t[d] - mu * (2.0 / 3.0) * _I4(div, d)
    return t


def _div_u(u, h):
    return _Gc(u[0], 0, h) + _Gc(u[1], 1, h) + _Gc(u[2], 2, h)


def _viscous(u, mu, h):
    div = _div_u(u, h)
    out = [0.0, 0.0, 0.0]
    for d in range(3):
        t = _stress(u, mu, h, d, div)
        for m in range(3):
            out[m] = out[m] + _D1(t[m], d, h)
    return out


def _momentum(u, phi, mu, h):
    out = _viscous(u, mu, h)
    for m in range(3):
        for d in range(3):
            out[m] = out[m] - _D1(phi[d] * _I4(u[m], d), d, h)
    return out


# ---- inputs: a decaying turbulent flow, its pressure in balance with it --------------------------
def _noise(N, g):
    return torch.randn((N, N, N), generator=g, device=DEV, dtype=torch.float32).double()


def _modes(N):
    k = torch.fft.fftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
    r = torch.fft.rfftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
    return r[None, None, :], k[None, :, None], k[:, None, None]


def _flow(N, mach, k0, g):
    """rho, u, p (FP64): solenoidal velocity of spectrum k^4 exp(-2 (k/k0)^2), incompressible pressure."""
    kv = _modes(N)
    k2 = kv[0] ** 2 + kv[1] ** 2 + kv[2] ** 2
    keep = (k2 > 0) & (k2 < (N / 2 - 1) ** 2)
    k2s = torch.where(k2 > 0, k2, torch.ones_like(k2))
    shape = torch.where(keep, torch.sqrt(k2s) * torch.exp(-k2s / k0 ** 2), torch.zeros_like(k2))
    uh = [torch.fft.rfftn(_noise(N, g)) * shape for _ in range(3)]
    kd = (kv[0] * uh[0] + kv[1] * uh[1] + kv[2] * uh[2]) / k2s
    u = [torch.fft.irfftn(uh[m] - kv[m] * kd, s=(N, N, N)) for m in range(3)]
    del uh, kd
    scale = mach / math.sqrt(float(sum((c * c).mean() for c in u)))
    u = [c * scale for c in u]
    ph = 0.0
    for i in range(3):
        for j in range(i, 3):
            ph = ph - (1.0 if i == j else 2.0) * kv[i] * kv[j] * torch.fft.rfftn(u[i] * u[j])
    p = torch.fft.irfftn(torch.where(keep, ph / k2s, torch.zeros_like(ph)), s=(N, N, N))
    p = (1.0 / GAMMA + p).clamp_(min=0.3)
    return (GAMMA * p) ** (1.0 / GAMMA), u, p, shape


def _scalar(N, shape, g):
    """A smooth random field of zero mean and unit r.m.s."""
    f = torch.fft.irfftn(torch.fft.rfftn(_noise(N, g)) * shape, s=(N, N, N))
    return f / f.square().mean().sqrt()


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _sizes(case):
    if not case.get("sizes"):
        return [case["N"]]
    s = [int(v) for v in case["sizes"].split(",")]
    return [s[b % len(s)] for b in range(case["boxes"])]


def _box(case, b, N):
    """Parameters of box b; the boxes of an ensemble differ in Mach number and relaxation time."""
    many = bool(case.get("sizes"))
    nd = case.get("dust", 0)
    return dict(N=N, nu=case.get("nu", 0.001), mach_rms=(case["mach"], 0.5)[(b // 4) % 2] if many else case["mach"],
                tau_p=[TAU[j] * (1.0 + 0.05 * b if many else 1.0) for j in range(nd)], Y0=list(LOAD[:nd]),
                k0=case["k0"], seed=b)


def _names(case):
    n = ["rho", "ux", "uy", "uz", "p"] + (["T"] if case.get("closure") == "fourier" else [])
    n += ["phix", "phiy", "phiz"] + ["Y%d" % j for j in range(case.get("dust", 0))]
    if case.get("model") == "two-fluid":
        n += ["V%d%s" % (j, x) for j in range(case["dust"]) for x in "xyz"]
    return n


def _field_id(name):
    if name[0] == "V":
        return fe.FE_V0 + 3 * int(name[1]) + "xyz".index(name[2])
    if name[0] == "Y":
        return fe.FE_Y0 + int(name[1])
    return dict(rho=fe.FE_RHO, ux=fe.FE_UX, uy=fe.FE_UY, uz=fe.FE_UZ, p=fe.FE_P, T=fe.FE_T, phix=fe.FE_PHIX,
                phiy=fe.FE_PHIY, phiz=fe.FE_PHIZ)[name]


def _state(case, seed, b, N):
    """All state fields of box b in the precision of the context."""
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + 7919 * b + 17) % (1 << 62))
    box = _box(case, b, N)
    rho, u, p, shape = _flow(N, box["mach_rms"], case["k0"], g)
    t = _dtype(case)
    st = dict(rho=rho.to(t), ux=u[0].to(t), uy=u[1].to(t), uz=u[2].to(t), p=p.to(t))
    if case.get("closure") == "fourier":
        st["T"] = (GAMMA * p / rho).to(t)
    for d in range(3):
        st["phi" + "xyz"[d]] = (_I4(rho, d) * _I4(u[d], d)).to(t)
    for j in range(case.get("dust", 0)):
        st["Y%d" % j] = (LOAD[j] * (1.0 + 0.1 * _scalar(N, shape, g)).clamp(0.2, 2.0)).to(t)
    if case.get("model") == "two-fluid":
        for j in range(case["dust"]):
            for m in range(3):
                st["V%d%s" % (j, "xyz"[m])] = (u[m] + 0.02 * box["mach_rms"] * _scalar(N, shape, g)).to(t)
    return st


def _solver(case, **kw):
    boxes = [_box(case, b, N) for b, N in enumerate(_sizes(case))]
    return fe.Solver(boxes, precision=fe.FE_FP64 if case["precision"] == "fp64" else fe.FE_FP32_MIXED,
                     gamma=GAMMA, Pr=PRANDTL, p_tol=case.get("tol", 1e-8), **kw)


def _courant_dt(st, N):
    s = st["ux"].double().abs() + st["uy"].double().abs() + st["uz"].double().abs()
    return 0.5 * (2.0 * math.pi / N) / float(s.max())


def _set(s, b, st, names):
    fe.fe_set_fields(s.ctx, b, [_field_id(n) for n in names], [st[n].data_ptr() for n in names], True)


# ---- what a program has in hand before the call ---------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        names, sizes = _names(case), _sizes(case)
        s = _solver(case, closure=fe.FE_FOURIER if case["closure"] == "fourier" else fe.FE_BAROTROPIC,
                    solver=SOLVERS[case["solver"]], transonic=case["solver"] == "bicgstab",
                    dust_model=fe.FE_DUST_TWO_FLUID if case["model"] == "two-fluid" else fe.FE_DUST_EQUILIBRIUM,
                    coupling=fe.FE_COUPLING_TWO_WAY if case["coupling"] == "two-way" else fe.FE_COUPLING_ONE_WAY)
        s.use_graphs(case["graphs"])
        total = sum(N ** 3 for N in sizes)
        new = {n: torch.empty(total, dtype=_dtype(case), device=DEV) for n in names}
        ids, sets, at = [_field_id(n) for n in names], [], 0
        for b, N in enumerate(sizes):
            st = _state(case, seed, b, N)
            sets.append((b, st, [st[n].data_ptr() for n in names], [new[n][at:at + N ** 3].data_ptr() for n in names]))
            at += N ** 3
        return dict(kind=kind, s=s, ids=ids, sets=sets, new=new, steps=case["steps"])
    N = case["N"]
    st = _state(case, seed, 0, N)
    names = _names(case)
    if kind == "analysis":
        s = _solver(case)
        _set(s, 0, st, names)
        return dict(kind=kind, s=s, N=N, m=case["filter"], q=torch.empty((N, N, N), dtype=_dtype(case), device=DEV),
                    les=torch.empty((10, N, N, N), dtype=_dtype(case), device=DEV))
    if kind == "surface":
        s = _solver(case)
        q, iso = _surface_field(case, st)
        return dict(kind=kind, s=s, q=q, iso=iso, tri=torch.zeros((_room(N), 3, 3), dtype=torch.float64, device=DEV),
                    width=case["width"], depth=torch.empty((case["width"],) * 2, dtype=torch.float32, device=DEV))
    s = _solver(case, solver=fe.FE_FCG_LEARNED, learned_every=case.get("every", 1))
    _set(s, 0, st, names)
    r, e, dt = _pair(case, st, seed)
    fe.fe_load_preconditioner(s.ctx, _weights(seed).cpu().numpy())
    return dict(kind=kind, s=s, r=r, e=e, dt=dt, tol=case.get("tol"), rate=case.get("rate"))


# ---- one pass -------------------------------------------------------------------------------------
def run(state):
    s, kind = state["s"], state["kind"]
    if kind == "step":
        for b, _, src, _ in state["sets"]:
            fe.fe_set_fields(s.ctx, b, state["ids"], src, True)
            fe.fe_set_clock(s.ctx, b, 0.0, 0.0)
        code, info = s.step(state["steps"])
        if code != fe.FE_OK:
            raise fe.FeError(code, "fe_step")
        for b, _, _, dst in state["sets"]:
            fe.fe_get_fields(s.ctx, b, state["ids"], dst, True)
        return dict(state["new"], t=[i["t"] for i in info] if len(info) <= 4 else float(sum(i["t"] for i in info)))
    if kind == "solve":
        code, x, _ = s.solve_pressure(0, state["r"], state["dt"], state["tol"], 500)
        if code != fe.FE_OK:
            raise fe.FeError(code, "fe_solve_pressure")
        return x
    if kind == "train":
        loss = fe.fe_precond_train_step(s.ctx, 0, state["r"].data_ptr(), state["e"].data_ptr(), state["dt"],
                                        state["rate"])
        return dict(loss=loss, weights=fe.fe_get_preconditioner(s.ctx),
                    gradients=fe.fe_get_preconditioner(s.ctx, gradients=True))
    if kind == "analysis":
        d = s.diagnostics(0, state["N"] // 2)
        fe.fe_q_criterion(s.ctx, 0, state["q"].data_ptr())
        les = fe.fe_les_apriori(s.ctx, 0, state["m"], CS, state["les"].data_ptr())
        keys = ("ke", "ke_u", "enstrophy", "taylor", "rho_rms", "mass", "energy")
        return dict(diag={k: d[k] for k in keys}, spectrum=d["spectrum"], q=state["q"], les=les, fields=state["les"])
    n, area = fe.fe_isosurface(s.ctx, 0, state["q"].data_ptr(), state["iso"], state["tri"].data_ptr(),
                               state["tri"].shape[0])
    n = min(n, state["tri"].shape[0])
    fe.fe_raster_depth(s.ctx, state["tri"].data_ptr(), n, state["width"], 2.0 * math.pi, state["depth"].data_ptr())
    return dict(n=n, tri=state["tri"], area=area, depth=state["depth"])


def work(case):
    n = sum(N ** 3 for N in _sizes(case))
    word = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "step":  # state in, state out; stencils, and about eight iterations of each solve
        fields = len(_names(case))
        per = 1100 + 250 * case["dust"] + (700 if case["closure"] == "fourier" else 0) + 2 * 8 * 30
        return dict(bytes=2.0 * fields * word * n, flops=float(per * case["steps"]) * n)
    if case["kind"] == "solve":  # psi and b in, x out; the network's multiply-adds, each of a dozen directions
        per = 2 * 27 * (16 * 32 + (16 * 32 + 32 * 32 + 96 * 32) / 8 + (32 * 64 + 64 * 64) / 64 + 48 * 16 + 16)
        return dict(bytes=3.0 * word * n, flops=(12 if case["every"] else 1) * per * n)
    if case["kind"] == "train":  # the pair in; forward, data gradients and weight gradients
        per = 2 * 27 * (2 * 16 + 256 + (16 * 32 + 32 * 32 + 96 * 32) / 8 + (32 * 64 + 64 * 64) / 64 + 48 * 16 + 16)
        return dict(bytes=3.0 * word * n, flops=3.0 * per * n)
    if case["kind"] == "analysis":  # rho and u in, Q and ten filtered fields out; transforms, gradients, filters
        return dict(bytes=15.0 * word * n, flops=(15 * math.log2(float(n)) + 600.0) * n)
    # field in, triangles (about half a cell each) and image out; about 60 operations per triangle
    return dict(bytes=word * n + 36.0 * n + 4.0 * case["width"] ** 2, flops=60.0 * n)


# ---- the same in 64 bits ----------------------------------------------------------------------------
def _dot(a, b):
    return (a * b).sum(dim=(-3, -2, -1), keepdim=True)


def _cg(M, b, diag):
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag
    pd, rz, bb = z.clone(), _dot(r, z), _dot(b, b)
    for _ in range(400):
        q = M(pd)
        a = rz / _dot(pd, q).clamp(min=1e-300)
        x, r = x + a * pd, r - a * q
        if bool((_dot(r, r) <= 1e-27 * bb).all()):
            break
        z = r / diag
        new = _dot(r, z)
        pd, rz = z + (new / rz.clamp(min=1e-300)) * pd, new
    return x


def _bicgstab(M, b, diag):
    x, r = torch.zeros_like(b), b.clone()
    r0, rho, alpha, w = b.clone(), 1.0, 1.0, 1.0
    v = pd = torch.zeros_like(b)
    bb = _dot(b, b)
    for _ in range(400):
        new = _dot(r0, r)
        pd = r + (new / rho) * (alpha / w) * (pd - w * v)
        y = pd / diag
        v = M(y)
        alpha = new / _dot(r0, v)
        s = r - alpha * v
        z = s / diag
        t = M(z)
        w = _dot(t, s) / _dot(t, t)
        x, r, rho = x + alpha * y + w * z, s - w * t, new
        if bool((_dot(r, r) <= 1e-26 * bb).all()):
            break
    return x


def _exact_step(case, prm, st, dt_prev):
    """One step of boxes of one size: fields (B, N, N, N), parameters (B, 1, 1, 1)."""
    N = st["rho"].shape[-1]
    h = 2.0 * math.pi / N
    mu, tau, nd = prm["nu"], prm["tau"], case["dust"]
    fourier, two_fluid, two_way = (case["closure"] == "fourier", case["model"] == "two-fluid",
                                   case["coupling"] == "two-way" and case["dust"] > 0)
    transonic = case["solver"] == "bicgstab"
    R = 1.0 / GAMMA
    cv = R / (GAMMA - 1.0)
    kappa = mu * GAMMA * cv / PRANDTL
    rn, pn = st["rho"], st["p"]
    un, phn = [st["u" + x] for x in "xyz"], [st["phi" + x] for x in "xyz"]
    Yn = [st["Y%d" % j] for j in range(nd)]
    umax = (un[0].abs() + un[1].abs() + un[2].abs()).amax(dim=(-3, -2, -1), keepdim=True)
    dt = torch.minimum(0.5 * h / umax, 1.2 * dt_prev)
    psi = rn / (GAMMA * pn)
    Ysum = sum(Yn) if two_way else None

    def accel(rho, u, p):
        v = _viscous(u, mu, h)
        inertia = rho * (1.0 + Ysum) if two_way else rho
        return [(v[m] - _Gc(p, m, h)) / inertia for m in range(3)]

    def dust_div(phi, rho, a, j, Y):
        F = 0.0
        for d in range(3):
            F = F + _D1((phi[d] - tau[j] * _I4(rho, d) * _I4(a[d], d)) * _I4(Y, d), d, h)
        return F

    def energy_div(phi, u, rho, p, E, T):
        H, div, out = E + p / rho, _div_u(u, h), 0.0
        for d in range(3):
            t = _stress(u, mu, h, d, div)
            F = phi[d] * _I4(H, d) - kappa * _G4(T, d, h)
            for m in range(3):
                F = F - t[m] * _I4(u[m], d)
            out = out + _D1(F, d, h)
        return out

    divn = _D(phn, h)
    rho = rn - dt * divn
    an = accel(rn, un, pn)
    Rn = _momentum(un, phn, mu, h)
    if two_way:
        Rn = [Rn[m] - rn * Ysum * an[m] for m in range(3)]
    u = [(rn * un[m] + dt * (Rn[m] - _Gc(pn, m, h))) / rho for m in range(3)]
    FYn = [dust_div(phn, rn, an, j, Yn[j]) for j in range(0 if two_fluid else nd)]
    if fourier:
        En = cv * st["T"] + 0.5 * (un[0] ** 2 + un[1] ** 2 + un[2] ** 2)
        FEn = energy_div(phn, un, rn, pn, En, st["T"])
        E = En
    phi, p, Y, a = phn, pn, list(Yn), an
    for _ in range(2):
        Lk = _momentum(u, phi, mu, h)
        if two_way:
            Lk = [Lk[m] - rho * Ysum * a[m] for m in range(3)]
        hb = [(rn * un[m] + dt * 0.5 * (Rn[m] + Lk[m])) / rho for m in range(3)]
        del Lk
        ps = [_I4(rho, d) * _I4(hb[d], d) - dt * _G2(p, d, h) for d in range(3)]
        b = -((rho - rn) / dt + 0.5 * divn + 0.5 * _D(ps, h))
        face = [_I4(hb[d], d) for d in range(3)] if transonic else None

        def M(x):
            y = psi * x / dt
            for d in range(3):
                y = y - 0.5 * dt * _D1(_G2(x, d, h), d, h)
                if transonic:
                    y = y + 0.5 * _D1(_I4(psi * x, d) * face[d], d, h)
            return y

        pc = (_bicgstab if transonic else _cg)(M, b, psi / dt + 3.0 * dt / (h * h))
        p = p + pc
        phi = [ps[d] - dt * _G2(pc, d, h) + (_I4(psi * pc, d) * face[d] if transonic else 0.0) for d in range(3)]
        del ps, b
        u = [hb[m] - (dt / rho) * _Gc(p, m, h) for m in range(3)]
        rho = rn - 0.5 * dt * (divn + _D(phi, h))
        a = accel(rho, u, p)
        if not two_fluid:
            Y = [(rn * Yn[j] - 0.5 * dt * (FYn[j] + dust_div(phi, rho, a, j, Y[j]))) / rho for j in range(nd)]
        if fourier:
            FEk = energy_div(phi, u, rho, p, E, p / (rho * R))
            E = (rn * En - 0.5 * dt * (FEn + FEk)) / rho
    new = dict(rho=rho, ux=u[0], uy=u[1], uz=u[2], phix=phi[0], phiy=phi[1], phiz=phi[2])
    if fourier:
        new["T"] = (E - 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)) / cv
        new["p"] = rho * R * new["T"]
    else:
        new["p"] = rho ** GAMMA / GAMMA
    for j in range(nd):
        if not two_fluid:
            new["Y%d" % j] = Y[j]
            continue
        Vn = [st["V%d%s" % (j, x)] for x in "xyz"]

        def fluxes(phi_, rho_, u_, Y_, V_):
            F = [(phi_[d] + _I4(rho_, d) * _I4(V_[d] - u_[d], d)) * _I4(Y_, d) for d in range(3)]
            return _D(F, h), [_D([F[d] * _I4(V_[m], d) for d in range(3)], h) for m in range(3)]

        def drag(sig, mom):
            return [u[m] + (mom[m] / sig - u[m]) * (tau[j] / (tau[j] + dt)) for m in range(3)]

        sn = rn * Yn[j]
        F0, G0 = fluxes(phn, rn, un, Yn[j], Vn)
        ss = sn - dt * F0
        Vs = drag(ss, [sn * Vn[m] - dt * G0[m] for m in range(3)])
        F1, G1 = fluxes(phi, rho, u, ss / rho, Vs)
        ss = sn - 0.5 * dt * (F0 + F1)
        V = drag(ss, [sn * Vn[m] - 0.5 * dt * (G0[m] + G1[m]) for m in range(3)])
        new["Y%d" % j] = ss / rho
        for m in range(3):
            new["V%d%s" % (j, "xyz"[m])] = V[m]
    return new, dt


def _exact_steps(case, seed):
    sizes, names = _sizes(case), _names(case)
    out = {n: [None] * len(sizes) for n in names}
    times = [0.0] * len(sizes)
    for N in sorted(set(sizes)):
        at = [b for b, v in enumerate(sizes) if v == N]
        many = [_state(case, seed, b, N) for b in at]
        st = {n: torch.stack([m[n].double() for m in many]) for n in names}
        del many
        boxes = [_box(case, b, N) for b in at]
        col = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV).reshape(-1, 1, 1, 1)  # noqa: E731
        prm = dict(nu=col([b["nu"] for b in boxes]),
                   tau=[col([b["tau_p"][j] for b in boxes]) for j in range(case["dust"])])
        dt, t = col([math.inf] * len(at)), 0.0
        for _ in range(case["steps"]):
            st, dt = _exact_step(case, prm, st, dt)
            t = t + dt
        for q, b in enumerate(at):
            times[b] = float(t.reshape(-1)[q])
            for n in names:
                out[n][b] = st[n][q].reshape(-1)
    res = {n: torch.cat(v) if len(v) > 1 else v[0] for n, v in out.items()}
    res["t"] = times if len(times) <= 4 else float(sum(times))
    return res


def _grad(u, h):
    return [[_Gc(u[c], d, h) for d in range(3)] for c in range(3)]  # [component][direction]


def _q_field(u, h):
    A = _grad(u, h)
    q = 0.0
    for i in range(3):
        for j in range(3):
            q = q + 0.125 * ((A[i][j] - A[j][i]) ** 2 - (A[i][j] + A[j][i]) ** 2)
    return q


def _exact_analysis(case, seed):
    N, m = case["N"], case["filter"]
    h = 2.0 * math.pi / N
    st = _state(case, seed, 0, N)
    rho, u = st["rho"].double(), [st["u" + x].double() for x in "xyz"]
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    A = _grad(u, h)
    mean = lambda f: float(f.mean())  # noqa: E731
    w2 = (A[2][1] - A[1][2]) ** 2 + (A[0][2] - A[2][0]) ** 2 + (A[1][0] - A[0][1]) ** 2
    diag = dict(ke=0.5 * mean(rho * uu), ke_u=0.5 * mean(uu), enstrophy=0.5 * mean(w2),
                taylor=math.sqrt(mean(uu) / mean(A[0][0] ** 2 + A[1][1] ** 2 + A[2][2] ** 2)),
                rho_rms=mean((rho - rho.mean()) ** 2) ** 0.5, mass=(2 * math.pi) ** 3 * mean(rho),
                energy=(2 * math.pi) ** 3 * 0.5 * mean(rho * uu))
    k = torch.fft.fftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
    shell = torch.floor(torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2) + 0.5)
    dens = sum(torch.fft.fftn(c).abs().square() for c in u) / (2.0 * float(N) ** 6)
    spec = torch.bincount(shell.long().reshape(-1), weights=dens.reshape(-1))[:N // 2]
    q = _q_field(u, h)
    del A, w2, shell, dens

    def bar(f):
        for d in range(3):
            s = 0.5 * (_at(f, d, -m) + _at(f, d, m))
            for o in range(1 - m, m):
                s = s + _at(f, d, o)
            f = s / (2 * m)
        return f

    pairs = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
    weight = [1.0 if i == j else 2.0 for i, j in pairs]
    rb = bar(rho)
    ru = [bar(rho * c) for c in u]
    ut = [c / rb for c in ru]
    tau = [bar(rho * u[i] * u[j]) - ru[i] * ru[j] / rb for i, j in pairs]
    G = _grad(ut, h)
    S = [0.5 * (G[i][j] + G[j][i]) for i, j in pairs]

    def dev(t):
        tr = (t[0] + t[3] + t[5]) / 3.0
        return [t[a] - tr if i == j else t[a] for a, (i, j) in enumerate(pairs)]

    def dot(a, b):
        return sum(w * x * y for w, x, y in zip(weight, a, b))

    delta = 2 * m * h
    B = [-2.0 * rb * delta ** 2 * torch.sqrt(2.0 * dot(S, S)) * s for s in dev(S)]
    td = dev(tau)
    tb, bb, tt = mean(dot(td, B)), mean(dot(B, B)), mean(dot(td, td))
    les = dict(delta=delta, k_sgs=0.5 * mean(tau[0] + tau[3] + tau[5]), pi_sgs=-mean(dot(td, S)), cs2_opt=tb / bb,
               corr=tb / math.sqrt(tt * bb), pi_model=-CS * CS * mean(dot(B, S)))
    return dict(diag=diag, spectrum=spec, q=q, les=les, fields=torch.stack([rb] + ut + tau))


def _room(N):
    """Triangles that a program makes room for (the rest of the buffer keeps its zeros)."""
    return 3 * N ** 3 // 2


def _surface_field(case, st):
    """The Q field of the flow, and the level: a share of the mean enstrophy."""
    N = case["N"]
    h = 2.0 * math.pi / N
    u = [st["u" + x].double() for x in "xyz"]
    A = _grad(u, h)
    w2 = (A[2][1] - A[1][2]) ** 2 + (A[0][2] - A[2][0]) ** 2 + (A[1][0] - A[0][1]) ** 2
    q = _q_field(u, h).to(_dtype(case)).contiguous()
    return q, round(case["level"] * 0.5 * float(w2.mean()), 9)


def _exact_surface(case, seed):
    """Marching tetrahedra in double precision: the triangles in cube order, then tetrahedron, and the area."""
    N = case["N"]
    h = 2.0 * math.pi / N
    q, iso = _surface_field(case, _state(case, seed, 0, N))
    f = q.double()
    inside = f > iso
    corner = [torch.roll(inside, (-((b >> 2) & 1), -((b >> 1) & 1), -(b & 1)), (0, 1, 2)) for b in range(8)]
    every, some = corner[0].clone(), corner[0].clone()
    for c in corner[1:]:
        every, some = every & c, some | c
    cut = (some & ~every).reshape(-1).nonzero().reshape(-1)
    ijk = [cut % N, (cut // N) % N, cut // (N * N)]
    val, pos = [], []
    for b in range(8):
        o = [(ijk[d] + ((b >> d) & 1)) for d in range(3)]
        val.append(f[o[2] % N, o[1] % N, o[0] % N])
        pos.append(torch.stack([(o[d].double() + 0.5) * h for d in range(3)], 1))
    val, pos = torch.stack(val, 1), torch.stack(pos, 1)

    def point(rows, a, b):
        a, b = min(a, b), max(a, b)
        t = (iso - val[rows, a]) / (val[rows, b] - val[rows, a])
        return pos[rows, a] + t[:, None] * (pos[rows, b] - pos[rows, a])

    key, tri = [], []
    for n, tet in enumerate(((0, 1, 3, 7), (0, 1, 5, 7), (0, 2, 3, 7), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 6, 7))):
        mask = sum((val[:, v] > iso).long() << q_ for q_, v in enumerate(tet))
        for case_ in range(1, 15):
            rows = (mask == case_).nonzero().reshape(-1)
            ins = [v for q_, v in enumerate(tet) if (case_ >> q_) & 1]
            outs = [v for v in tet if v not in ins]
            if len(ins) == 2:
                (a, b), (c, d) = ins, outs
                made = [((a, c), (a, d), (b, d)), ((a, c), (b, d), (b, c))]
            else:
                lone = (ins if len(ins) == 1 else outs)[0]
                made = [tuple((lone, v) for v in tet if v != lone)]
            for w, edges in enumerate(made):
                key.append(rows * 12 + 2 * n + w)
                tri.append(torch.stack([point(rows, *e) for e in edges], 1))
    tri = torch.cat(tri)[torch.argsort(torch.cat(key))]
    e1, e2 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    area = 0.5 * float(torch.linalg.cross(e1, e2).norm(dim=1).sum())
    room = torch.zeros((_room(N), 3, 3), dtype=torch.float64, device=DEV)
    room[:len(tri)] = tri[:len(room)]
    return dict(n=len(tri), tri=room, area=area, depth=None)  # the image is defined by its single-precision steps


# ---- the learned preconditioner: a pair (r, e) with M e = r, weights early in training --------------
LAYERS = ((2, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (48, 16), (16, 1))


def _weights(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed % (1 << 40) + 5)
    parts = []
    for n, (ci, co) in enumerate(LAYERS):
        scale = math.sqrt(2.0 / (27 * ci)) * (0.05 if n == 8 else 1.0)
        parts += [scale * torch.randn(27 * ci * co, generator=g, device=DEV, dtype=torch.float32),
                  torch.zeros(co, device=DEV)]
    return torch.cat(parts)


def _operator(st, dt, h):
    psi = st["rho"].double() / (GAMMA * st["p"].double())

    def M(x):
        y = psi * x / dt
        for d in range(3):
            y = y - 0.5 * dt * _D1(_G2(x, d, h), d, h)
        return y

    return M, psi / dt + 3.0 * dt / (h * h)


def _pair(case, st, seed):
    """A correction with the scales of a corrector's solution and its right-hand side."""
    N = case["N"]
    h, dt = 2.0 * math.pi / N, _courant_dt(st, N)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed % (1 << 40) + 11)
    kv = _modes(N)
    k2 = kv[0] ** 2 + kv[1] ** 2 + kv[2] ** 2
    e = _scalar(N, torch.where(k2 > 0, 1.0 / (1.0 + k2 / case["k0"] ** 2), torch.zeros_like(k2)), g)
    e = (1e-3 * e).to(_dtype(case)).contiguous()
    r = _operator(st, dt, h)[0](e.double())
    return r.to(_dtype(case)).contiguous(), e, dt


def _network(w, x):
    at, n, layers = 0, x.shape[-1], []
    for ci, co in LAYERS:
        layers.append((w[at:at + 27 * ci * co].reshape(27, ci, co), w[at + 27 * ci * co:at + 27 * ci * co + co]))
        at += 27 * ci * co + co

    def conv(v, layer, stride=1):
        W, bias = layer
        out = bias.reshape(-1, 1, 1, 1)
        for t in range(27):
            s = torch.roll(v, (1 - t // 9, 1 - (t // 3) % 3, 1 - t % 3), (1, 2, 3))
            out = out + torch.einsum("io,izyx->ozyx", W[t], s[:, ::stride, ::stride, ::stride])
        return out

    def up(v):
        return v.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    e1 = conv(conv(x, layers[0]).relu(), layers[1]).relu()
    e2 = conv(conv(e1, layers[2], 2).relu(), layers[3]).relu()
    e3 = conv(conv(e2, layers[4], 2).relu(), layers[5]).relu()
    u2 = conv(torch.cat([up(e3), e2]), layers[6]).relu()
    u1 = conv(torch.cat([up(u2), e1]), layers[7]).relu()
    return conv(u1, layers[8])[0]


def _exact_train(case, seed):
    N = case["N"]
    h = 2.0 * math.pi / N
    st = _state(case, seed, 0, N)
    r, e, dt = _pair(case, st, seed)
    r, e = r.double(), e.double()
    diag = _operator(st, dt, h)[1]
    scale = float(r.square().mean().sqrt()) / (1.0 / dt + 3.0 * dt / (h * h))
    x = torch.stack([(r / diag) / scale, (3.0 * dt / (h * h)) / diag])
    target = (e - r / diag) / scale
    w = _weights(seed).double().requires_grad_(True)
    loss = (_network(w, x) - target).square().sum() / target.square().sum()
    loss.backward()
    g = w.grad
    m, v = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
    return dict(loss=float(loss), weights=w.detach() - case["rate"] * m / (v.sqrt() + 1e-8), gradients=g)


def _exact_solve(case, seed):
    N = case["N"]
    st = _state(case, seed, 0, N)
    r, _, dt = _pair(case, st, seed)
    M, diag = _operator(st, dt, 2.0 * math.pi / N)
    return _cg(M, r.double(), diag)


def exact(case, seed):
    """What run() returns for these inputs, in plain torch in 64 bits."""
    kind = case["kind"]
    if kind == "step":
        return _exact_steps(case, seed)
    return {"analysis": _exact_analysis, "surface": _exact_surface, "train": _exact_train,
            "solve": _exact_solve}[kind](case, seed)
