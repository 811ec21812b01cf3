"""Performance cases of the formal solver: the calls that a program makes through
the Python package, from one tiny formal solution to iterations of whole boxes.

listed() and draw(rng) describe cases as plain dicts, prepare(case, seed) builds
the inputs and the solver context a program has in hand, run(state) makes one
pass through the public entry points, work(case) counts the bytes and operations
a pass cannot do without, and exact(case, seed) computes the same outputs in
double precision with plain torch operations.

Kinds of case
  formal    porta_formal_solve + porta_accumulate_jkq: J^K_Q and Lambda-bar*
  jacobi    Jacobi iterations replayed as a CUDA graph: the unknowns after them
  batch     the same for a batch of uneven boxes in one context
  emergent  emergent Stokes profiles along several lines of sight
  vjp       gradients of emergent profiles (chi, emission scale, field)
  itervjp   gradients through checkpointed Jacobi iterations
  vcycle    one non-linear multigrid V-cycle
  ml        five-level atom, populations: line formal solutions and one update
  mlpol     five-level atom, all multipoles: the same with dichroism
"""
import math
from fractions import Fraction
from functools import lru_cache

import numpy as np
import torch
import torch.utils.checkpoint

import paper_1307_4217_gb300 as P

H_KM, L_KM = 100.0, 800.0                # opacity scale height, horizontal period
TAU_TOP, TAU_BOT = 1e-4, 1e3             # vertical line-centre optical depth of the box
X_MAX = 4.0                              # frequency grid half-width (Doppler widths)
BCRIT, GBAR = 25.0, 1.0                  # two-level atom: Hanle critical field (G), Lande factor
ZETA, ML_ZETA = 3.5e-4, 1e-5             # Zeeman splitting per gauss (Doppler widths)
# five-level atom: J, energies (eV), lines (upper, lower)
ML_J = (0, 1, 2, 1, 2)
ML_E = (0.0, 1.692, 1.700, 3.123, 3.151)
ML_LINES = ((3, 0), (3, 1), (4, 1), (4, 2))


def _case(name, kind, nx, ny, nz, quad, **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, n_mu=quad[0], n_chi=quad[1], n_nu=quad[2], pol=True, f64=False, eps=1e-2)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one formal solution of a small unpolarized box, where launches
        # and fixed costs count (an inner call of a 1D-like or test setup)
        _case("formal_unpol_f32_8x8x16", "formal", 8, 8, 16, (2, 4, 7), pol=False),
        # the plain method: FP64, unpolarized atom, 48 rays x 11 frequencies, Jacobi by graph replay
        _case("jacobi_unpol_f64_16x16x32", "jacobi", 16, 16, 32, (3, 8, 11), pol=False, f64=True, iters=10),
        # the polarized atom in FP64, as run to check an FP32 result
        _case("formal_pol_f64_24x24x32", "formal", 24, 24, 32, (3, 8, 11), f64=True),
        # an ordinary FP32 formal solution with odd, ragged plane sizes
        _case("formal_pol_f32_33x27x41", "formal", 33, 27, 41, (4, 10, 21)),
        # the main workload: Jacobi iterations of the 64^3 polarized box, autotuned once
        _case("jacobi_pol_f32_64x64x64", "jacobi", 64, 64, 64, (5, 16, 21), iters=2, tune=True, eps=1e-3),
        # many independent boxes of uneven size in one launch (inversion-like use), autotuned once
        _case("batch_pol_f32_32_boxes", "batch", 48, 48, 64, (4, 10, 21), boxes=32, tune=True),
        # synthetic observations: the vertical and four oblique lines of sight
        _case("emergent_pol_f32_64x64x64", "emergent", 64, 64, 64, (5, 16, 21), ndir=5),
        # gradients of emergent profiles for a fit of the atmosphere
        _case("vjp_pol_f32_48x48x40", "vjp", 48, 48, 40, (5, 16, 21), ndir=5),
        # gradients through the iterations themselves, in FP64: the control points' kinks make
        # FP32 gradients through several iterations good to a few digits only
        _case("itervjp_pol_f64_16x16x24", "itervjp", 16, 16, 24, (2, 8, 7), ndir=5, iters=3, ckpt=2, f64=True),
        # one multigrid V-cycle over three grids (its coarse grids are small launches)
        _case("vcycle_pol_f32_32x32x32", "vcycle", 32, 32, 32, (3, 8, 11), levels=3),
        # five-level atom, populations only: four lines x 31 frequencies, one iteration
        _case("ml_f32_64x64x48", "ml", 64, 64, 48, (5, 16, 31), pol=False),
        # five-level atom with all 69 multipoles and dichroism, one iteration
        _case("mlpol_f32_32x32x24", "mlpol", 32, 32, 24, (5, 16, 31)),
    ]


def _updates(case):
    """voxel-ray-frequency updates of one formal solution of the case"""
    n = case["nx"] * case["ny"] * case["nz"] * 2 * case["n_mu"] * case["n_chi"] * case["n_nu"]
    if case["kind"] == "batch":
        n = sum(x * y * z for x, y, z in _boxes(case)) * 2 * case["n_mu"] * case["n_chi"] * case["n_nu"]
    return n * (len(ML_LINES) if case["kind"] in ("ml", "mlpol") else 1)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: plane sizes 8..64, 16..64 planes, 16..160 rays, 5..31 frequencies."""
    kind = rng.choice(["formal", "formal", "formal", "jacobi", "jacobi", "batch", "emergent", "vjp", "itervjp",
                       "vcycle", "ml", "mlpol"])
    # most updates per formal solution of the kind (those of the listed case, or near)
    cap = {"formal": 4e8, "jacobi": 8e8, "batch": 1.5e9, "ml": 2e9, "mlpol": 3e8, "vcycle": 1.7e7}.get(kind, 1e9)
    f64 = kind == "itervjp" or (kind in ("formal", "jacobi") and rng.random() < 0.25)
    pol = kind not in ("ml",) and not (kind in ("formal", "jacobi") and rng.random() < 0.3)
    if f64:
        cap = 8e5 if kind == "itervjp" else 3e7
    while True:
        quad = (rng.randint(2, 5), rng.choice([4, 6, 8, 10, 12, 16]), rng.randint(5, 31))
        nx, ny, nz = _log_int(rng, 8, 64), _log_int(rng, 8, 64), _log_int(rng, 16, 64)
        if kind == "itervjp":
            quad = (rng.randint(2, 3), rng.choice([4, 6, 8]), rng.randint(5, 11))
            nx, ny, nz = _log_int(rng, 8, 20), _log_int(rng, 8, 20), _log_int(rng, 16, 28)
        c = _case(None, kind, nx, ny, nz, quad, pol=pol, f64=f64)
        if kind == "jacobi":
            c.update(iters=rng.randint(1, 4) if nx * ny * nz > 30000 else rng.randint(2, 8), tune=False)
        elif kind == "batch":
            c.update(nx=48, ny=48, nz=64, boxes=_log_int(rng, 4, 32), tune=True)
        elif kind in ("emergent", "vjp"):
            c.update(ndir=rng.randint(1, 6))
        elif kind == "itervjp":
            c.update(ndir=rng.randint(1, 5), iters=rng.randint(2, 4), ckpt=rng.randint(1, 2))
        elif kind == "vcycle":
            c.update(levels=rng.randint(2, 3))
            m = 1 << (c["levels"] - 1)
            c.update(nx=max(nx // m, 4) * m, ny=max(ny // m, 4) * m)
        scale = 2.5 if kind == "jacobi" and c["iters"] > 2 else 1.0
        if _updates(c) * scale <= cap:
            return c


# ---------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt=0):
    return torch.Generator(device=_device()).manual_seed((int(seed) * 1000003 + salt) % (2 ** 62))


def _heights(nz):
    tau = np.geomspace(TAU_BOT, TAU_TOP, nz)
    return -H_KM * np.log(tau)


def _field(g, nx, ny, nz):
    """standardized Gaussian random field, power k^(-11/3), periodic in x and y"""
    dev, f64 = _device(), torch.float64
    f = torch.fft.fftn(torch.randn((2 * nz, ny, nx), generator=g, device=dev, dtype=f64))
    kz, ky, kx = (torch.fft.fftfreq(n, device=dev, dtype=f64) for n in (2 * nz, ny, nx))
    k = torch.sqrt(kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2)
    amp = torch.where(k > 0, torch.clamp(k, min=1e-9) ** (-11.0 / 6.0), torch.zeros_like(k))
    r = torch.fft.ifftn(f * amp).real[:nz]
    return ((r - r.mean()) / r.std()).contiguous()


def _atmosphere(case, seed, nx, ny, nz):
    """random stratified atmosphere: log-normal opacity, Planck function (or temperature)
    and field strength, isotropic field directions, Gaussian vertical velocity"""
    g = _gen(seed, nx * 65536 + ny * 256 + nz)
    dev, f64 = _device(), torch.float64
    shape = (nz, ny, nx)
    z = _heights(nz)
    zt = torch.tensor(z, device=dev)
    ml = case["kind"] in ("ml", "mlpol")
    g1, g2, g3 = (_field(g, nx, ny, nz) for _ in range(3))
    a = dict(nx=nx, ny=ny, nz=nz, lx=L_KM, ly=L_KM, z=z, zeta=ML_ZETA if ml else ZETA, gbar=GBAR, bcrit=BCRIT)
    a["chi"] = torch.exp(-zt / H_KM)[:, None, None] / H_KM * torch.exp(0.2 * g2)
    a["vel"] = g3
    if ml:
        a["kT"] = 0.5 * torch.exp(0.05 * g1)
    else:
        a["bpl"] = torch.exp(0.3 * g1)
        a["eps"] = torch.full(shape, case["eps"], device=dev, dtype=f64)
    if case["pol"]:
        # strengths bounded where the first-order Zeeman term stays a propagation matrix
        med, top = (30.0, 2000.0) if ml else (10.0, 100.0)
        b = torch.clamp(med * torch.exp(torch.randn(shape, generator=g, device=dev, dtype=f64)), max=top)
        d = torch.randn((3,) + shape, generator=g, device=dev, dtype=f64)
        d = b * d / torch.linalg.vector_norm(d, dim=0)
        a["bx"], a["by"], a["bz"] = (d[i].contiguous() for i in range(3))
    return a


def _atom(seed):
    """Einstein A (s^-1) and collisional destruction probability per line, log-uniform"""
    r = np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed) % (2 ** 32), 7])))
    n = len(ML_LINES)
    return dict(J=np.array(ML_J), E=np.array(ML_E), lines=np.array(ML_LINES),
                A=np.exp(r.uniform(np.log(1e7), np.log(1e8), n)), eps=np.exp(r.uniform(np.log(1e-4), np.log(1e-2), n)))


def _boxes(case):
    """plane sizes and heights of a batch: fixed by the case, so that work is known"""
    r = np.random.Generator(np.random.PCG64(np.random.SeedSequence([11, case["boxes"]])))
    out = []
    for _ in range(case["boxes"]):
        n = int(r.choice([8, 16, 24, 32, 48]))
        out.append((n, n, int(r.integers(16, case["nz"] + 1))))
    return out


def _start(a, pol, g):
    """unknowns of a two-level problem under way: S00 near B, multipoles of a few per cent"""
    b = a["bpl"]
    s00 = b * (0.5 + 0.5 * torch.rand(b.shape, generator=g, device=b.device, dtype=b.dtype))
    if not pol:
        return s00[..., None].contiguous()
    s2 = 0.02 * s00[..., None] * torch.randn(b.shape + (5,), generator=g, device=b.device, dtype=b.dtype)
    return torch.cat([s00[..., None], s2], -1).contiguous()


def _sight(n):
    """outgoing lines of sight: the vertical and oblique ones at mu = 0.5"""
    mu = np.array([1.0] + [0.5] * (n - 1))
    az = np.array([0.0] + [2.0 * np.pi * k / max(n - 1, 1) for k in range(n - 1)])
    return mu, az


def _inputs(case, seed):
    """everything a case's outputs depend on"""
    kind, pol = case["kind"], case["pol"]
    if kind == "batch":
        atms = [_atmosphere(case, seed * 4096 + b, *s) for b, s in enumerate(_boxes(case))]
        g = _gen(seed, 1)
        return dict(atms=atms, rho=[_start(a, pol, g) for a in atms])
    a = _atmosphere(case, seed, case["nx"], case["ny"], case["nz"])
    g = _gen(seed, 1)
    if kind in ("ml", "mlpol"):
        atom = _atom(seed)
        pops = _lte(atom, a["kT"]) * torch.exp(0.1 * torch.randn(a["kT"].shape + (len(ML_J),), generator=g,
                                                                 device=_device(), dtype=torch.float64))
        pops = pops / pops.sum(-1, keepdim=True)
        if not pol:
            return dict(atm=a, atom=atom, x=pops)
        # multipoles of the order of a per cent of the populations
        x = torch.randn(a["kT"].shape + (sum((2 * j + 1) ** 2 for j in ML_J),), generator=g, device=_device(),
                        dtype=torch.float64)
        n = 0
        for i, j in enumerate(ML_J):
            r00 = pops[..., i] / math.sqrt(2 * j + 1)
            x[..., n] = r00
            x[..., n + 1:n + (2 * j + 1) ** 2] *= 0.01 * r00[..., None]
            n += (2 * j + 1) ** 2
        return dict(atm=a, atom=atom, x=x)
    d = dict(atm=a, rho=_start(a, pol, g))
    if "ndir" in case:
        d["mu"], d["az"] = _sight(case["ndir"])
        shape = (case["ndir"], case["n_nu"], case["ny"], case["nx"], 4 if pol else 1)
        d["grad"] = 0.1 * torch.randn(shape, generator=g, device=_device(), dtype=torch.float64)
    return d


# ---------------------------------------------------------------- the framework's calls

def prepare(case, seed):
    d = _inputs(case, seed)
    kind, pol = case["kind"], case["pol"]
    quad = (case["n_mu"], case["n_chi"], case["n_nu"], X_MAX)
    prec = P.PORTA_FP64 if case["f64"] else P.PORTA_FP32
    model = P.PORTA_MODEL_TWOLEVEL_HANLE if pol else P.PORTA_MODEL_TWOLEVEL_UNPOL
    dev, f64 = _device(), torch.float64
    st = dict(case=case, kind=kind)
    if kind == "batch":
        ctx = P.BatchContext(d["atms"], model, *quad, precision=prec)
        # the concatenated arrays of the boxes, on the device
        cat = {k: torch.cat([a[k].reshape(-1) for a in d["atms"]]) for k in d["atms"][0]
               if torch.is_tensor(d["atms"][0][k])}
        P.Context.set_atmosphere(ctx, cat)
        st["rho"] = torch.cat([r.reshape(-1, r.shape[-1]) for r in d["rho"]])
    elif kind in ("ml", "mlpol"):
        ctx = P.MlContext(d["atm"], d["atom"], *quad, precision=prec, polarized=pol, zeta=ML_ZETA)
        ctx.set_atmosphere(d["atm"])
        st["x"] = d["x"]
        st["jbar"] = torch.empty(ctx.shape + ((9,) if pol else ()), device=dev, dtype=f64)
        st["lstar"] = torch.empty(ctx.shape, device=dev, dtype=f64)
        st["out"] = torch.empty_like(d["x"])
    else:
        ctx = P.Context(d["atm"], model, *quad, precision=prec)
        ctx.set_atmosphere(d["atm"])
        st["rho"] = d["rho"]
    st["ctx"] = ctx
    if "rho" in st:
        ctx.set_rho(st["rho"])
        st["out"] = torch.empty_like(st["rho"])
    if kind == "formal":
        st["jkq"] = torch.empty(ctx.shape + (ctx.nj,), device=dev, dtype=f64)
        st["lstar"] = torch.empty(ctx.shape, device=dev, dtype=f64)
    if "ndir" in case:
        st["mu"], st["az"], st["grad"] = d["mu"], d["az"], d["grad"]
        st["prof"] = torch.empty_like(d["grad"])
        st["g"] = [torch.empty(ctx.shape, device=dev, dtype=f64) for _ in range(2)] + [
            torch.empty((3,) + ctx.shape, device=dev, dtype=f64)]
    if kind == "vcycle":
        ctx.mg_setup(case["levels"])
    if kind in ("jacobi", "batch"):
        st["stream"] = torch.cuda.Stream()
        torch.cuda.current_stream().synchronize()
        ctx.set_stream(st["stream"])
    if case.get("tune"):
        ctx.autotune()
    torch.cuda.synchronize()
    st["f32"] = {}
    return st


def _handed_on(state, **out):
    """the outputs as a program keeps them: what FP32 sweeps computed in single precision"""
    if state["case"]["f64"]:
        return out
    for k, v in out.items():
        if k not in state["f32"]:
            state["f32"][k] = torch.empty_like(v, dtype=torch.float32)
        state["f32"][k].copy_(v)
    return dict(state["f32"])


def run(state):
    kind, ctx, case = state["kind"], state["ctx"], state["case"]
    if kind == "formal":
        ctx.formal_solve()
        ctx.accumulate_jkq(state["jkq"], state["lstar"])
        return _handed_on(state, jkq=state["jkq"], lstar=state["lstar"])
    if kind in ("jacobi", "batch"):
        s, cur = state["stream"], torch.cuda.current_stream()
        s.wait_stream(cur)
        ctx.set_rho(state["rho"])
        ctx.run_iterations(case.get("iters", 1), residual=False)
        ctx.get_rho(state["out"])
        cur.wait_stream(s)
        return _handed_on(state, rho=state["out"])
    if kind == "emergent":
        return _handed_on(state, stokes=ctx.emergent_stokes(state["mu"], state["az"], state["prof"]))
    if kind == "vjp":
        g = ctx.emergent_vjp(state["mu"], state["az"], state["grad"], state["prof"], *state["g"])
        return _handed_on(state, g_chi=g[0], g_e=g[1], g_b=g[2], stokes=g[3])
    if kind == "itervjp":
        ctx.set_rho(state["rho"])
        ctx.iterate_ckpt(case["iters"], case["ckpt"], residual=False)
        g = ctx.iterate_vjp(state["mu"], state["az"], state["grad"], state["prof"], *state["g"])
        return _handed_on(state, g_chi=g[0], g_f=g[1], g_b=g[2], stokes=g[3])
    if kind == "vcycle":
        ctx.set_rho(state["rho"])
        ctx.mg_vcycle(2, 4, 8, residual=False)
        ctx.get_rho(state["out"])
        return _handed_on(state, rho=state["out"])
    if state["case"]["pol"]:
        ctx.set_unknowns(state["x"])
    else:
        ctx.set_pops(state["x"])
    ctx.ml_formal_solve(state["jbar"], state["lstar"])
    ctx.ml_see_update(residual=False)
    if state["case"]["pol"]:
        ctx.get_unknowns(state["out"])
    else:
        ctx.get_pops(state["out"])
    return _handed_on(state, jbar=state["jbar"], lstar=state["lstar"], x=state["out"])


# algorithmic operations of one voxel-ray-frequency update: the polarized step (293, each
# node's coefficients once per ray and frequency), the same step for Stokes I alone, and
# the reverse step (about twice the forward one on top of it)
_OPS = {True: 293.0, False: 95.0}


def work(case):
    kind, pol = case["kind"], case["pol"]
    upd = _updates(case)
    vox = case["nx"] * case["ny"] * case["nz"]
    if kind == "batch":
        vox = sum(x * y * z for x, y, z in _boxes(case))
    nl = 6 if pol else 1
    atm = 8.0 * vox * (7 if pol else 4)
    plane = 8.0 * case["nx"] * case["ny"] * case["n_nu"] * (4 if pol else 1)
    if kind == "formal":
        return {"bytes": atm + 8.0 * vox * (2 * nl + 1), "flops": upd * _OPS[pol]}
    if kind in ("jacobi", "batch"):
        return {"bytes": atm + 16.0 * vox * nl, "flops": upd * _OPS[pol] * case.get("iters", 1)}
    if kind in ("emergent", "vjp"):
        n = float(vox) * case["n_nu"] * case["ndir"]
        if kind == "emergent":
            return {"bytes": atm + 8.0 * vox * nl + plane * case["ndir"], "flops": n * _OPS[pol]}
        return {"bytes": atm + 8.0 * vox * (nl + 5) + 2 * plane * case["ndir"], "flops": 3 * n * _OPS[pol]}
    if kind == "itervjp":
        return {"bytes": atm + 8.0 * vox * (nl + 5) + 2 * plane * case["ndir"],
                "flops": (4 * case["iters"]) * upd * _OPS[pol]}
    if kind == "vcycle":
        # per level: 2 + 4 iterations and one residual, one residual of the coarse problem
        f, total = float(upd), 0.0
        for l in range(case["levels"]):
            total += f * (8 if l == case["levels"] - 1 else 7) + (f if l else 0.0)
            f /= 8.0
        return {"bytes": atm + 16.0 * vox * nl, "flops": total * _OPS[pol]}
    nunk, nj = (sum((2 * j + 1) ** 2 for j in ML_J), 9) if pol else (len(ML_J), 1)
    see = vox * (2.0 / 3.0) * (nunk - len(ML_J) if pol else nunk) ** 3
    return {"bytes": 8.0 * vox * ((6 if pol else 3) + 2 * nunk + len(ML_LINES) * (nj + 1)),
            "flops": upd * _OPS[pol] + see}


# ---------------------------------------------------------------- the same in 64 bits, plain torch

def _gauss01(n):
    x, w = np.polynomial.legendre.leggauss(n)
    for _ in range(2):                                 # polish the roots
        p = np.polynomial.legendre.Legendre.basis(n)
        x = x - p(x) / p.deriv()(x)
    w = 2.0 / ((1.0 - x * x) * np.polynomial.legendre.Legendre.basis(n).deriv()(x) ** 2)
    return 0.5 * (x + 1.0), 0.5 * w


def _rays(case):
    x, w = _gauss01(case["n_mu"])
    nc = case["n_chi"]
    mu, az, wt = [], [], []
    for sgn in (1.0, -1.0):
        for i in range(case["n_mu"]):
            for a in range(nc):
                mu.append(sgn * x[i])
                az.append((a + 0.5) * 2.0 * np.pi / nc)
                wt.append(0.5 * w[i] / nc)
    return np.array(mu), np.array(az), np.array(wt)


def _freqs(case):
    n = case["n_nu"]
    x = np.linspace(-X_MAX, X_MAX, n)
    w = np.full(n, 2.0 * X_MAX / (n - 1))
    w[0] *= 0.5
    w[-1] *= 0.5
    return x, w


def _tensors(mu, az):
    """T^K_Q(i, Omega), i = I, Q, U: (rays, 3, 6), components 00, 20, Re/Im 21, Re/Im 22"""
    st2 = 1.0 - mu * mu
    st = np.sqrt(np.maximum(st2, 0.0))
    r3, r2 = math.sqrt(3.0), math.sqrt(2.0)
    c1, s1, c2, s2 = np.cos(az), np.sin(az), np.cos(2 * az), np.sin(2 * az)
    o = np.zeros_like(mu)
    ti = [o + 1.0, (3 * mu * mu - 1) / (2 * r2), -0.5 * r3 * mu * st * c1, -0.5 * r3 * mu * st * s1,
          0.25 * r3 * st2 * c2, 0.25 * r3 * st2 * s2]
    tq = [o, -3 / (2 * r2) * st2, -0.5 * r3 * mu * st * c1, -0.5 * r3 * mu * st * s1,
          -0.25 * r3 * (1 + mu * mu) * c2, -0.25 * r3 * (1 + mu * mu) * s2]
    tu = [o, o, 0.5 * r3 * st * s1, -0.5 * r3 * st * c1, 0.5 * r3 * mu * s2, -0.5 * r3 * mu * c2]
    return np.stack([np.stack(t, -1) for t in (ti, tq, tu)], 1)


def _coefficients(t):
    """e^-t, w_M, w_O, w_C of the upwind optical path t (series below 0.5)"""
    e = torch.exp(-t)
    ts, tb = torch.clamp(t, max=0.5), torch.clamp(t, min=0.5)
    wm = wo = wc = torch.zeros_like(t)
    for k in range(15, 0, -1):
        s = (1.0 if k % 2 else -1.0) / math.factorial(k + 2)
        wm = (wm + s * k * (k + 1)) * ts
        wo = (wo + s * 2.0) * ts
        wc = (wc + s * 2.0 * k) * ts
    eb, i2 = torch.exp(-tb), 1.0 / (tb * tb)
    small = t < 0.5
    wm = torch.where(small, wm, (2.0 - eb * (tb * tb + 2.0 * tb + 2.0)) * i2)
    wo = torch.where(small, wo, 1.0 - 2.0 * (eb + tb - 1.0) * i2)
    wc = torch.where(small, wc, 2.0 * (tb - 2.0 + eb * (tb + 2.0)) * i2)
    return e, wm, wo, wc


def _control(yM, yO, yP, hM, hP):
    """monotonic Bezier control point of the upwind interval"""
    dm, dp = yO - yM, yP - yO
    yp = hM / (hP * (hM + hP)) * dp + hP / (hM * (hM + hP)) * dm
    w, u = 0.5 * hM * yp, 0.5 * hP * yp
    u = torch.where(u * (u - dp) > 0, dp, u)
    c = yO - hM / hP * u
    c = torch.where((dm - w) * w < 0, yM, c)
    return torch.where(dm * dp <= 0, yO, c)


class _Stencil:
    """bilinear interpolation on a periodic plane at fixed offsets (cells) per ray"""

    def __init__(self, fx, fy, nx, ny, dev):
        ix, iy = np.floor(fx).astype(np.int64), np.floor(fy).astype(np.int64)
        tx, ty = fx - ix, fy - iy
        i, j = np.arange(nx), np.arange(ny)
        self.idx, self.w = [], []
        for b in (0, 1):
            for a in (0, 1):
                jj = (j[None, :] + iy[:, None] + b) % ny
                ii = (i[None, :] + ix[:, None] + a) % nx
                idx = (jj[:, :, None] * nx + ii[:, None, :]).reshape(len(fx), 1, ny * nx)
                self.idx.append(torch.tensor(idx, device=dev))
                w = (tx if a else 1 - tx) * (ty if b else 1 - ty)
                self.w.append(torch.tensor(w, device=dev)[:, None, None])

    def __call__(self, q):
        """q (rays, frequencies, points)"""
        out = 0.0
        for idx, w in zip(self.idx, self.w):
            out = out + w * torch.gather(q, 2, idx.expand(-1, q.shape[1], -1))
        return out


def _sweep(a, src, mu, az, x, dich=None, orient=None, dich1=None):
    """Stokes vectors and Lambda* of rays of one hemisphere, plane by plane in sweep order:
    yields (plane index, I [ns] (rays, freq, points), Lambda*, profile). src: unknowns
    (nz, ny, nx, 1 or 6); dich (.., 5), orient, dich1 (.., 3): multilevel line terms."""
    dev = a["chi"].device
    nx, ny, nz = a["nx"], a["ny"], a["nz"]
    n, R, F = nx * ny, len(mu), len(x)
    pol = src.shape[-1] == 6
    st = np.sqrt(np.maximum(0.0, 1.0 - mu * mu))
    om = np.stack([st * np.cos(az), st * np.sin(az), mu], 0)
    up = mu[0] > 0
    xt = torch.tensor(x, device=dev)[None, :, None]
    mut = torch.tensor(mu, device=dev)[:, None, None]
    omt = torch.tensor(om, device=dev)
    T = torch.tensor(_tensors(mu, az), device=dev)
    mult = torch.tensor([1.0, 1.0, 2.0, 2.0, 2.0, 2.0], device=dev, dtype=torch.float64)
    t1 = torch.stack([math.sqrt(1.5) * omt[2], -2 * math.sqrt(0.75) * omt[0], -2 * math.sqrt(0.75) * omt[1]], -1)
    flat = {k: a[k].reshape(nz, n) for k in ("chi", "vel", "bx", "by", "bz") if a.get(k) is not None}
    ns = 4 if pol else 1

    def node(k):
        """per node of plane k: phi, eta (I[, Q, U, V]), eps (ns)"""
        xs = xt - flat["vel"][k][None, None, :] * mut
        phi = torch.exp(-xs * xs)
        e0 = flat["chi"][k] * phi
        s = src[k].reshape(n, -1)
        if not pol:
            return phi, [e0], [e0 * s[:, 0]]
        b = 2.0 * a["gbar"] * a["zeta"] * sum(omt[i][:, None] * flat[c][k][None, :]
                                              for i, c in enumerate(("bx", "by", "bz")))
        S = torch.einsum("ric,c,nc->irn", T, mult, s)
        eV = b[:, None, :] * xs * e0
        eps = [e0 * S[i][:, None, :] for i in range(3)] + [s[:, 0] * eV]
        eta = [e0, None, None, eV]
        if orient is not None:
            eps[3] = eps[3] + e0 * torch.einsum("rc,nc->rn", t1, orient[k].reshape(n, 3))[:, None, :]
        if dich1 is not None:
            eta[3] = eta[3] + e0 * torch.einsum("rc,nc->rn", t1, dich1[k].reshape(n, 3))[:, None, :]
        if dich is not None:
            d = dich[k].reshape(n, 5)
            d = torch.cat([torch.ones_like(d[:, :1]), d], -1)
            D = torch.einsum("ric,c,nc->irn", T, mult, d)
            eta[:3] = [e0 * D[i][:, None, :] for i in range(3)]
        return phi, eta, eps

    ks = list(range(nz)) if up else list(range(nz - 1, -1, -1))
    z, amu = a["z"], np.abs(mu)
    dx, dy = a["lx"] / nx, a["ly"] / ny
    prev, cur, nxt = None, node(ks[0]), node(ks[1])
    zero = torch.zeros((R, F, n), device=dev, dtype=torch.float64)
    I = [zero + a["bpl"].reshape(nz, n)[ks[0]] if up else zero] + [zero] * (ns - 1)
    yield ks[0], I, zero, cur[0]
    for q in range(1, nz):
        prev, cur = cur, nxt
        has_p = q + 1 < nz
        nxt = node(ks[q + 1]) if has_p else None
        ds = abs(z[ks[q]] - z[ks[q - 1]]) / amu
        M = _Stencil(-ds * om[0] / dx, -ds * om[1] / dy, nx, ny, dev)
        etaM = [None if e is None else M(e) for e in prev[1]]
        SM = [M(e) / etaM[0] for e in prev[2]]
        IM = [M(i) for i in I]
        etaO = cur[1]
        SO = [e / etaO[0] for e in cur[2]]
        t = 0.5 * (etaM[0] + etaO[0]) * torch.tensor(ds, device=dev)[:, None, None]
        e, wm, wo, wc = _coefficients(t)
        if has_p:
            dp = abs(z[ks[q + 1]] - z[ks[q]]) / amu
            Pt = _Stencil(dp * om[0] / dx, dp * om[1] / dy, nx, ny, dev)
            etaP = Pt(nxt[1][0])
            tp = 0.5 * (etaO[0] + etaP) * torch.tensor(dp, device=dev)[:, None, None]
            cM = [_control(SM[i], SO[i], Pt(nxt[2][i]) / etaP, t, tp) for i in range(ns)]
        else:
            cM = [0.5 * (SM[i] + SO[i]) for i in range(ns)]
        r = [e * IM[i] + wm * SM[i] + wo * SO[i] + wc * cM[i] for i in range(ns)]
        if pol:
            pm, po = wm + 0.5 * wc, wo + 0.5 * wc
            kM = [None if v is None else v / etaM[0] for v in etaM]
            kO = [None if v is None else v / etaO[0] for v in etaO]
            on = [i for i in (1, 2, 3) if kO[i] is not None]
            r[0] = r[0] - pm * sum(kM[i] * IM[i] for i in on)
            for i in on:
                r[i] = r[i] - pm * kM[i] * IM[0]
            num = r[0] - po * sum(kO[i] * r[i] for i in on)
            I0 = num / (1.0 - po * po * sum(kO[i] * kO[i] for i in on))
            r = [I0] + [r[i] - po * kO[i] * I0 if i in on else r[i] for i in (1, 2, 3)]
        I = r
        yield ks[q], I, wo + (wc if has_p else 0.5 * wc), cur[0]


def _formal(a, src, case, **line):
    """J^K_Q (nz, ny, nx, nj), Lambda-bar* (nz, ny, nx) and J^1_Q (nz, ny, nx, 3)"""
    mu, az, w = _rays(case)
    x, wf = _freqs(case)
    dev = a["chi"].device
    nx, ny, nz = a["nx"], a["ny"], a["nz"]
    pol = src.shape[-1] == 6
    half = len(mu) // 2
    chunk = max(1, int(6e6 // (len(x) * nx * ny)))
    wft = torch.tensor(wf, device=dev)[None, :, None]
    J, L, J1 = [0.0] * nz, [0.0] * nz, [0.0] * nz
    for h in (0, half):
        for m0 in range(h, h + half, chunk):
            m = slice(m0, min(m0 + chunk, h + half))
            T = torch.tensor(_tensors(mu[m], az[m]), device=dev)
            wm = torch.tensor(w[m], device=dev)
            st = np.sqrt(1.0 - mu[m] ** 2)
            t1 = torch.tensor(np.stack([math.sqrt(1.5) * mu[m], -math.sqrt(0.75) * st * np.cos(az[m]),
                                        -math.sqrt(0.75) * st * np.sin(az[m])], -1), device=dev)
            for k, I, ls, phi in _sweep(a, src, mu[m], az[m], x, **line):
                wt = wft * phi
                wt = wt / wt.sum(1, keepdim=True) * wm[:, None, None]
                L[k] = L[k] + (wt * ls).sum((0, 1))
                if pol:
                    Ibar = torch.stack([(wt * I[i]).sum(1) for i in range(3)], 1)
                    J[k] = J[k] + torch.einsum("ric,rin->nc", T, Ibar)
                    if line:
                        J1[k] = J1[k] + torch.einsum("rc,rn->nc", t1, (wt * I[3]).sum(1))
                else:
                    J[k] = J[k] + (wt * I[0]).sum((0, 1))[:, None]
    jkq = torch.stack(J).reshape(nz, ny, nx, -1)
    return jkq, torch.stack(L).reshape(nz, ny, nx), torch.stack(J1).reshape(nz, ny, nx, 3) if line else None


def _hanle(a, s2, eps):
    """(1 - i (1-eps) Gamma K) S for K = 2 as a real 5x5 matrix per voxel; returns the matrix"""
    f = -(1.0 - eps) / a["bcrit"]
    gx, gy, gz = (f * a[k] for k in ("bx", "by", "bz"))
    s6, o, i = math.sqrt(6.0), torch.zeros_like(gx), torch.ones_like(gx)
    rows = [[i, s6 * gy, -s6 * gx, o, o],
            [-0.5 * s6 * gy, i, -gz, gy, -gx],
            [0.5 * s6 * gx, gz, i, gx, gy],
            [o, -gy, -gx, i, -2 * gz],
            [o, gx, -gy, 2 * gz, i]]
    return torch.stack([torch.stack(r, -1) for r in rows], -2)


def _update(a, jkq, ls, rho, f):
    """Jacobi update with the right-hand side f (nz, ny, nx, nl)"""
    e = a["eps"]
    s00 = rho[..., 0] + ((1 - e) * jkq[..., 0] + f[..., 0] - rho[..., 0]) / (1 - (1 - e) * ls)
    if rho.shape[-1] == 1:
        return s00[..., None]
    r = (1 - e)[..., None] * jkq[..., 1:] + f[..., 1:]
    return torch.cat([s00[..., None], torch.linalg.solve(_hanle(a, None, e), r[..., None])[..., 0]], -1)


def _thermal(a, nl):
    f = torch.zeros(a["chi"].shape + (nl,), device=a["chi"].device, dtype=torch.float64)
    f[..., 0] = a["eps"] * a["bpl"]
    return f


def _iterate(a, rho, case, n, f=None):
    f = _thermal(a, rho.shape[-1]) if f is None else f
    for _ in range(n):
        jkq, ls, _ = _formal(a, rho, case)
        rho = _update(a, jkq, ls, rho, f)
    return rho


def _emergent(a, rho, case, mu, az):
    x, _ = _freqs(case)
    for k, I, _, _ in _sweep(a, rho, mu, az, x):
        pass
    return torch.stack(I, -1).reshape(len(mu), len(x), a["ny"], a["nx"], len(I))


# multigrid: grid transfer matrices per axis, coarse node = every other fine node
def _prolong_matrices(a):
    def periodic(nf):
        m = np.zeros((nf, nf // 2))
        for i in range(nf):
            m[i, i // 2] += 0.5 if i % 2 else 1.0
            if i % 2:
                m[i, (i // 2 + 1) % (nf // 2)] += 0.5
        return m
    z, nf = a["z"], a["nz"]
    nc = (nf + 1) // 2 if nf % 2 else nf // 2
    mz = np.zeros((nf, nc))
    for k in range(nf):
        if k % 2 == 0:
            mz[k, k // 2] = 1.0
        else:
            k0 = min(k // 2, nc - 2)
            t = (z[k] - z[2 * k0]) / (z[2 * k0 + 2] - z[2 * k0])
            mz[k, k0], mz[k, k0 + 1] = 1.0 - t, t
    return [torch.tensor(m, device=a["chi"].device) for m in (mz, periodic(a["ny"]), periodic(a["nx"]))]


def _coarsen(a):
    nc = (a["nz"] + 1) // 2 if a["nz"] % 2 else a["nz"] // 2
    c = dict(a, nx=a["nx"] // 2, ny=a["ny"] // 2, nz=nc, z=a["z"][0:2 * nc:2])
    for k, v in a.items():
        if torch.is_tensor(v):
            c[k] = v[0:2 * nc:2, 0::2, 0::2].contiguous()
    return c


def _operator(a, rho, case):
    """A(rho) of the statistical equilibrium written as A(rho) = f"""
    jkq, _, _ = _formal(a, rho, case)
    e = (1 - a["eps"])[..., None]
    out = rho - e * jkq
    if rho.shape[-1] == 6:
        s2 = (_hanle(a, None, a["eps"]) @ rho[..., 1:, None])[..., 0]
        out = torch.cat([out[..., :1], s2 - e * jkq[..., 1:]], -1)
    return out


def _vcycle(a, rho, f, case, levels):
    if levels == 1:
        return _iterate(a, rho, case, 8, f)
    mz, my, mx = _prolong_matrices(a)
    den = torch.einsum("K,J,I->KJI", mz.sum(0), my.sum(0), mx.sum(0))[..., None]

    def restrict(v):
        return torch.einsum("kK,jJ,iI,kjic->KJIc", mz, my, mx, v) / den
    rho = _iterate(a, rho, case, 2, f)
    c = _coarsen(a)
    rc = restrict(rho)
    fc = _operator(c, rc, case) + restrict(f - _operator(a, rho, case))
    d = _vcycle(c, rc, fc, case, levels - 1) - rc
    rho = rho + torch.einsum("kK,jJ,iI,KJIc->kjic", mz, my, mx, d)
    return _iterate(a, rho, case, 4, f)


# five-level atom
def _line_tables(atom):
    g = 2.0 * np.asarray(atom["J"]) + 1.0
    up, lo = atom["lines"][:, 0], atom["lines"][:, 1]
    dE = atom["E"][up] - atom["E"][lo]
    s = g[up] / g[lo] * atom["A"] / dE ** 2
    r3 = (dE / dE[0]) ** 3
    bul = atom["A"] / r3
    return g, up, lo, dE, r3, s / s[0], bul, g[up] / g[lo] * bul


def _lte(atom, kT):
    g = torch.tensor(2.0 * np.asarray(atom["J"]) + 1.0, device=kT.device)
    w = g * torch.exp(-torch.tensor(atom["E"], device=kT.device) / kT[..., None])
    return w / w.sum(-1, keepdim=True)


def _lines(a, atom, pops):
    """per line the two-level atmosphere (opacity, Planck function) and the source function"""
    g, up, lo, dE, r3, s, _, _ = _line_tables(atom)
    out = []
    for k, (u, l) in enumerate(zip(up, lo)):
        n = pops[..., l] - pops[..., u] * (g[l] / g[u])
        b = dict(a, chi=a["chi"] * s[k] * n, bpl=r3[k] / torch.expm1(dE[k] / a["kT"]))
        out.append((b, r3[k] * pops[..., u] / (pops[..., l] * (g[u] / g[l]) - pops[..., u])))
    return out


def _collisions(atom, kT):
    g, up, lo, dE, *_ = _line_tables(atom)
    cul = atom["eps"] / (1.0 - atom["eps"]) * atom["A"]
    return cul, torch.stack([g[u] / g[l] * cul[k] * torch.exp(-dE[k] / kT) for k, (u, l) in enumerate(zip(up, lo))], -1)


def _ml_exact(case, d):
    a, atom, pops = d["atm"], d["atom"], d["x"]
    g, up, lo, _, _, _, bul, blu = _line_tables(atom)
    jb, ls, S = [], [], []
    for b, s in _lines(a, atom, pops):
        j, l, _ = _formal(b, s[..., None], case)
        jb.append(j[..., 0])
        ls.append(l)
        S.append(s)
    cul, clu = _collisions(atom, a["kT"])
    n = len(ML_J)
    M = torch.zeros(pops.shape[:-1] + (n, n), device=pops.device, dtype=torch.float64)
    for k, (u, l) in enumerate(zip(up, lo)):
        je = jb[k] - ls[k] * S[k]
        pul = atom["A"][k] * (1 - ls[k]) + bul[k] * je + cul[k]
        plu = blu[k] * je + clu[..., k]
        M[..., l, u] += pul
        M[..., u, u] -= pul
        M[..., u, l] += plu
        M[..., l, l] -= plu
    M[..., 0, :] = 1.0
    rhs = torch.zeros_like(pops)
    rhs[..., 0] = 1.0
    return {"jbar": torch.stack(jb), "lstar": torch.stack(ls), "x": torch.linalg.solve(M, rhs[..., None])[..., 0]}


# angular-momentum coupling symbols (Racah's sums; integer arguments)
_f = math.factorial


def _tri(a, b, c):
    return abs(a - b) <= c <= a + b


def _dlt(a, b, c):
    return Fraction(_f(a + b - c) * _f(a - b + c) * _f(b + c - a), _f(a + b + c + 1))


@lru_cache(maxsize=None)
def _w3j(a, b, c, x, y, z):
    if x + y + z or not _tri(a, b, c) or abs(x) > a or abs(y) > b or abs(z) > c:
        return 0.0
    pre = _dlt(a, b, c) * _f(a + x) * _f(a - x) * _f(b + y) * _f(b - y) * _f(c + z) * _f(c - z)
    s = Fraction(0)
    for k in range(max(0, b - c - x, a - c + y), min(a + b - c, a - x, b + y) + 1):
        s += Fraction((-1) ** k, _f(k) * _f(c - b + x + k) * _f(c - a - y + k) * _f(a + b - c - k) * _f(a - x - k) *
                      _f(b + y - k))
    return (-1) ** (a - b - z) * float(s) * math.sqrt(pre)


@lru_cache(maxsize=None)
def _w6j(a, b, c, d, e, f):
    if not (_tri(a, b, c) and _tri(a, e, f) and _tri(d, b, f) and _tri(d, e, c)):
        return 0.0
    pre = _dlt(a, b, c) * _dlt(a, e, f) * _dlt(d, b, f) * _dlt(d, e, c)
    lo, hi = (a + b + c, a + e + f, d + b + f, d + e + c), (a + b + d + e, b + c + e + f, c + a + f + d)
    s = Fraction(0)
    for k in range(max(lo), min(hi) + 1):
        den = 1
        for t in lo:
            den *= _f(k - t)
        for t in hi:
            den *= _f(t - k)
        s += Fraction((-1) ** k * _f(k + 1), den)
    return float(s) * math.sqrt(pre)


@lru_cache(maxsize=None)
def _w9j(a, b, c, d, e, f, g, h, i):
    lo, hi = max(abs(a - i), abs(h - d), abs(b - f)), min(a + i, h + d, b + f)
    return sum((2 * x + 1) * _w6j(a, b, c, f, i, x) * _w6j(d, e, f, b, x, h) * _w6j(g, h, i, x, a, d)
               for x in range(lo, hi + 1))


def _wk(K, J, Jp):
    return 0.0 if 2 * J < K else (-1) ** (1 + J + Jp) * math.sqrt(3 * (2 * J + 1)) * _w6j(1, 1, K, J, J, Jp)


def _multipole_index():
    """(level, K, Q) -> position of the complex multipole, and the map from the real unknowns"""
    cb = [(i, K, Q) for i, J in enumerate(ML_J) for K in range(2 * J + 1) for Q in range(-K, K + 1)]
    rb = [(i, K, Q, p) for i, J in enumerate(ML_J) for K in range(2 * J + 1) for Q in range(K + 1)
          for p in range(2 if Q else 1)]
    at = {b: n for n, b in enumerate(cb)}
    C = np.zeros((len(cb), len(rb)), dtype=complex)
    for n, (i, K, Q, p) in enumerate(rb):
        v = 1j if p else 1.0
        C[at[(i, K, Q)], n] = v
        if Q:
            C[at[(i, K, -Q)], n] = (-1) ** Q * np.conj(v)
    return cb, rb, at, C


def _mlpol_matrices(atom):
    """fixed complex matrices of the rate equations: constant part, and one per voxel quantity
    (C_lu per line; J^Kr_Qr per line; population terms of J^0_0 and of A per line; B per axis)"""
    g, up, lo, _, _, _, bul, blu = _line_tables(atom)
    cb, rb, at, C = _multipole_index()
    n, jk = len(cb), [(K, Q) for K in range(3) for Q in range(-K, K + 1)]
    nl, A = len(up), atom["A"]
    Mr = np.zeros((nl, len(jk), n, n), dtype=complex)
    pop, spop = np.zeros((nl, n, n), dtype=complex), np.zeros((nl, n, n), dtype=complex)
    const, unit, Mh = np.zeros((n, n), dtype=complex), np.zeros((nl, n, n), dtype=complex), np.zeros((3, n, n), dtype=complex)
    cul = atom["eps"] / (1.0 - atom["eps"]) * A

    def radiative(k, i, row, lev, weight, term):
        """add sign * sum over (K', Q') of level lev and (Kr, Qr)"""
        _, K, Q = cb[row]
        for Kp in range(2 * ML_J[lev] + 1):
            for Qp in range(-Kp, Kp + 1):
                for c, (Kr, Qr) in enumerate(jk):
                    v = term(K, Q, Kp, Qp, Kr, Qr)
                    if v:
                        v *= weight * math.sqrt(3 * (2 * K + 1) * (2 * Kp + 1) * (2 * Kr + 1))
                        Mr[k, c, row, at[(lev, Kp, Qp)]] += v
                        if K == Kp == Kr == 0:
                            pop[k, row, at[(lev, Kp, Qp)]] += v
    for k, (u, l) in enumerate(zip(up, lo)):
        Ju, Jl = ML_J[u], ML_J[l]

        def relax(Ja, Jb, extra):
            def term(K, Q, Kp, Qp, Kr, Qr):
                if (K + Kp + Kr) % 2:
                    return 0.0
                return (-1) ** (1 + Jb - Ja + (Kr if extra else 0) + Qp) * _w6j(K, Kp, Kr, Ja, Ja, Ja) * \
                    _w6j(1, 1, Kr, Ja, Ja, Jb) * _w3j(K, Kp, Kr, Q, -Qp, Qr)
            return term
        for row, (lev, K, Q) in enumerate(cb):
            if lev == u:
                radiative(k, u, row, l, (2 * Jl + 1) * blu[k], lambda K, Q, Kp, Qp, Kr, Qr: (-1) ** (Kp + Qp) *
                          _w9j(Ju, Jl, 1, Ju, Jl, 1, K, Kp, Kr) * _w3j(K, Kp, Kr, -Q, Qp, -Qr))
                radiative(k, u, row, u, -(2 * Ju + 1) * bul[k], relax(Ju, Jl, False))
                const[row, row] -= A[k] + cul[k]
                if K == 0:
                    spop[k, row, row] -= A[k]
            elif lev == l:
                radiative(k, l, row, u, (2 * Ju + 1) * bul[k], lambda K, Q, Kp, Qp, Kr, Qr: (-1) ** (Kr + Kp + Qp) *
                          _w9j(Ju, Jl, 1, Ju, Jl, 1, Kp, K, Kr) * _w3j(K, Kp, Kr, -Q, Qp, -Qr))
                radiative(k, l, row, l, -(2 * Jl + 1) * blu[k], relax(Jl, Ju, True))
                if (u, K, Q) in at:
                    v = (2 * Ju + 1) * A[k] * (-1) ** (1 + Ju + Jl + K) * _w6j(Ju, Ju, K, Jl, Jl, 1)
                    const[row, at[(u, K, Q)]] += v
                    if K == 0:
                        spop[k, row, at[(u, K, Q)]] += v
                unit[k, row, row] -= 1.0
        unit[k, at[(u, 0, 0)], at[(l, 0, 0)]] += math.sqrt(g[l] / g[u])
        const[at[(l, 0, 0)], at[(u, 0, 0)]] += cul[k] * math.sqrt(g[u] / g[l])
    larmor = -2.0 * math.pi * 1.3996e6
    for row, (i, K, Q) in enumerate(cb):
        Mh[2, row, row] += 1j * larmor * Q
        if Q > -K:
            f = 0.5 * math.sqrt((K + Q) * (K - Q + 1))
            Mh[0, row, at[(i, K, Q - 1)]] += 1j * larmor * f
            Mh[1, row, at[(i, K, Q - 1)]] += larmor * f
        if Q < K:
            f = 0.5 * math.sqrt((K - Q) * (K + Q + 1))
            Mh[0, row, at[(i, K, Q + 1)]] += 1j * larmor * f
            Mh[1, row, at[(i, K, Q + 1)]] -= larmor * f
    return const, np.concatenate([unit, Mr.reshape(-1, n, n), pop, spop, Mh]), jk


def _mlpol_exact(case, d):
    a, atom, x = d["atm"], d["atom"], d["x"]
    dev = x.device
    g, up, lo, _, _, _, bul, blu = _line_tables(atom)
    cb, rb, at, C = _multipole_index()
    xc = x.to(torch.complex128) @ torch.tensor(C.T, device=dev)
    k00 = [rb.index((i, 0, 0, 0)) for i in range(len(ML_J))]
    pops = x[..., k00] * torch.tensor(np.sqrt(g), device=dev)
    jb, ls, src = [], [], []
    for k, (b, S) in enumerate(_lines(a, atom, pops)):
        u, l = int(up[k]), int(lo[k])
        Ju, Jl = ML_J[u], ML_J[l]

        def parts(c):
            return [c[0].real] + [p for v in c[1:] for p in (v.real, v.imag)]
        em = {K: [torch.conj(xc[..., at[(u, K, Q)]]) / xc[..., at[(u, 0, 0)]].real * _wk(K, Ju, Jl) * S
                  for Q in range(K + 1)] for K in (1, 2)}
        al, au = blu[k] * math.sqrt(2 * Jl + 1), bul[k] * math.sqrt(2 * Ju + 1)
        den = al * xc[..., at[(l, 0, 0)]].real - au * xc[..., at[(u, 0, 0)]].real
        dc = {}
        for K in (1, 2):
            dc[K] = []
            for Q in range(K + 1):
                num = -au * _wk(K, Ju, Jl) * xc[..., at[(u, K, Q)]]
                if 2 * Jl >= K:
                    num = num + (-1) ** K * al * _wk(K, Jl, Ju) * xc[..., at[(l, K, Q)]]
                dc[K].append(torch.conj(num / den))
        j, lb, j1 = _formal(b, torch.stack([S] + parts(em[2]), -1), case, orient=torch.stack(parts(em[1]), -1),
                            dich=torch.stack(parts(dc[2]), -1), dich1=torch.stack(parts(dc[1]), -1))
        jb.append(torch.cat([j[..., :1], j1, j[..., 1:]], -1))
        ls.append(lb)
        src.append(S)
    const, mats, jk = _mlpol_matrices(atom)
    _, clu = _collisions(atom, a["kT"])
    cf = [clu + 0j]
    for k in range(len(up)):
        jr = jb[k]
        col = {(0, 0): jr[..., 0] + 0j, (1, 0): jr[..., 1] + 0j, (1, 1): torch.complex(jr[..., 2], jr[..., 3]),
               (2, 0): jr[..., 4] + 0j, (2, 1): torch.complex(jr[..., 5], jr[..., 6]),
               (2, 2): torch.complex(jr[..., 7], jr[..., 8])}
        cf.append(torch.stack([col[(K, Q)] if Q >= 0 else (-1) ** Q * torch.conj(col[(K, -Q)]) for K, Q in jk], -1))
    lst, S = torch.stack(ls, -1), torch.stack(src, -1)
    cf += [-lst * S + 0j, -lst + 0j, torch.stack([a["bx"], a["by"], a["bz"]], -1) + 0j]
    n, nr = len(cb), len(rb)
    cf = torch.cat(cf, -1).reshape(-1, mats.shape[0])
    # rows of the real equations: the Q >= 0 multipoles' real and imaginary parts
    Y = torch.tensor((mats @ C).reshape(mats.shape[0], -1), device=dev)
    Y0 = torch.tensor(const @ C, device=dev)
    rows = torch.tensor([at[b[:3]] for b in rb], device=dev)
    imag = torch.tensor([b[3] for b in rb], device=dev, dtype=torch.bool)[:, None]
    k0 = torch.tensor(k00, device=dev)
    kp = torch.tensor([i for i in range(nr) if i not in k00], device=dev)
    xf, out = x.reshape(-1, nr), torch.empty_like(x).reshape(-1, nr)
    for v0 in range(0, cf.shape[0], 8192):
        v = slice(v0, v0 + 8192)
        Mv = ((cf[v] @ Y).reshape(-1, n, nr) + Y0)[:, rows, :]
        R = torch.where(imag, Mv.imag, Mv.real)
        R[:, k00[0], :] = 0.0
        R[:, k00[0], k0] = torch.tensor(np.sqrt(g), device=dev)
        rhs = torch.zeros_like(xf[v])
        rhs[:, k00[0]] = 1.0
        # population block with the old multipoles, then the multipoles with the new populations
        r1 = rhs[:, k0] - (R[:, k0][:, :, kp] @ xf[v][:, kp, None])[..., 0]
        y = torch.linalg.solve(R[:, k0][:, :, k0], r1[..., None])[..., 0]
        r2 = rhs[:, kp] - (R[:, kp][:, :, k0] @ y[..., None])[..., 0]
        out[v.start:v.start + y.shape[0], k0] = y
        out[v.start:v.start + y.shape[0], kp] = torch.linalg.solve(R[:, kp][:, :, kp], r2[..., None])[..., 0]
    return {"jbar": torch.stack(jb), "lstar": torch.stack(ls), "x": out.reshape(x.shape)}


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ml":
        return _ml_exact(case, d)
    if kind == "mlpol":
        return _mlpol_exact(case, d)
    if kind == "batch":
        out = [_iterate(a, r, case, case.get("iters", 1)) for a, r in zip(d["atms"], d["rho"])]
        return {"rho": torch.cat([r.reshape(-1, r.shape[-1]) for r in out])}
    a, rho = d["atm"], d["rho"]
    if kind == "formal":
        jkq, ls, _ = _formal(a, rho, case)
        return {"jkq": jkq, "lstar": ls}
    if kind == "jacobi":
        return {"rho": _iterate(a, rho, case, case["iters"])}
    if kind == "emergent":
        return {"stokes": _emergent(a, rho, case, d["mu"], d["az"])}
    if kind == "vcycle":
        return {"rho": _vcycle(a, rho, _thermal(a, rho.shape[-1]), case, case["levels"])}
    # gradients, by automatic differentiation of the above
    chi = a["chi"].clone().requires_grad_()
    B = torch.stack([a["bx"], a["by"], a["bz"]]).requires_grad_()
    av = dict(a, chi=chi, bx=B[0], by=B[1], bz=B[2])
    if kind == "vjp":
        e = (a["chi"] * rho[..., 0]).clone().requires_grad_()
        r = (rho / rho[..., :1]) * (e / chi)[..., None]
        out = _emergent(av, r, case, d["mu"], d["az"])
        gc, ge, gb = torch.autograd.grad(out, (chi, e, B), d["grad"])
        return {"g_chi": gc, "g_e": ge, "g_b": gb, "stokes": out.detach()}
    f = _thermal(a, rho.shape[-1]).requires_grad_()
    step = torch.utils.checkpoint.checkpoint
    r = rho
    for _ in range(case["iters"]):
        r = step(lambda c, b, q, s: _iterate(dict(a, chi=c, bx=b[0], by=b[1], bz=b[2]), q, case, 1, s), chi, B, r, f,
                 use_reentrant=False)
    out = _emergent(av, r, case, d["mu"], d["az"])
    gc, gf, gb = torch.autograd.grad(out, (chi, f, B), d["grad"])
    return {"g_chi": gc, "g_f": gf[..., 0].contiguous(), "g_b": gb, "stokes": out.detach()}
