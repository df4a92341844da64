"""Workloads of the hybrid LB/EPD time stepper, from the smallest call to the
largest run, each through the entry points a program uses.

A case is a dict of plain values; its "kind" says which entry points it takes:

  step       a handle over a batch of runs: `steps` coupled steps, then the
             fields, velocity and Q of every run read back on the device
  solve      one stateless single-chain solve on device pointers
  solve3d    the same on a 3D box
  step3d     one coupled step on a 3D box
  sur_infer  the learned surrogate: densities and their tangent
  sur_train  one training step of the surrogate

States are a structured system: composition fields with a domain size of a few
R_G on top of the quench noise, and the reverse-Poiseuille flow with the small
velocities the domains drive.  A MIXED_FP32 run's results carry FP32 precision
and a program keeps them so: they are returned in FP32; PLAIN_FP64 results in
FP64.
"""
from __future__ import annotations

import ctypes
import math

import torch

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import surrogate as S

MIXED, PLAIN = "mixed", "fp64"
DX, DT, RG, N_SEG = 1.0 / 3.0, 0.002, 1.0, 17.0
FSTAR = (RG / DX) * DT ** 2  # f* in lattice units (D_S = 1)

# the model sets the runs differ in
SYSTEMS = {
    "diblock": dict(f_a=0.5, phi_p=0.2, chi_bs=0.75),   # symmetric diblock in solvent
    "droplet": dict(f_a=0.882, phi_p=0.1, chi_bs=0.75),  # the paper's droplet system
    "vesicle": dict(f_a=0.3, phi_p=0.15, chi_bs=-0.15),  # the paper's vesicle system
}
MODEL = dict(chi_ab=1.05, chi_as=1.20, kappa_h=1.176, d_s=1.0, d_p=1.0 / 17.0)


def listed():
    return [
        # one small FP64 run, 10 steps between two looks at it: launch and latency bound
        dict(name="small_fp64", kind="step", prec=PLAIN, system="diblock", grids="64x64", ns="32", runs=1, f0=1e-6, steps=10, cg=0),
        # the benchmark batch: four runs of a 256 x 512 channel at four shear amplitudes
        dict(name="channel_mixed", kind="step", prec=MIXED, system="diblock", grids="256x512", ns="64", runs=4, f0=1.6e-5, steps=4, cg=0),
        # the same with the exact step (convection of Phi and the CG inversion)
        dict(name="channel_mixed_exact", kind="step", prec=MIXED, system="diblock", grids="256x512", ns="64", runs=4, f0=1.6e-5, steps=1, cg=100),
        # the same batch in FP64 throughout
        dict(name="channel_fp64", kind="step", prec=PLAIN, system="diblock", grids="256x512", ns="64", runs=4, f0=1.6e-5, steps=1, cg=0),
        # an ensemble of 32 runs of uneven grids and contour lengths
        dict(name="ensemble_mixed", kind="step", prec=MIXED, system="diblock", grids="128x128,256x128,256x512,512x256", ns="32,64,96,128", runs=32, f0=1e-5, steps=2, cg=0),
        # the large run that forms vesicles
        dict(name="vesicle_mixed", kind="step", prec=MIXED, system="vesicle", grids="1024x2048", ns="128", runs=1, f0=8e-6, steps=2, cg=0),
        # the paper's own system: an ensemble of 150 x 150 boxes (not a power of two), N_s = 17
        dict(name="paper150_mixed", kind="step", prec=MIXED, system="droplet", grids="150x150", ns="17", runs=64, f0=1e-3, steps=8, cg=0),
        # a single stateless solve, as a program with its own integrator calls it
        dict(name="solve_mixed", kind="solve", prec=MIXED, system="diblock", ny=128, nx=128, ns=64),
        # a solve on a 3D box with ragged sides
        dict(name="solve3d_mixed", kind="solve3d", prec=MIXED, system="vesicle", nz=48, ny=90, nx=96, ns=32),
        # a coupled step on a 3D box
        dict(name="step3d_fp64", kind="step3d", prec=PLAIN, system="diblock", nz=64, ny=128, nx=128, ns=16, f0=2.0),
        # the surrogate's inference (densities and tangent) and training step on the channel batch
        dict(name="surrogate_infer", kind="sur_infer", batch=4, ny=256, nx=512),
        dict(name="surrogate_train", kind="sur_train", batch=4, ny=256, nx=512),
    ]


# ---------------------------------------------------------------------------
# draws
# ---------------------------------------------------------------------------

def _smooth_even(lo, hi):
    """Even lengths 2^a 3^b 5^c in [lo, hi]."""
    out = []
    for v in range(lo + lo % 2, hi + 1, 2):
        w = v
        for p in (2, 3, 5):
            while w % p == 0:
                w //= p
        if w == 1:
            out.append(v)
    return out


def _log_choice(rng, values):
    """A value, spread over the logarithm of the range."""
    t = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / t)))


POW2 = [64, 128, 256, 512, 1024, 2048]
ANY = _smooth_even(30, 480)
SUR = [v for v in _smooth_even(48, 512) if v % 16 == 0]


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["solve", "solve3d", "step3d", "sur_infer", "sur_train"])
    system = rng.choice(sorted(SYSTEMS))
    if kind == "step":
        prec = rng.choice([MIXED, MIXED, MIXED, PLAIN])
        pow2 = rng.random() < 0.6
        sides = [v for v in POW2 if prec == MIXED or v <= 512] if pow2 else ANY
        ny, nx = _log_choice(rng, sides), _log_choice(rng, sides)
        ns = 2 * rng.randint(8, 64) if pow2 else rng.randint(16, 64)
        most = 2.6e8 if prec == MIXED else 3.2e7  # sites x contour steps of a step
        most = most / 3 if not pow2 else most
        while ny * nx * ns > most:
            ny, nx = (ny, max(v for v in sides if v < nx)) if nx >= ny else (max(v for v in sides if v < ny), nx)
        if ny & (ny - 1) == 0 and nx & (nx - 1) == 0:  # N_s is even on power-of-two grids
            ns += ns % 2
        runs = max(1, min(64, int(math.exp(rng.uniform(0, math.log(max(1.0, most / (ny * nx * ns))))))))
        steps = max(1, min(4, int(most / (ny * nx * ns * runs))))
        cg = 100 if prec == MIXED and ny * nx * ns * runs < most / 6 and rng.random() < 0.25 else 0
        return dict(kind=kind, prec=prec, system=system, grids=f"{ny}x{nx}", ns=str(ns), runs=runs, f0=10.0 ** rng.uniform(-7, -5),
                    steps=1 if cg else steps, cg=cg)
    if kind == "solve":
        pow2 = rng.random() < 0.5
        sides = POW2[:5] if pow2 else ANY
        ny, nx = _log_choice(rng, sides), _log_choice(rng, sides)
        return dict(kind=kind, prec=rng.choice([MIXED, PLAIN]), system=system, ny=ny, nx=nx, ns=2 * rng.randint(8, 48))
    if kind in ("solve3d", "step3d"):
        sides = _smooth_even(24, 128)
        nz, ny, nx = (_log_choice(rng, sides) for _ in range(3))
        if kind == "step3d":
            return dict(kind=kind, prec=PLAIN, system=system, nz=nz, ny=ny, nx=nx, ns=rng.randint(8, 16), f0=rng.uniform(0.5, 2.0))
        return dict(kind=kind, prec=rng.choice([MIXED, MIXED, PLAIN]), system=system, nz=nz, ny=ny, nx=nx, ns=rng.randint(8, 32))
    ny, nx = _log_choice(rng, SUR), _log_choice(rng, SUR)
    return dict(kind=kind, batch=rng.randint(1, max(1, min(8, 4 * 256 * 512 // (ny * nx)))), ny=ny, nx=nx)


# ---------------------------------------------------------------------------
# runs and inputs
# ---------------------------------------------------------------------------

def _params(case, ny, nx, ns, f0=0.0):
    return P.RunParams(nx=nx, ny=ny, ns=ns, precision=P.MIXED_FP32 if case.get("prec", MIXED) == MIXED else P.PLAIN_FP64,
                       f0=f0, **MODEL, **SYSTEMS[case.get("system", "diblock")])


def _runs(case):
    """(ny, nx, ns, f0) of every run of a step case: grids cycle fastest, then
    contour lengths; amplitudes log-spaced from f0 / 100 to f0."""
    grids = [tuple(int(v) for v in g.split("x")) for g in case["grids"].split(",")]
    nss = [int(v) for v in case["ns"].split(",")]
    R = case["runs"]
    return [(*grids[k % len(grids)], nss[(k // len(grids)) % len(nss)], case["f0"] * 100.0 ** ((k + 1 - R) / max(1, R - 1)))
            for k in range(R)]


def _lowpass(shape, gen, k0, rms):
    """Smooth random periodic fields: white noise filtered with
    exp(-(k / k0)^2), zero mean, of the given RMS; the last dimensions of
    `shape` after the first are the grid."""
    d = len(shape) - 1
    f = torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    k2 = torch.zeros((), dtype=torch.float64, device="cuda")
    for a, n in enumerate(shape[1:]):
        k = 2 * math.pi * torch.fft.fftfreq(n, d=DX, dtype=torch.float64, device="cuda")
        k2 = k2 + (k ** 2).reshape([n if i == a else 1 for i in range(d)])
    dims = tuple(range(1, d + 1))
    f = torch.fft.ifftn(torch.fft.fftn(f, dim=dims) * torch.exp(-k2 / k0 ** 2), dim=dims).real
    f = f - f.mean(dim=dims, keepdim=True)
    return rms * f / f.square().mean(dim=dims, keepdim=True).sqrt()


def _fields(grid, gen):
    """omega_{A,B,S}: domains a few R_G wide (RMS 0.05) and the quench noise."""
    noise = 2e-3 * torch.rand((3, *grid), generator=gen, dtype=torch.float64, device="cuda") - 1e-3
    return _lowpass((3, *grid), gen, 2.0, 0.05) + noise


C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0),
      (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _dot(c, v):
    """c . v for a lattice direction c and a vector field v."""
    s = torch.zeros_like(v[0])
    for ca, va in zip(c, v):
        if ca:
            s = s + ca * va
    return s


def _body_force(f0, ny):
    """Reverse-Poiseuille body force along x of the rows, lattice units (Eq. (23))."""
    f = torch.full((ny,), f0 * FSTAR, dtype=torch.float64, device="cuda")
    f[: ny // 2] *= -1
    return f


def _flow(grid, f0, gen):
    """Velocity (components first) and pre-collision populations: the steady
    reverse-Poiseuille profile (viscosity 1/6) plus driven velocities of 1e-4."""
    d = len(grid)
    ny = grid[-2]
    y = torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * ny
    prof = -(f0 * FSTAR * 3.0) * y * (y.abs() - 0.5 * ny)
    vel = _lowpass((d, *grid), gen, 2.0, 1e-4)
    vel[0] += prof[:, None]
    j = vel.clone()
    j[0] -= 0.5 * _body_force(f0, ny)[:, None]
    jj = (j * j).sum(0)
    cs, ws = (C2, W2) if d == 2 else (C3, W3)
    pop = torch.stack([w * (1 + 3 * _dot(c, j) + 4.5 * _dot(c, j) ** 2 - 1.5 * jj) for c, w in zip(cs, ws)])
    return vel, pop


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    return g


def _step_inputs(case, seed):
    gen = _gen(seed)
    for ny, nx, ns, f0 in _runs(case):
        om = _fields((ny, nx), gen)
        yield (ny, nx, ns, f0), om, *_flow((ny, nx), f0, gen)


def _workspace(nbytes):
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    return ws, (ws.data_ptr() + 255) & ~255


def _sur_fields(case, seed):
    """Field batch, the fields a diffusion step later, and target densities."""
    gen = _gen(seed)
    om = torch.stack([_fields((case["ny"], case["nx"]), gen) for _ in range(case["batch"])])
    om2 = om + torch.stack([_lowpass((3, case["ny"], case["nx"]), gen, 4.0, 1e-4) for _ in range(case["batch"])])
    # densities respond to the fields with a range of about R_G
    phi = 0.1 - 0.05 * torch.stack([_lowpass((3, case["ny"], case["nx"]), gen, 2.0, 0.05) + 0.5 * o for o in om])
    return om, om2, phi


SUR_IN, SUR_OUT, SUR_LR = 20.0, 2.5e-3, 1e-3
LAYERS, DILATIONS = ((3, 32), (32, 32), (32, 32), (32, 2)), (1, 2, 2, 4)


def _sur_params(seed):
    """Network parameters, W ~ N(0, 1 / (9 c_in)) and small biases, layer by layer."""
    gen = torch.Generator().manual_seed(seed & 0x7FFFFFFF)
    parts = []
    for ci, co in LAYERS:
        parts += [torch.randn(co * ci * 9, generator=gen) / math.sqrt(9.0 * ci), 0.05 * torch.randn(co, generator=gen)]
    return torch.cat(parts)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "step":
        inputs = list(_step_inputs(case, seed))
        runs = [_params(case, *i[0]) for i in inputs]
        h = P.EpdLb(runs)
        for r, (_, om, vel, pop) in enumerate(inputs):
            h.set_state(r, om.cpu().numpy(), pop.cpu().numpy(), vel.cpu().numpy())
        if case["cg"]:
            h.set_inversion(case["cg"], 1e-8)
        sizes = [r.n for r in runs]
        # the program's own buffers for what it reads back
        bufs = {k: [torch.empty(c * n, dtype=torch.float64, device="cuda") for n in sizes] for k, c in (("omega", 3), ("phi", 3), ("vel", 2))}
        big = {}
        for k, parts in bufs.items():
            big[k] = torch.empty(sum(p.numel() for p in parts), dtype=torch.float64, device="cuda")
            bufs[k] = list(big[k].split([p.numel() for p in parts]))
        q = torch.empty((len(runs), 2), dtype=torch.float64, device="cuda")
        st.update(h=h, bufs=bufs, big=big, q=q)
    elif kind == "solve":
        run = _params(case, case["ny"], case["nx"], case["ns"])
        om = _fields((case["ny"], case["nx"]), _gen(seed))
        nb = P.epd_prop_solve_workspace_bytes(run)
        ws, ptr = _workspace(nb)
        st.update(run=run, om=om, phi=torch.empty_like(om), q=torch.empty(2, dtype=torch.float64, device="cuda"), ws=ws, ptr=ptr, nb=nb)
    elif kind in ("solve3d", "step3d"):
        grid = (case["nz"], case["ny"], case["nx"])
        run = _params(case, case["ny"], case["nx"], case["ns"], case.get("f0", 0.0))
        gen = _gen(seed)
        om = _fields(grid, gen)
        if kind == "step3d":
            vel, pop = _flow(grid, run.f0, gen)
            nb = ctypes.c_size_t()
            if P.lib().epd_step3d_workspace_bytes(ctypes.byref(run.c()), grid[0], ctypes.byref(nb)):
                raise RuntimeError("epd_step3d_workspace_bytes")
            nb = nb.value
            st.update(vel=vel.contiguous(), pop=pop.contiguous(), force=torch.empty_like(om))
        else:
            nb = P.epd_prop_solve3d_workspace_bytes(run, grid[0])
        ws, ptr = _workspace(nb)
        st.update(run=run, om=om, phi=torch.empty_like(om), q=torch.empty(2, dtype=torch.float64, device="cuda"), ws=ws, ptr=ptr, nb=nb)
    else:
        run = P.RunParams(nx=case["nx"], ny=case["ny"], ns=64, precision=P.MIXED_FP32, **MODEL, **SYSTEMS["diblock"])
        om, om2, phi = _sur_fields(case, seed)
        st.update(sur=S.Surrogate(run, case["batch"], params=_sur_params(seed).numpy(), s_in=SUR_IN, s_out=SUR_OUT), om=om, om2=om2, phi=phi)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    keep = (lambda t: t.float()) if case.get("prec", MIXED) == MIXED else (lambda t: t)
    if kind == "step":
        h, bufs = state["h"], state["bufs"]
        h.step(case["steps"])
        for r in range(case["runs"]):
            h.fields_dev(r, bufs["omega"][r])
            h.densities_dev(r, bufs["phi"][r], state["q"][r])
            h.velocity_dev(r, bufs["vel"][r])
        with torch.cuda.stream(h.stream):
            return {**{k: keep(v) for k, v in state["big"].items()}, "q": keep(state["q"])}
    if kind == "solve":
        P.epd_prop_solve(state["run"], state["om"].data_ptr(), state["phi"].data_ptr(), state["q"].data_ptr(), state["ptr"], state["nb"],
                         torch.cuda.current_stream().cuda_stream)
        return {"phi": keep(state["phi"]), "q": keep(state["q"])}
    if kind in ("solve3d", "step3d"):
        c = ctypes.byref(state["run"].c())
        stream = torch.cuda.current_stream().cuda_stream
        om, phi, q = (state[k].data_ptr() for k in ("om", "phi", "q"))
        if kind == "solve3d":
            rc = P.lib().epd_prop_solve3d(c, case["nz"], om, phi, q, state["ptr"], state["nb"], stream)
            names = ("phi", "q")
        else:
            rc = P.lib().epd_step3d(c, case["nz"], om, state["pop"].data_ptr(), state["vel"].data_ptr(), phi, q, state["force"].data_ptr(),
                                    state["ptr"], state["nb"], stream)
            names = ("om", "pop", "vel", "phi", "q", "force")
        if rc:
            raise RuntimeError(f"{kind}: error {rc}")
        return {k: keep(state[k]) for k in names}
    sur = state["sur"]
    if kind == "sur_infer":
        phi0, phi = sur.tangent(state["om"], state["om2"])
        return {"phi0": keep(phi0), "phi": keep(phi)}
    loss = sur.train_step(state["om"], state["phi"], lr=SUR_LR)
    return {"loss": keep(loss), "params": sur.params, "m": sur.m, "v": sur.v}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _solve_flops(n, ns, axes):
    """Both chains over the contour: a forward and an inverse transform of one
    complex field per step (g and g' are real), 5 n log2 n each."""
    return ns * n * 10 * sum(math.log2(a) for a in axes)


def work(case):
    kind = case["kind"]
    if kind == "step":
        b = 4 if case["prec"] == MIXED else 8
        flops = byts = 0.0
        for ny, nx, ns, _ in _runs(case):
            n = ny * nx
            solves = 2 if not case["cg"] else 5  # one inversion iteration costs two, Phi(t) one
            flops += case["steps"] * (solves * _solve_flops(n, ns, (ny, nx)) + 11 * n * 5 * (math.log2(nx) + math.log2(ny)) + 300 * n)
            # state in and out: omega, populations, velocity; Phi out
            byts += n * (2 * 24 + 2 * 9 * b + 2 * 2 * b + 24)
        return {"bytes": byts, "flops": flops}
    if kind == "solve":
        n = case["ny"] * case["nx"]
        return {"bytes": 48.0 * n, "flops": _solve_flops(n, case["ns"], (case["ny"], case["nx"]))}
    if kind in ("solve3d", "step3d"):
        axes = (case["nz"], case["ny"], case["nx"])
        n = axes[0] * axes[1] * axes[2]
        f = _solve_flops(n, case["ns"], axes)
        if kind == "solve3d":
            return {"bytes": 48.0 * n, "flops": f}
        return {"bytes": n * 8.0 * (2 * 3 + 2 * 19 + 2 * 3 + 3 + 3), "flops": 2 * f + 16 * n * 5 * sum(math.log2(a) for a in axes) + 800 * n}
    pix = case["batch"] * case["ny"] * case["nx"]
    conv = 2 * 9 * (3 * 32 + 2 * 32 * 32 + 32 * 2) * pix
    if kind == "sur_infer":
        return {"bytes": pix * 24.0 * 4, "flops": 2 * conv}
    return {"bytes": pix * 24.0 * 2 + 16.0 * sum(co * (9 * ci + 1) for ci, co in LAYERS), "flops": 3 * conv}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------

class _Spectral:
    """Continuum wavenumbers of a periodic grid (component x first) and the
    operators built on them: first derivatives drop the Nyquist bin."""

    def __init__(self, grid):
        d = len(grid)
        self.dims = tuple(range(-d, 0))
        self.k, self.ko = [], []
        for a in range(d):  # x is the last axis
            n = grid[d - 1 - a]
            k = 2 * math.pi * torch.fft.fftfreq(n, d=DX, dtype=torch.float64, device="cuda")
            ko = k.clone()
            ko[n // 2] = 0
            shape = [1] * d
            shape[d - 1 - a] = n
            self.k.append(k.reshape(shape))
            self.ko.append(ko.reshape(shape))
        self.k2 = sum(k * k for k in self.k)

    def apply(self, f, factor):
        return torch.fft.ifftn(torch.fft.fftn(f, dim=self.dims) * factor, dim=self.dims).real

    def grad(self, f, a):
        return self.apply(f, 1j * self.ko[a])

    def lap(self, f):
        return self.apply(f, -self.k2)


def _ref_solve(om, ns, system, sp):
    """Phi and (Q_P, Q_S) of the fields om (3, grid): Eqs. (6)-(11)."""
    s = SYSTEMS[system]
    na = int(math.floor(s["f_a"] * ns + 0.5))
    ds = 1.0 / ns
    e = [torch.exp(-0.5 * N_SEG * ds * om[0]), torch.exp(-0.5 * N_SEG * ds * om[1])]
    kern = torch.exp(-RG ** 2 * ds * sp.k2)
    fac = lambda j: e[0] if j < na else e[1]  # noqa: E731
    hist = [torch.ones_like(om[0])]
    for j in range(ns):
        hist.append(fac(j + 1) * sp.apply(fac(j) * hist[-1], kern))
    qp = hist[ns].mean()
    ia, ib = torch.zeros_like(om[0]), torch.zeros_like(om[0])
    gp = torch.ones_like(om[0])
    for m in range(ns + 1):  # node m of the backward chain meets node ns - m
        j = ns - m
        t = hist[j] * gp
        if na > 0 and j <= na:
            ia += (0.5 if j in (0, na) else 1.0) * ds * t
        if na < ns and j >= na:
            ib += (0.5 if j in (na, ns) else 1.0) * ds * t
        hist[j] = None
        if m < ns:
            gp = fac(j - 1) * sp.apply(fac(j) * gp, kern)
    es = torch.exp(-om[2])
    qs = es.mean()
    phi = torch.stack([s["phi_p"] / qp * ia, s["phi_p"] / qp * ib, (1 - s["phi_p"]) / qs * es])
    return phi, torch.stack([qp, qs])


def _ref_mu(phi, om, system):
    inc = MODEL["kappa_h"] * (phi.sum(0) - 1)
    ab, as_, bs = MODEL["chi_ab"], MODEL["chi_as"], SYSTEMS[system]["chi_bs"]
    return torch.stack([ab * phi[1] + as_ * phi[2] + inc - om[0], ab * phi[0] + bs * phi[2] + inc - om[1],
                        as_ * phi[0] + bs * phi[1] + inc - om[2]])


def _ref_lb(pop, force):
    """BGK with tau = 1 and Guo's forcing (every relaxation parameter 0), then
    streaming: (populations, velocity)."""
    d = force.shape[0]
    cs, ws = (C2, W2) if d == 2 else (C3, W3)
    rho = pop.sum(0)
    j = torch.stack([sum(c[a] * pop[i] for i, c in enumerate(cs) if c[a]) for a in range(d)])
    u = (j + 0.5 * force) / rho
    uu, uf = (u * u).sum(0), (u * force).sum(0)
    out = torch.empty_like(pop)
    for i, (c, w) in enumerate(zip(cs, ws)):
        cu, cf = _dot(c, u), _dot(c, force)
        eq = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
        guo = 0.5 * w * (3 * cf + 9 * cu * cf - 3 * uf)
        out[i] = torch.roll(eq + guo, shifts=[c[a] for a in range(d)], dims=[-1 - a for a in range(d)])
    return out, u


def _ref_step(om, pop, vel, ns, system, f0, sp, cg):
    """One coupled step: (omega, pop, vel, phi, q, polymer force)."""
    d = vel.shape[0]
    v = vel * (DX / DT)
    diff = torch.tensor([MODEL["d_p"], MODEL["d_p"], MODEL["d_s"]], dtype=torch.float64, device="cuda").reshape([3] + [1] * d)
    wt = om - DT * sum(v[a] * sp.grad(om, a) for a in range(d))
    pt, _ = _ref_solve(wt, ns, system, sp)
    if cg:
        phi0, _ = _ref_solve(om, ns, system, sp)
        target = phi0 - DT * sum(sp.grad(v[a] * phi0, a) for a in range(d))
        wt, pt = _ref_invert(wt, pt, target, ns, system, sp, cg, 1e-8)
    om = wt - DT * diff * sp.lap(_ref_mu(pt, wt, system))
    phi, q = _ref_solve(om, ns, system, sp)
    s = torch.fft.fftn(((phi - pt) / diff).sum(0), dim=sp.dims)
    k2 = torch.where(sp.k2 == 0, torch.ones_like(sp.k2), sp.k2)
    force = torch.stack([FSTAR / DT * torch.fft.ifftn(s * 1j * sp.ko[a] / k2, dim=sp.dims).real for a in range(d)])
    total = force.clone()
    total[0] += _body_force(f0, om.shape[-2])[:, None]
    pop, vel = _ref_lb(pop, total)
    return om, pop, vel, phi, q, force


def _ref_invert(w, phi, target, ns, system, sp, most, tol):
    """Fletcher-Reeves inversion of the density map with one secant step as
    the line search (the exact step of App. C)."""
    n = w[0].numel()
    g = target - phi
    gg = (g * g).sum()
    d, h0, at = -g, -gg, 1.0
    for _ in range(most):
        if math.sqrt(float(gg) / n) < tol:
            break
        ht = ((target - _ref_solve(w + at * d, ns, system, sp)[0]) * d).sum()
        if h0 - ht < 0:
            at = at * h0 / (h0 - ht)
        w = w + at * d
        phi, _ = _ref_solve(w, ns, system, sp)
        g = target - phi
        new = (g * g).sum()
        beta = new / gg
        h0 = -new + beta * (g * d).sum()
        if h0 >= 0:
            beta, h0 = 0.0, -new
        d = -g + beta * d
        gg = new
    return w, phi


def _sur_layers(params):
    out, o = [], 0
    for ci, co in LAYERS:
        w = params[o : o + co * ci * 9].reshape(co, ci, 3, 3)
        o += w.numel()
        out.append((w, params[o : o + co]))
        o += co
    return out


def _conv(x, w, dil):
    return torch.nn.functional.conv2d(torch.nn.functional.pad(x, (dil,) * 4, mode="circular"), w, dilation=dil)


def _centred(x):
    return x - x.mean(dim=(-2, -1), keepdim=True)


def _ref_sur(layers, om, dom=None):
    """The network's output for the fields om and, along dom, its tangent."""
    x = SUR_IN * _centred(om)
    t = None if dom is None else SUR_IN * _centred(dom)
    for i, ((w, b), dil) in enumerate(zip(layers, DILATIONS)):
        x = _conv(x, w, dil) + b.reshape(1, -1, 1, 1)
        t = None if t is None else _conv(t, w, dil)
        if i < 3:
            x = torch.tanh(x)
            t = None if t is None else (1 - x * x) * t
    return x, t


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        parts = []
        for (ny, nx, ns, f0), om, vel, pop in _step_inputs(case, seed):
            sp = _Spectral((ny, nx))
            for _ in range(case["steps"]):
                om, pop, vel, phi, q, _ = _ref_step(om, pop, vel, ns, case["system"], f0, sp, case["cg"])
            parts.append((om.reshape(-1), phi.reshape(-1), vel.reshape(-1), q))
        om, phi, vel, q = zip(*parts)
        return {"omega": torch.cat(om), "phi": torch.cat(phi), "vel": torch.cat(vel), "q": torch.stack(q)}
    if kind == "solve":
        grid = (case["ny"], case["nx"])
        phi, q = _ref_solve(_fields(grid, _gen(seed)), case["ns"], case["system"], _Spectral(grid))
        return {"phi": phi, "q": q}
    if kind in ("solve3d", "step3d"):
        grid = (case["nz"], case["ny"], case["nx"])
        gen = _gen(seed)
        om, sp = _fields(grid, gen), _Spectral(grid)
        if kind == "solve3d":
            phi, q = _ref_solve(om, case["ns"], case["system"], sp)
            return {"phi": phi, "q": q}
        vel, pop = _flow(grid, case["f0"], gen)
        om, pop, vel, phi, q, force = _ref_step(om, pop, vel, case["ns"], case["system"], case["f0"], sp, 0)
        return {"om": om, "pop": pop, "vel": vel, "phi": phi, "q": q, "force": force}
    om, om2, phi = _sur_fields(case, seed)
    params = _sur_params(seed).cuda().double()
    s = SYSTEMS["diblock"]
    if kind == "sur_infer":
        y, t = _ref_sur(_sur_layers(params), om, om2 - om)
        out = []
        for o, dy in ((om, 0.0), (om2, t)):
            es = torch.exp(-o[:, 2:])
            ab = 0.5 * s["phi_p"] + SUR_OUT * _centred(y + dy)
            out.append(torch.cat([ab, (1 - s["phi_p"]) * es / es.mean(dim=(-2, -1), keepdim=True)], 1))
        return {"phi0": out[0], "phi": out[1]}
    params.requires_grad_(True)
    y, _ = _ref_sur(_sur_layers(params), om)
    loss = (y - _centred(phi[:, :2]) / SUR_OUT).square().mean()
    (g,) = torch.autograd.grad(loss, params)
    m, v = 0.1 * g, 1e-3 * g * g
    new = params.detach() - SUR_LR * (m / 0.1) / ((v / 1e-3).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "params": new, "m": m, "v": v}
