"""Performance cases of the TDGL + Poisson step: what users of the library have
it do, through ``Film``, ``Batch``, ``trajectory`` and ``pf_step_host``.

A case is a dict of plain values.  ``kind`` says which call a pass makes:
  film     ``Film.step(steps)``: a run in progress, each pass its next steps
  host     ``pf_step_host``: the same with P and phi in pinned host memory
  solve    ``Film.solve_potential()`` of a given polarization from phi = 0
  diag     ``Film.diagnostics()`` of a given state
  batch    ``Batch.step(steps)``: many films with voltage ramps
  adjoint  ``trajectory(...)`` and the gradient of a loss through it
``exact`` computes the same outputs with torch operations in 64 bits: its
Poisson solve is conjugate gradients preconditioned by a Fourier transform in
x and y and a tridiagonal solve in z (direct where both z faces are uniform).
"""
import math

import numpy as np
import torch

from paper_1202_6116_gb300 import adjoint, pf
from paper_1202_6116_gb300 import workloads as W
from paper_1202_6116_gb300.batch import Batch
from paper_1202_6116_gb300.film import Film

DEV = "cuda"


def listed():
    return [
        # The plain FP64 film between grounded electrodes: the smallest call, a launch every few microseconds.
        dict(name="grounded 32^3 fp64", kind="film", nx=32, ny=32, nz=32, precision="fp64", solver="pcg", rtol=1e-12,
             face="grounded", init="small", dt=0.01, steps=10),
        # The thin film with two strip electrodes as its workload ships (Jacobi-PCG).
        dict(name="strips jacobi", kind="film", nx=256, ny=256, nz=64, precision="fp32", solver="pcg", rtol=1e-8,
             face="strips", init="poled", dt=0.01, steps=10),
        # The same film with multigrid, the solver its 5000-step runs use: levels too small to fill the GPU.
        dict(name="strips multigrid", kind="film", nx=256, ny=256, nz=64, precision="fp32", solver="mg", rtol=1e-8,
             face="strips", init="poled", dt=0.01, steps=20),
        # Its FP64 twin, run to state the error of the FP32 form.
        dict(name="strips fp64", kind="film", nx=256, ny=256, nz=64, precision="fp64", solver="mg", rtol=1e-8,
             face="strips", init="poled", dt=0.01, steps=4),
        # The micron-scale film with a tip electrode: the headline workload, the largest grid.
        dict(name="tip 1024x1024x128", kind="film", nx=1024, ny=1024, nz=128, precision="fp32", solver="mg", rtol=1e-7,
             face="tip", init="stripes", dt=0.005, steps=4),
        # The open-circuit device: five air layers, a permittivity field, an odd number of planes.
        dict(name="open air 512x512x37", kind="film", nx=512, ny=512, nz=37, precision="fp32", solver="mg", rtol=1e-8,
             face="bottom", init="stripes", dt=0.005, steps=4, n_air=5),
        # The paper's predictor-corrector on a grid whose tiles are ragged in x and y.
        dict(name="predictor-corrector ragged", kind="film", nx=336, ny=216, nz=32, precision="fp32", solver="mg",
             rtol=1e-7, face="tip", init="stripes", dt=0.01, steps=4, heun=True),
        # A potential for a polarization from elsewhere, on an odd grid (no 16-byte rows).
        dict(name="solve odd 101x75x19", kind="solve", nx=101, ny=75, nz=19, precision="fp32", solver="pcg", rtol=1e-7,
             face="tip", init="stripes"),
        # Mean polarization, switched fraction and energies, taken every so many steps of a run.
        dict(name="diagnostics 512x512x64", kind="diag", nx=512, ny=512, nz=64, precision="fp32", solver="mg",
             rtol=1e-7, face="tip", init="stripes"),
        # A program that keeps its state in host memory and calls for every step.
        dict(name="host state 512x512x64", kind="host", nx=512, ny=512, nz=64, precision="fp32", solver="mg",
             rtol=1e-7, face="tip", init="stripes", dt=0.005, steps=2),
        # The hysteresis sweep: films of four sizes with their own voltage ramps in one launch.
        dict(name="hysteresis batch", kind="batch", films=30, precision="fp32", solver="mg", rtol=1e-6, dt=0.01,
             steps=20),
        # Gradient of a domain-pattern loss through the discrete adjoint (forward, recomputation, backward).
        dict(name="adjoint 128x128x32", kind="adjoint", nx=128, ny=128, nz=32, precision="fp64", solver="mg",
             rtol=1e-12, face="strips", init="poled", dt=0.01, steps=6, checkpoint_every=3),
    ]


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mg_size(rng, lo, hi):
    """An extent that halves down to an odd factor of at most 9."""
    best = None
    t = _spread(rng, lo, hi)
    for m in (1, 3, 5, 7, 9):
        v = m * 2 ** max(2, round(math.log2(t / m)))
        if best is None or abs(v - t) < abs(best - t) or rng.random() < 0.25:
            best = v
    return best


def _odd(n):
    while n % 2 == 0:
        n //= 2
    return n


def draw(rng):
    kind = rng.choice(["film"] * 6 + ["host", "solve", "diag", "batch", "adjoint"])
    if kind == "batch":
        return dict(kind="batch", films=rng.randint(4, 30), precision="fp32", solver="mg", rtol=1e-6, dt=0.01,
                    steps=rng.randint(4, 20))
    if kind == "adjoint":
        return dict(kind="adjoint", nx=_mg_size(rng, 32, 128), ny=_mg_size(rng, 32, 128), nz=_mg_size(rng, 8, 32),
                    precision="fp64", solver="mg", rtol=1e-12, face="strips", init="poled", dt=0.01,
                    steps=rng.randint(2, 6), checkpoint_every=rng.choice([2, 3]))
    face, init = rng.choice([("strips", "poled"), ("tip", "stripes"), ("grounded", "small"), ("bottom", "stripes")])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    solver = rng.choice(["mg", "mg", "pcg"])
    if solver == "mg":
        big = 640 if precision == "fp32" else 256
        nx, ny, nz = _mg_size(rng, 32, big), _mg_size(rng, 32, big), _mg_size(rng, 8, 64)
    else:
        big = 256 if precision == "fp32" else 96
        nx, ny, nz = int(_spread(rng, 32, big)), int(_spread(rng, 32, big)), int(_spread(rng, 8, 48))
    rtol = (1e-8 if precision == "fp32" else 1e-12) if face in ("strips", "grounded") else 1e-7
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, solver=solver, rtol=rtol, face=face, init=init)
    if kind in ("film", "host"):
        c.update(dt=0.005 if init == "stripes" else 0.01, steps=rng.randint(2, 6))
    if kind == "film":
        option = rng.choice(["", "", "", "heun", "noise", "air"])
        if option == "heun":
            c.update(heun=True)
        elif option == "noise":
            c.update(noise=0.05)
        elif option == "air":
            c.update(n_air=rng.randint(2, 5), nz=int(nz + rng.randint(0, 7)), face="bottom", init="stripes",
                     rtol=1e-8, dt=0.005)
            if solver == "mg":                      # the coarsest level holds at most 1024 cells
                while _odd(c["nx"]) * _odd(c["ny"]) * _odd(c["nz"]) > 1024:
                    c["nz"] += 1
    return c


# ----------------------------------------------------------------- inputs


def _faces(case):
    nx, ny = case["nx"], case["ny"]
    if case["face"] == "strips":
        return W.strip_electrodes(nx, ny)
    if case["face"] == "tip":
        return W.tip_electrode(nx, ny)
    if case["face"] == "grounded":
        return W.grounded_both(nx, ny)
    lo, hi = np.ones((ny, nx), np.int8), np.zeros((ny, nx), np.int8)      # grounded bottom, open top
    return lo, np.zeros((ny, nx)), hi, np.zeros((ny, nx))


def _eps(case):
    if not case.get("n_air"):
        return None
    e = np.full((case["nz"], case["ny"], case["nx"]), 100.0)
    e[case["nz"] - case["n_air"]:] = 1.0
    return e


def _initial(case, seed):
    """P (3, nz, ny, nx), float64 on the GPU, from the seed: the recipes of the workloads with torch's generator."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    P = torch.rand(3, nz, ny, nx, generator=g, device=DEV, dtype=torch.float32).double()
    if case["init"] == "small":                     # U[-0.01, 0.01]
        P.sub_(0.5).mul_(0.02)
    elif case["init"] == "poled":                   # +z with 1 % noise
        P.sub_(0.5).mul_(0.02)
        P[2] += 1.0
    else:                                           # <111> stripes normal to [110], width 16, 2 % noise
        P.sub_(0.5).mul_(0.04)
        sid = (torch.arange(nx, device=DEV)[None, :] + torch.arange(ny, device=DEV)[:, None]) // 16
        v = torch.tensor([[1, 1, -1], [-1, 1, -1], [-1, -1, -1], [1, -1, -1]], device=DEV, dtype=torch.float64)
        pick = torch.randint(0, 4, (int(sid.max()) + 1,), generator=g, device=DEV)
        for c in range(3):
            P[c] += (v[pick, c] / math.sqrt(3.0))[sid][None]
    if case.get("n_air"):
        P[:, nz - case["n_air"]:] = 0.0
    return P.float().double()                       # representable in FP32: every precision starts from the same state


def _workload(case):
    tl, vl, th, vh = _faces(case)
    return W.Workload(case.get("name", case["kind"]), case["nx"], case["ny"], case["nz"], None, tl, vl, th, vh,
                      eps=_eps(case), dt=case.get("dt", 0.005), rtol=case["rtol"], maxit=20000,
                      precision=case["precision"], solver=case["solver"], n_air=case.get("n_air", 0))


def _film(case, seed):
    over = dict(integrator=pf.PF_HEUN) if case.get("heun") else {}
    f = Film(_workload(case), device=DEV, P0=_initial(case, seed), **over)
    if case.get("noise"):
        f.set_noise(case["noise"], seed)
    return f


def _batch_films(case, seed):
    """(film case, ramp amplitude, ramp period, seed) of the films: the shapes and ramps of a sweep, drawn from it."""
    return [(dict(kind="film", nx=nx, ny=ny, nz=nz, precision=case["precision"], solver=case["solver"],
                  rtol=case["rtol"], face="grounded", init="small", dt=case["dt"]), amp, period, 1000 * seed + i)
            for i, ((nx, ny, nz), amp, period) in enumerate(W.batch_draws(case["films"], 4))]


COEFFS = (-1.0, 0.5, 0.8, 0.5)                      # a1, a11, a12, g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        films = _batch_films(case, seed)
        b = Batch([_film(c, s) for c, _, _, s in films], max_records=4000, record_every=10)
        for i, (_, amp, period, _) in enumerate(films):
            b.set_ramp(i, pf.PF_ZHI, amp, period)
        return dict(case=case, batch=b)
    if kind == "adjoint":
        w = _workload(case)
        P0 = _initial(case, seed).requires_grad_()
        coeffs = torch.tensor(COEFFS, dtype=torch.float64, requires_grad=True)
        vlo = torch.tensor(w.volt_lo, requires_grad=True)
        vhi = torch.tensor(w.volt_hi, requires_grad=True)
        spec = adjoint.TrajectorySpec(w, case["steps"], case["checkpoint_every"], DEV)
        return dict(case=case, spec=spec, inputs=(P0, coeffs, vlo, vhi), target=_initial(case, seed + 1)[2] * 0.9)
    f = _film(case, seed)
    s = dict(case=case, film=f)
    if kind == "host":
        s["P"] = f.P.cpu().pin_memory()
        s["phi"] = f.phi.cpu().pin_memory()
    if kind == "diag":
        f.phi.copy_(0.3 * f.P[0] + 0.1 * f.P[2])    # a potential of the field's size; the sums depend on it alone
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "film":
        f = state["film"]
        f.step(case["steps"])
        return {"P": f.P, "phi": f.phi}
    if kind == "host":
        pf.pf_step_host(state["film"].ctx, state["P"], state["phi"], case["steps"])
        return {"P": state["P"], "phi": state["phi"]}
    if kind == "solve":
        f = state["film"]
        f.phi.zero_()
        f.solve_potential()
        return {"phi": f.phi}
    if kind == "diag":
        return state["film"].diagnostics()
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        return {"P": [f.P for f in b.films], "phi": [f.phi for f in b.films]}
    P = adjoint.trajectory(*state["inputs"], state["spec"])
    loss = (P[2] - state["target"]).square().mean()
    grads = torch.autograd.grad(loss, state["inputs"])
    return {"P": P, "dP0": grads[0], "dcoeffs": grads[1], "dvolt_lo": grads[2], "dvolt_hi": grads[3]}


def work(case):
    """State read and written once a step (P and phi), and the step's own arithmetic: about 60 operations a cell for
    the update, 20 for the right-hand side, 20 for one application of the operator."""
    if case["kind"] == "batch":
        cells = sum(c["nx"] * c["ny"] * c["nz"] for c, _, _, _ in _batch_films(case, 0))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    w = 4 if case["precision"] == "fp32" else 8
    kind = case["kind"]
    if kind == "diag":
        return {"bytes": 4 * w * cells, "flops": 60 * cells}
    if kind == "solve":
        return {"bytes": 4 * w * cells, "flops": 40 * cells}
    steps = case["steps"] * (3 if kind == "adjoint" else 1)      # forward, recomputed, backward
    twice = 2 if case.get("heun") else 1
    return {"bytes": 8 * w * cells * steps * twice, "flops": 100 * cells * steps * twice}


# ------------------------------------------------- the same in 64 bits with torch


class _Poisson:
    """A phi = b with A = -div(eps grad .), dx = 1: periodic x and y, electrode (2 eps phi) or open z faces, eps a
    function of z."""

    def __init__(self, case):
        tl, vl, th, vh = _faces(case)
        e = _eps(case)
        self.nz = case["nz"]
        eps = np.ones(self.nz) if e is None else e[:, 0, 0].copy()
        t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        self.eps, self.tlo, self.thi, self.vlo, self.vhi = t(eps), t(tl), t(th), t(vl), t(vh)
        self.wz = t(2 * eps[1:] * eps[:-1] / (eps[1:] + eps[:-1]))
        self.clo, self.chi = 2 * eps[0] * self.tlo, 2 * eps[-1] * self.thi
        nx, ny = case["nx"], case["ny"]
        kx = 4 * torch.sin(torch.arange(nx // 2 + 1, device=DEV, dtype=torch.float64) * (math.pi / nx)) ** 2
        ky = 4 * torch.sin(torch.arange(ny, device=DEV, dtype=torch.float64) * (math.pi / ny)) ** 2
        lam = ky[:, None] + kx[None, :]
        wz = self.wz.tolist()
        self.cp, self.inv = [], []
        for z in range(self.nz):                    # the elimination of the tridiagonal systems, one per (ky, kx)
            d = eps[z] * lam
            d = d + (wz[z - 1] if z else float(self.clo.mean())) + (wz[z] if z < self.nz - 1 else float(self.chi.mean()))
            if z:
                d = d + wz[z - 1] * self.cp[-1]
            self.inv.append(1.0 / d)
            self.cp.append(-wz[z] / d if z < self.nz - 1 else None)
        self.wzl = wz

    def apply(self, v):
        out = 4 * v
        for dim in (1, 2):
            out -= torch.roll(v, 1, dim)
            out -= torch.roll(v, -1, dim)
        out *= self.eps[:, None, None]
        d = (v[1:] - v[:-1]) * self.wz[:, None, None]
        out[1:] += d
        out[:-1] -= d
        out[0] += self.clo * v[0]
        out[-1] += self.chi * v[-1]
        return out

    def precondition(self, r):
        f = torch.fft.rfft2(r)
        for z in range(self.nz):
            if z:
                f[z] += self.wzl[z - 1] * f[z - 1]
            f[z] *= self.inv[z]
        for z in range(self.nz - 2, -1, -1):
            f[z] -= self.cp[z] * f[z + 1]
        return torch.fft.irfft2(f, s=r.shape[1:])

    def solve(self, b, x=None):
        x = torch.zeros_like(b) if x is None else x.clone()
        nb = float(b.norm())
        if nb == 0.0:
            return torch.zeros_like(b)
        r = b - self.apply(x)
        p, rz = None, None
        for _ in range(80):
            if float(r.norm()) <= 1e-14 * nb:
                break
            z = self.precondition(r)
            rzn = float((r * z).sum())
            p = z if p is None else z + (rzn / rz) * p
            rz = rzn
            q = self.apply(p)
            a = rz / float((p * q).sum())
            x = x + a * p
            r = r - a * q
        return x

    def rhs(self, P, vlo, vhi):
        """b = -div P + electrode terms."""
        div = 0.5 * (torch.roll(P[0], -1, 2) - torch.roll(P[0], 1, 2))
        div = div + 0.5 * (torch.roll(P[1], -1, 1) - torch.roll(P[1], 1, 1))
        face = 0.5 * (P[2][1:] + P[2][:-1])
        top = torch.cat([face, (self.thi * P[2][-1])[None]])
        bottom = torch.cat([(self.tlo * P[2][0])[None], face])
        b = -(div + top - bottom)
        edge = torch.zeros_like(b)
        edge[0] += self.clo
        b = b + edge * vlo
        edge = torch.zeros_like(b)
        edge[-1] += self.chi
        return b + edge * vhi


class _Solve(torch.autograd.Function):
    """phi = A^-1 b; A is symmetric, so its gradient is one more solve."""

    @staticmethod
    def forward(ctx, b, poisson):
        ctx.poisson = poisson
        return poisson.solve(b)

    @staticmethod
    def backward(ctx, g):
        return ctx.poisson.solve(g), None


def _rate(ps, P, phi, vlo, vhi, coeffs, n_air):
    """L (-df/dP + g Lap P + E)."""
    a1, a11, a12, g = coeffs
    nz = ps.nz
    mid = 0.5 * (phi[1:] + phi[:-1])
    top = torch.cat([mid, (ps.thi * vhi + (1 - ps.thi) * phi[-1])[None]])
    bottom = torch.cat([(ps.tlo * vlo + (1 - ps.tlo) * phi[0])[None], mid])
    E = [-0.5 * (torch.roll(phi, -1, 2) - torch.roll(phi, 1, 2)),
         -0.5 * (torch.roll(phi, -1, 1) - torch.roll(phi, 1, 1)), -(top - bottom)]
    out = []
    film = nz - n_air
    for i in range(3):
        p, q, s = P[i], P[(i + 1) % 3], P[(i + 2) % 3]
        f = 2 * a1 * p + 4 * a11 * p ** 3 + 2 * a12 * p * (q * q + s * s)
        lap = torch.roll(p, 1, 2) + torch.roll(p, -1, 2) + torch.roll(p, 1, 1) + torch.roll(p, -1, 1) - 4 * p
        d = p[1:] - p[:-1]
        if n_air:
            d = d.clone()
            d[film - 1:] = 0.0                      # no wall term across the film's free surface
        zero = torch.zeros_like(p[:1])
        lap = lap + torch.cat([d, zero]) - torch.cat([zero, d])
        r = -f + g * lap + E[i]
        if n_air:
            r = r.clone()
            r[film:] = 0.0
        out.append(r)
    return torch.stack(out)


def _steps(case, seed, ramp=None):
    ps = _Poisson(case)
    P, phi = _initial(case, seed), None
    dt, air = case["dt"], case.get("n_air", 0)
    for s in range(case["steps"]):
        vhi = ps.vhi if ramp is None else torch.full_like(ps.vhi, W.ramp_volts(ramp[0], ramp[1], s))
        phi = ps.solve(ps.rhs(P, ps.vlo, vhi), phi)
        R = _rate(ps, P, phi, ps.vlo, vhi, COEFFS, air)
        if case.get("heun"):
            Pp = P + dt * R
            phi = ps.solve(ps.rhs(Pp, ps.vlo, vhi), phi)
            P = 0.5 * (P + Pp + dt * _rate(ps, Pp, phi, ps.vlo, vhi, COEFFS, air))
        else:
            P = P + dt * R
    return P, phi


def exact(case, seed):
    kind = case["kind"]
    if case.get("noise"):
        return None                                 # the random numbers are the library's own
    with torch.no_grad():
        if kind in ("film", "host"):
            P, phi = _steps(case, seed)
            return {"P": P, "phi": phi}
        if kind == "solve":
            ps = _Poisson(case)
            return {"phi": ps.solve(ps.rhs(_initial(case, seed), ps.vlo, ps.vhi))}
        if kind == "batch":
            outs = [_steps(dict(c, steps=case["steps"]), s, (amp, period))
                    for c, amp, period, s in _batch_films(case, seed)]
            return {"P": [o[0] for o in outs], "phi": [o[1] for o in outs]}
        if kind == "diag":
            return _diagnostics(case, seed)
    ps = _Poisson(case)
    P0 = _initial(case, seed).requires_grad_()
    coeffs = torch.tensor(COEFFS, dtype=torch.float64, device=DEV, requires_grad=True)
    vlo, vhi = ps.vlo.clone().requires_grad_(), ps.vhi.clone().requires_grad_()
    P = P0
    for _ in range(case["steps"]):
        phi = _Solve.apply(ps.rhs(P, vlo, vhi), ps)
        P = P + case["dt"] * _rate(ps, P, phi, vlo, vhi, coeffs, 0)
    target = _initial(case, seed + 1)[2] * 0.9
    g = torch.autograd.grad((P[2] - target).square().mean(), (P0, coeffs, vlo, vhi))
    return {"P": P.detach(), "dP0": g[0], "dcoeffs": g[1], "dvolt_lo": g[2], "dvolt_hi": g[3]}


def _diagnostics(case, seed):
    ps = _Poisson(case)
    P = _initial(case, seed)
    a1, a11, a12, g = COEFFS
    f32 = case["precision"] == "fp32"
    phi = 0.3 * (P[0].float() if f32 else P[0]) + 0.1 * (P[2].float() if f32 else P[2])
    phi = phi.double()
    p2 = P * P
    landau = a1 * p2.sum() + a11 * (p2 * p2).sum() + a12 * (p2[0] * p2[1] + p2[1] * p2[2] + p2[2] * p2[0]).sum()
    film = case["nz"] - case.get("n_air", 0)
    grad = sum(((torch.roll(P, -1, d) - P) ** 2).sum() for d in (2, 3)) + ((P[:, 1:film] - P[:, :film - 1]) ** 2).sum()
    zero = torch.zeros((), dtype=torch.float64, device=DEV)
    E = _rate(ps, P, phi, ps.vlo, ps.vhi, (zero, zero, zero, zero), 0)
    out = {"mean_p%s" % c: P[i].mean() for i, c in enumerate("xyz")}
    out["switched_fraction"] = (P[0] > 0.3).double().mean()
    out.update(f_landau=landau, f_grad=0.5 * g * grad, f_elec=-0.5 * (P * E).sum())
    return {k: float(v) for k, v in out.items()}
