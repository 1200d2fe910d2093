"""The work that programs have this framework do, as cases to be timed.

A case is one call (or one short sequence of calls) of the package's public
entry points on data like those the ground-state workloads produce: smooth
states of trap size with a one-percent noise, as the seeded initial data of the
rotating problems.  ``listed()`` holds the fixed cases, ``draw()`` further ones
of the same ranges.  ``exact()`` gives the same outputs by plain torch in 64
bits, with nothing of the package.
"""
import math

import numpy as np
import torch

import paper_1504_02891_gb300 as G

HALF = {1: 16.0, 2: 16.0, 3: 8.0}      # half-widths of the box by dimension


def listed():
    return [
        # One energy evaluation of the 1D benchmark problem: the smallest call, a host value comes back.
        dict(name="energy_1d_512_f64", op="energy", disc="fourier", n0=512, prec="f64", complex=False,
             beta=400.0, omega=0.0, trap="harmonic", batch=1),
        # Hessian-vector product of the rotating 512^2 problem in float64: the inner operation of the
        # second-order certificate and of float64 Newton steps.
        dict(name="hessvec_2d_512_c128", op="hessvec", disc="fourier", n0=512, n1=512, prec="f64", complex=True,
             beta=1000.0, omega=0.9, trap="harmonic", batch=1),
        # The operator roofline workload: a batch of 64 rotating 512^2 states, the largest call.
        dict(name="grad_2d_512_c64_b64", op="grad", disc="fourier", n0=512, n1=512, prec="f32", complex=True,
             beta=1000.0, omega=0.9, trap="harmonic", batch=64),
        # One feasible-gradient iteration through the entry points (gradient, Cayley step, energy) on a
        # batch of the sweep's middle grid.
        dict(name="step_2d_128_c64_b128", op="step", disc="fourier", n0=128, n1=128, prec="f32", complex=True,
             beta=500.0, omega=0.5, trap="harmonic", batch=128),
        # Gradient with energies of the 3D optical-lattice problem in float64 (sine grid, odd extents 127^3).
        dict(name="grad_3d_sine_128_f64", op="gradE", disc="sine", n0=128, n1=128, n2=128, prec="f64", complex=False,
             beta=1600.0, omega=0.0, trap="lattice", batch=1),
        # Hessian-vector product of the same problem in the bulk precision.
        dict(name="hessvec_3d_sine_128_f32", op="hessvec", disc="sine", n0=128, n1=128, n2=128, prec="f32",
             complex=False, beta=1600.0, omega=0.0, trap="lattice", batch=1),
        # Gradient of the 3D rotating problem (64^3 Fourier).
        dict(name="grad_3d_rot_64_c64", op="grad", disc="fourier", n0=64, n1=64, n2=64, prec="f32", complex=True,
             beta=200.0, omega=0.7, trap="harmonic", batch=1),
        # Finite differences on a ragged 3D grid (the accuracy study's discretisation, any number of intervals).
        dict(name="grad_3d_fd_ragged_f64", op="gradE", disc="fd", n0=150, n1=101, n2=77, prec="f64", complex=False,
             beta=200.0, omega=0.0, trap="stirrer", batch=1),
        # Cascade transfer 64^3 -> 128^3 of the 3D lattice problem in the bulk precision.
        dict(name="prolong_3d_sine_64_f32", op="prolong", disc="sine", n0=64, n1=64, n2=64, prec="f32", complex=False,
             beta=1600.0, omega=0.0, trap="lattice", batch=1),
        # Whole solve, the 2D benchmark problem: cascade 64^2 -> 128^2 -> 256^2, mixed precision.
        dict(name="solve_2d_256_mixed", op="solve", disc="fourier", n0=256, n1=256, prec="f64", complex=False,
             beta=1000.0, omega=0.0, trap="harmonic", batch=1, levels=3),
        # Whole solve in 3D: the anisotropic harmonic trap of the accuracy study on a sine grid, cascade 32^3 -> 64^3.
        dict(name="solve_3d_sine_64_mixed", op="solve", disc="sine", n0=64, n1=64, n2=64, prec="f64", complex=False,
             beta=200.0, omega=0.0, trap="anisotropic", batch=1, levels=2),
        # Many independent problems in one call: grids, couplings and slow rotations drawn like the batched sweep's.
        dict(name="sweep_2d_24", op="sweep", count=24, mix=1504),
    ]


def _pow2(rng, lo, hi):
    """A power of two between lo and hi, uniform in the exponent."""
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def draw(rng):
    op = rng.choice(["energy", "grad", "grad", "gradE", "hessvec", "hessvec", "step", "step", "prolong", "prolong",
                     "solve", "solve", "sweep"])
    if op == "sweep":
        return dict(op=op, count=rng.randint(4, 23), mix=rng.randrange(10000))
    if op == "solve":
        dim = rng.choice([1, 2, 3])
        disc = {1: "fourier", 2: "fourier", 3: "sine"}[dim]
        n = {1: _pow2(rng, 128, 512), 2: _pow2(rng, 64, 256), 3: _pow2(rng, 32, 64)}[dim]
        c = dict(op=op, disc=disc, prec="f64", complex=False, omega=0.0, batch=1, levels=rng.choice([1, 2]),
                 trap="anisotropic" if dim == 3 else "harmonic",
                 beta=round(math.exp(rng.uniform(math.log(100.0), math.log({1: 400.0, 2: 1000.0, 3: 200.0}[dim]))), 2))
        for a in range(dim):
            c["n%d" % a] = n
        return c
    dim = rng.choice([1, 2, 2, 3, 3])
    disc = rng.choice(["fourier", "fourier", "sine", "fd"])
    cplx = rng.random() < 0.5
    prec = rng.choice(["f32", "f32", "f64"])
    omega = round(rng.uniform(0.1, 0.9), 3) if cplx and dim >= 2 and disc != "sine" and rng.random() < 0.7 else 0.0
    # points of all instances together: up to the listed cases' (16.8M complex float32, 2M float64), and a
    # quarter of that for a step or a transfer, which move several times as much
    most = (1 << 24 if prec == "f32" and dim < 3 else 1 << 21) // (4 if op in ("step", "prolong") else 1)
    top = {1: 512, 2: 512, 3: 128}[dim] // (2 if op == "prolong" else 1)
    low = {1: 64, 2: 64, 3: 16}[dim] // (2 if op == "prolong" else 1)
    c = dict(op=op, disc=disc, prec=prec, complex=cplx, omega=omega,
             beta=round(math.exp(rng.uniform(math.log(50.0), math.log(1600.0))), 2),
             trap=rng.choice(["harmonic", "lattice", "stirrer"] if dim >= 2 else ["harmonic", "lattice"]))
    pts = 1
    same = rng.random() < 0.6
    first = None
    for a in range(dim):
        if disc == "fd" and op != "prolong":
            n = int(round(math.exp(rng.uniform(math.log(low), math.log(top)))))
        elif disc == "fd":
            n = rng.randint(low, top)
        else:
            n = first if same and first else _pow2(rng, low, top)
        first = first or n
        c["n%d" % a] = n
        pts *= n * (2 if op == "prolong" else 1)
    most_b = max(1, most // pts)
    c["batch"] = 1 if rng.random() < 0.4 else max(1, min(256, int(math.exp(rng.uniform(0.0, math.log(most_b + 0.5))))))
    return c


# ------------------------------------------------------------------ problems

def _dim(c):
    return sum("n%d" % a in c for a in range(3))


def _potential(kind):
    if kind == "harmonic":
        return {"kind": "harmonic", "gamma": (1.0, 1.0, 2.0)}
    if kind == "anisotropic":
        return {"kind": "harmonic", "gamma": (1.0, 2.0, 4.0)}
    if kind == "lattice":
        return {"kind": "lattice", "gamma": (1.0, 1.0, 1.0), "depth": 100.0, "k": math.pi / 4.0}
    return {"kind": "stirrer", "gamma": (1.0, 1.0, 2.0), "w0": 4.0, "delta": 1.0, "r0": 1.0}


def _params(c, refine=1):
    """The package's parameter dictionary of a case; refine = 2: the mesh of a transfer's finer side."""
    dim = _dim(c)
    half = (8.0, 6.0, 4.0) if c["trap"] == "anisotropic" else (HALF[dim],) * dim
    return dict(dim=dim, n=tuple(refine * c["n%d" % a] for a in range(dim)), lo=tuple(-h for h in half[:dim]),
                hi=half[:dim], disc=c["disc"], beta=c["beta"], omega=c["omega"], potential=_potential(c["trap"]),
                is_complex=c["complex"])


def _sweep_problems(c, seed):
    """The sweep's problems: grid of {64, 128, 256}^2 (the case's mix) on (-12, 12)^2; from the seed beta ~ U(100, 1000)
    and gamma_y ~ U(1, 1.2); every other one real without rotation, the others complex with a rotation below the first
    vortex's."""
    grids = np.random.default_rng(c["mix"]).choice([64, 128, 256], c["count"])
    rng = np.random.default_rng(seed)
    out = []
    for i, n in enumerate(int(g) for g in grids):
        beta, om, gy = float(rng.uniform(100, 1000)), float(rng.uniform(0, 0.15)), float(rng.uniform(1.0, 1.2))
        out.append(dict(dim=2, n=(n, n), lo=(-12.0, -12.0), hi=(12.0, 12.0), disc="fourier", beta=beta,
                        omega=om if i % 2 else 0.0, is_complex=bool(i % 2),
                        potential={"kind": "harmonic", "gamma": (1.0, gy, 1.0)}))
    return out


def _nodes(p, dev="cuda"):
    """Node coordinates (x, y, z), broadcast to the array shape (x last)."""
    out = []
    for a in range(p["dim"]):
        n, lo, hi = p["n"][a], p["lo"][a], p["hi"][a]
        j = torch.arange(0 if p["disc"] == "fourier" else 1, n, dtype=torch.float64, device=dev)
        shape = [1] * p["dim"]
        shape[p["dim"] - 1 - a] = len(j)
        out.append((lo + j * ((hi - lo) / n)).reshape(shape))
    return out


def _hvol(p):
    return math.prod((p["hi"][a] - p["lo"][a]) / p["n"][a] for a in range(p["dim"]))


def _shape(p):
    return tuple(p["n"][a] - (p["disc"] != "fourier") for a in reversed(range(p["dim"])))


def _V(p):
    xs, pot = _nodes(p), p["potential"]
    v = sum(0.5 * g * g * x * x for g, x in zip(pot["gamma"], xs))
    if pot["kind"] == "lattice":
        v = v + sum(pot["depth"] * torch.sin(pot["k"] * x) ** 2 for x in xs)
    elif pot["kind"] == "stirrer":
        v = v + pot["w0"] * torch.exp(-pot["delta"] * ((xs[0] - pot["r0"]) ** 2 + xs[1] ** 2))
    return v.expand(_shape(p)).contiguous()


def _unit(p, psi):
    """psi scaled to unit discrete norm, instance by instance."""
    axes = tuple(range(psi.dim() - p["dim"], psi.dim()))
    return psi / torch.sqrt(_hvol(p) * (psi.abs() ** 2).sum(axes, keepdim=True))


def _dtype(c):
    if c["complex"]:
        return torch.complex64 if c["prec"] == "f32" else torch.complex128
    return torch.float32 if c["prec"] == "f32" else torch.float64


def _states(c, p, seed):
    """States of the trap's size, one for each instance: a Gaussian (complex: with a vortex mixed in) and a noise of
    one percent, of amplitude for real data and of phase for complex data."""
    gen = torch.Generator("cuda").manual_seed(seed)
    xs, dim, nb = _nodes(p), p["dim"], c["batch"]
    s = (1.0 + 2.0 * torch.rand(nb, generator=gen, device="cuda", dtype=torch.float64)).reshape((nb,) + (1,) * dim)
    e = sum(g * x * x for g, x in zip(p["potential"]["gamma"], xs))
    real = torch.float32 if c["prec"] == "f32" else torch.float64
    env = torch.exp(-0.5 * e / s ** 2).to(real)
    xi = torch.randn((nb,) + _shape(p), generator=gen, device="cuda", dtype=real)
    if c["complex"]:
        vortex = 1.0 + torch.complex(xs[0], xs[1] if dim >= 2 else 0.5 * xs[0])
        psi = env * vortex.to(_dtype(c)) * torch.polar(torch.ones_like(xi), 0.01 * xi)
    else:
        psi = env * (1.0 + 0.01 * xi)
    psi = _unit(p, psi).to(_dtype(c)).contiguous()
    return psi if nb > 1 else psi[0].contiguous()


def _gaussian(p, width):
    xs = _nodes(p)
    psi = torch.exp(-0.5 * sum(g * x * x for g, x in zip(p["potential"]["gamma"], xs)) / width ** 2)
    return _unit(p, psi.expand(_shape(p)).contiguous())


def _guess(c, p, seed):
    """Initial guess of a solve: the trap's Gaussian, its width within a few percent of one."""
    return _gaussian(p, 1.0 + 0.05 * float(np.random.default_rng(seed).uniform(-1, 1)))


# ------------------------------------------------------------------ passes

def prepare(case, seed):
    c = case
    if c["op"] == "sweep":
        ps = _sweep_problems(c, seed)
        psi0 = [_gaussian(p, 1.0).to(torch.complex64 if p["is_complex"] else torch.float32) for p in ps]
        return dict(c=c, problems=ps, psi0=psi0, psi=[t.clone() for t in psi0])
    p = _params(c)
    prec = G.F32 if c["prec"] == "f32" else G.F64
    st = dict(c=c, plan=G.Plan(p, nbatch=c["batch"], prec=prec))
    if c["op"] == "solve":
        st["psi0"] = _guess(c, p, seed)
        st["psi"] = st["psi0"].clone()
        return st
    st["psi"] = _states(c, p, seed)
    if c["op"] == "hessvec":
        st["d"] = _states(c, p, seed + 7919)
    elif c["op"] == "prolong":
        st["fine"] = G.Plan(_params(c, 2), nbatch=c["batch"], prec=prec)
        st["out"] = st["fine"].empty()
        return st
    st["out"] = st["plan"].empty()
    if c["op"] == "step":
        st["next"] = st["plan"].empty()
    return st


def _host(v):
    """Host values of a batch as one tensor."""
    return torch.tensor(v, dtype=torch.float64) if isinstance(v, list) else v


def run(state):
    c = state["c"]
    op = c["op"]
    if op == "sweep":
        for t, t0 in zip(state["psi"], state["psi0"]):
            t.copy_(t0)
        reps = G.solve_batch(state["problems"], state["psi"], mode=1, res_tol=1e-9, max_outer=30)
        return {"psi": state["psi"], "E": torch.tensor([r["E"] for r in reps], dtype=torch.float64)}
    plan = state["plan"]
    if op == "energy":
        E, mu, norm2 = plan.energy(state["psi"])
        return {"E": _host(E), "mu": _host(mu), "norm2": _host(norm2)}
    if op == "grad":
        return {"hpsi": plan.grad(state["psi"], out=state["out"])}
    if op == "gradE":
        out, (E, mu) = plan.grad(state["psi"], out=state["out"], with_energy=True)
        return {"hpsi": out, "E": _host(E), "mu": _host(mu)}
    if op == "hessvec":
        return {"hd": plan.hessvec(state["psi"], state["d"], 0.5, out=state["out"])}
    if op == "step":
        hpsi = plan.grad(state["psi"], out=state["out"])
        out, E = plan.feasible_step(state["psi"], hpsi, 1e-2, out=state["next"], with_energy=True)
        return {"hpsi": hpsi, "psi": out, "E": _host(E)}
    if op == "prolong":
        return {"psi": plan.prolong_to(state["fine"], state["psi"], out=state["out"])}
    state["psi"].copy_(state["psi0"])
    # to a residual at which two solves agree in nine digits of the state: Eq. crit2 off, as in the accuracy study
    rep = plan.solve(state["psi"], mode=1, levels=c["levels"], res_tol=1e-10, delta_stop=1e-14)
    return {"psi": state["psi"], "E": rep["E"], "mu": rep["mu"]}


# ------------------------------------------------------------------ work

def _op_flops(p):
    """One operator application: a forward and an inverse transform of every line of every axis (5/2 n log2 n flops for
    n real values), or the stencil, and about 20 pointwise."""
    pts, per = math.prod(_shape(p)), 2 if p["is_complex"] else 1
    if p["disc"] == "fd":
        return per * pts * (5 * p["dim"] + 20)
    return per * pts * (sum(5.0 * math.log2(n) for n in p["n"]) + 20)


def work(case):
    c = case
    if c["op"] == "sweep":
        ps = _sweep_problems(c, 0)
        b = sum(math.prod(p["n"]) * (20 if p["is_complex"] else 12) for p in ps)
        return {"bytes": b, "flops": 30 * sum(_op_flops(p) for p in ps)}
    p = _params(c)
    nb = c["batch"]
    t = (4 if c["prec"] == "f32" else 8)
    v = t * (2 if c["complex"] else 1)
    pts = math.prod(_shape(p))
    reads = {"energy": 1, "grad": 1, "gradE": 1, "hessvec": 2, "step": 1, "solve": 1, "prolong": 1}[c["op"]]
    writes = {"energy": 0, "grad": 1, "gradE": 1, "hessvec": 1, "step": 2, "solve": 1}.get(c["op"])
    if c["op"] == "prolong":
        fine = math.prod(_shape(_params(c, 2)))
        return {"bytes": nb * v * (pts + fine), "flops": nb * (_op_flops(p) + _op_flops(_params(c, 2))) / 2}
    # a solve: at the least some tens of operator applications on the finest mesh
    times = {"step": 2, "solve": 30}.get(c["op"], 1)
    return {"bytes": nb * pts * v * (reads + writes) + pts * t, "flops": nb * times * _op_flops(p)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits

class _Ops:
    """The discrete operator of one problem on arrays of 64 bits, [batch] + grid."""

    def __init__(self, p):
        self.p, self.dim, self.h = p, p["dim"], _hvol(p)
        self.V, self.xs = _V(p), _nodes(p)
        self.lam, self.S = [], []
        for a in range(self.dim):
            n, L = p["n"][a], p["hi"][a] - p["lo"][a]
            if p["disc"] == "fourier":
                self.lam.append(2 * math.pi / L * torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda"))
            elif p["disc"] == "sine":
                k = torch.arange(1, n, dtype=torch.float64, device="cuda")
                self.lam.append(math.pi / L * k)
                m = torch.arange(1, n, device="cuda")
                self.S.append(math.sqrt(2.0 / n) * torch.sin(math.pi / n * ((m[:, None] * m[None, :]) % (2 * n)).double()))

    def along(self, a, v):
        """A vector over axis a (x = 0), broadcast to the array shape."""
        shape = [1] * self.dim
        shape[self.dim - 1 - a] = len(v)
        return v.reshape(shape)

    def to_modes(self, u, a, back=False):
        ax = -1 - a
        if self.p["disc"] == "fourier":
            return torch.fft.ifft(u, dim=ax) if back else torch.fft.fft(u, dim=ax)
        S = self.S[a].to(u.dtype)
        return torch.movedim(torch.movedim(u, ax, -1) @ S, -1, ax)

    def kinetic(self, u):
        p, out = self.p, 0
        for a in range(self.dim):
            if p["disc"] == "fd":
                h = (p["hi"][a] - p["lo"][a]) / p["n"][a]
                ax = u.dim() - 1 - a
                up, um = torch.zeros_like(u), torch.zeros_like(u)
                n = u.shape[ax]
                up.narrow(ax, 0, n - 1).copy_(u.narrow(ax, 1, n - 1))
                um.narrow(ax, 1, n - 1).copy_(u.narrow(ax, 0, n - 1))
                out = out + (u - 0.5 * (up + um)) / h ** 2
                if p["omega"] and a < 2:
                    # -Omega L_z = i Omega (x d_y - y d_x)
                    d = (up - um) / (2 * h)
                    out = out + 1j * p["omega"] * (-self.xs[1] * d if a == 0 else self.xs[0] * d)
                continue
            sym = self.along(a, 0.5 * self.lam[a] ** 2)
            if p["omega"] and a < 2:
                w = self.along(a, self.lam[a])
                sym = sym + (p["omega"] * self.xs[1] * w if a == 0 else -p["omega"] * self.xs[0] * w)
            k = self.to_modes(sym * self.to_modes(u, a), a, True)
            out = out + (k if p["is_complex"] else k.real)
        return out

    def lin(self, u):
        return self.kinetic(u) + self.V * u

    def H(self, u):
        return self.lin(u) + self.p["beta"] * u.abs() ** 2 * u

    def hess(self, psi, d, shift=0.0):
        r = (psi.conj() * d).real
        return self.lin(d) + self.p["beta"] * (psi.abs() ** 2 * d + 2 * r * psi) + shift * d

    def dot(self, a, b):
        axes = tuple(range(a.dim() - self.dim, a.dim()))
        return self.h * (a.conj() * b).real.sum(axes)

    def energy(self, u):
        e2, e4 = self.dot(u, self.lin(u)), self.dot(u.abs() ** 2, u.abs() ** 2)
        b = self.p["beta"]
        return e2 + 0.5 * b * e4, e2 + b * e4, self.dot(u, u)


def _prolong(pc, u):
    """Cascade transfer to the mesh of twice as many intervals on every axis, then unit norm."""
    dim = pc["dim"]
    for a in range(dim):
        ax, n = u.dim() - 1 - a, pc["n"][a]
        u = torch.movedim(u, ax, -1)
        if pc["disc"] == "fd":
            z = torch.zeros_like(u[..., :1])
            full = torch.cat([z, u, z], -1)                    # nodes 0..n
            fine = torch.zeros(u.shape[:-1] + (2 * n - 1,), dtype=u.dtype, device=u.device)
            fine[..., 1::2] = u
            fine[..., 0::2] = 0.5 * (full[..., :-1] + full[..., 1:])
            u = fine
        elif pc["disc"] == "sine":
            m, f = torch.arange(1, n, device="cuda"), torch.arange(1, 2 * n, device="cuda")
            fwd = torch.sin(math.pi / n * ((m[:, None] * m[None, :]) % (2 * n)).double()) * (2.0 / n)
            back = torch.sin(math.pi / (2 * n) * ((m[:, None] * f[None, :]) % (4 * n)).double())
            u = u @ (fwd @ back).to(u.dtype)
        else:
            w = torch.fft.fft(u, dim=-1) * 2.0
            pad = torch.zeros(u.shape[:-1] + (2 * n,), dtype=w.dtype, device=u.device)
            pad[..., : n // 2] = w[..., : n // 2]
            pad[..., 2 * n - n // 2 + 1:] = w[..., n // 2 + 1:]
            pad[..., n // 2] = 0.5 * w[..., n // 2]
            pad[..., 2 * n - n // 2] = 0.5 * w[..., n // 2]
            v = torch.fft.ifft(pad, dim=-1)
            u = v if pc["is_complex"] else v.real
        u = torch.movedim(u, -1, ax)
    return u


def _minimise(o, psi):
    """The ground state from psi: preconditioned nonlinear conjugate gradients on the unit sphere, then Newton steps
    whose systems are solved by preconditioned conjugate gradients.  psi: grid function of unit norm."""
    p = o.p
    k2 = sum(o.along(a, 0.5 * o.lam[a] ** 2) for a in range(o.dim))

    def kin_inv(u, c):
        for a in range(o.dim):
            u = o.to_modes(u, a)
        u = u / (c + k2)
        for a in range(o.dim):
            u = o.to_modes(u, a, True)
        return u if p["is_complex"] else u.real

    def tangent(u):
        u = u - o.dot(psi, u) * psi
        if p["is_complex"]:
            u = u - o.dot(1j * psi, u) * (1j * psi)
        return u

    def pre(u, mu):
        w = torch.sqrt(mu / (mu + o.V + p["beta"] * psi.abs() ** 2))
        return tangent(w * kin_inv(w * u, mu))

    d, rz = None, 1.0
    E = float(o.energy(psi)[0])
    for _ in range(2000):
        hp = o.H(psi)
        mu = float(o.dot(psi, hp))
        r = tangent(hp - mu * psi)
        if float(o.dot(r, r)) < 1e-10:
            break
        z = pre(r, mu)
        rz2 = float(o.dot(r, z))
        d = -z if d is None else tangent(-z + (rz2 / rz) * d)
        rz = rz2
        if float(o.dot(r, d)) >= 0:
            d = -z
        nd = math.sqrt(float(o.dot(d, d)))
        curv = float(o.dot(d, o.hess(psi, d, -mu)))
        th = -float(o.dot(r, d)) * nd / curv if curv > 0 else 0.1
        th = min(th, 0.5)
        for _ in range(40):
            new = math.cos(th) * psi + math.sin(th) / nd * d
            En = float(o.energy(new)[0])
            if En <= E + 1e-13 * abs(E):
                break
            th *= 0.5
        psi, E = new / math.sqrt(float(o.dot(new, new))), En
    for _ in range(12):
        hp = o.H(psi)
        mu = float(o.dot(psi, hp))
        r = tangent(mu * psi - hp)
        rr0 = math.sqrt(float(o.dot(r, r)))
        if rr0 < 2e-12:
            break
        x, q = torch.zeros_like(psi), r
        z = pre(q, mu)
        s, qz = z, float(o.dot(q, z))
        for _ in range(400):
            As = tangent(o.hess(psi, s, -mu))
            al = qz / float(o.dot(s, As))
            x, q = x + al * s, q - al * As
            if math.sqrt(float(o.dot(q, q))) < 1e-4 * rr0:
                break
            z = pre(q, mu)
            n = float(o.dot(q, z))
            s, qz = z + (n / qz) * s, n
        psi = psi + tangent(x)
        psi = psi / math.sqrt(float(o.dot(psi, psi)))
    return psi


def exact(case, seed):
    c = case
    if c["op"] == "sweep":
        psi, E = [], []
        for p in _sweep_problems(c, seed):
            o = _Ops(p)
            u = _minimise(o, _gaussian(p, 1.0).to(torch.complex128 if p["is_complex"] else torch.float64))
            # a complex state is determined up to its phase
            psi.append(None if p["is_complex"] else u)
            E.append(float(o.energy(u)[0]))
        return {"psi": psi, "E": torch.tensor(E, dtype=torch.float64)}
    p = _params(c)
    o = _Ops(p)

    def host(v):
        return v.cpu() if c["batch"] > 1 else float(v)

    if c["op"] == "solve":
        u = _minimise(o, _guess(c, p, seed))
        E, mu, _ = o.energy(u)
        return {"psi": u, "E": float(E), "mu": float(mu)}
    wide = torch.complex128 if c["complex"] else torch.float64
    psi = _states(c, p, seed).to(wide)
    if c["op"] == "energy":
        E, mu, n2 = o.energy(psi)
        return {"E": host(E), "mu": host(mu), "norm2": host(n2)}
    if c["op"] == "grad":
        return {"hpsi": o.H(psi)}
    if c["op"] == "gradE":
        E, mu, _ = o.energy(psi)
        return {"hpsi": o.H(psi), "E": host(E), "mu": host(mu)}
    if c["op"] == "hessvec":
        return {"hd": o.hess(psi, _states(c, p, seed + 7919).to(wide), 0.5)}
    if c["op"] == "prolong":
        return {"psi": _unit(_params(c, 2), _prolong(p, psi))}
    # Theorem 3.3's curve at tau, X = sqrt(h) psi and G = 2 sqrt(h) H psi, scaled to unit norm
    hp, tau = o.H(psi), 1e-2
    nX, XG, GG = o.dot(psi, psi), 2 * o.dot(psi, hp), 4 * o.dot(hp, hp)
    w = nX * (GG - XG ** 2 / nX)
    den = 1 + tau ** 2 * w
    a, b = (1 + 2 * tau * XG - tau ** 2 * w) / den, -2 * tau * nX / den

    def wide_as(v):
        return v.reshape(v.shape + (1,) * o.dim)

    y = _unit(p, wide_as(a) * psi + wide_as(b) * 2 * hp)
    return {"hpsi": hp, "psi": y, "E": host(o.energy(y)[0])}
