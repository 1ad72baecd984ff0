"""What is measured: passes of this library's solvers through its Python entry points.

A pass of a forward case advances a simulation by `steps` time steps and reads its macroscopic
fields back as device tensors, which is the loop that a program runs between two outputs; the
state goes on from pass to pass.  A pass of an adjoint case starts from its initial fields and
returns the loss and the gradient.  Every context keeps the schedule that the library gives it.

Sizes, parameters and initial fields are those of the paper's test cases and of the workloads that
this library is benchmarked and tested on.  Fields and forces are made on the GPU from the seed.
"""
import functools
import math
import random

import numpy as np
import torch

# c0^2 of D2Q37 and D3Q39 (only to turn viscosities and Mach numbers into lattice units)
CS2 = {"D2Q37": 0.6979533220196835, "D3Q39": 2.0 / 3.0}
# van der Waals a = 9/49, b = 2/21 and Carnahan-Starling a = 0.25, b = 4: T_c and the coexistence
# densities (gas, liquid) per reduced temperature, from Maxwell's rule
EOS = {"vdw": (9.0 / 49.0, 2.0 / 21.0, 4.0 / 7.0), "cs": (0.25, 4.0, 0.023582175788041854)}
COEXIST = {
    "vdw": {0.85: (1.119054875815994, 6.324991145677), 0.9: (1.490095732034194, 5.800445741994),
            0.95: (2.026552243876127, 5.116045703149)},
    "cs": {0.8: (0.021723243437775562, 0.3071956822831783), 0.85: (0.03158177953528134, 0.2792620941620207),
           0.9: (0.04542119811463903, 0.24808424109070054)},
}


def _case(name, family, nx, ny, steps, storage="f32", nz=1, **more):
    return dict(name=name, family=family, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, **more)


def listed():
    return [
        # the smallest domain, in the validation run of the start-up profile: launches and latency count
        _case("kolmogorov_64", "kolmogorov", 64, 64, 500, tau=0.8),
        # the benchmark workload (thermal decay with the Prandtl source), in 32-bit storage
        _case("thermal_1024", "thermal", 1024, 1024, 100, tau=0.7),
        # the same in 16-bit storage, as a throughput run that accepts its stated error uses it
        _case("thermal_1024_f16", "thermal", 1024, 1024, 100, storage="f16", tau=0.7),
        # a domain of odd size, whose rows start on no 16-byte boundary
        _case("thermal_ragged", "thermal", 901, 603, 100, tau=0.7),
        # the van der Waals droplet run
        _case("droplet_512", "droplet", 512, 512, 100, tau=0.8, eos="vdw", Tr=0.85, k=0.01, lag=False),
        # the Carnahan-Starling droplet at the paper's size, 16-bit storage
        _case("cs_droplet_200_f16", "droplet", 200, 200, 200, storage="f16", tau=0.8, eos="cs", Tr=0.9, k=3.02, lag=False),
        # Rayleigh-Benard convection between two walls at the paper's size, and at that of a production run
        _case("benard_200", "benard", 200, 102, 200, Pr=1.41),
        _case("benard_1024", "benard", 1024, 1026, 50, Pr=1.41),
        # the in-place step (half the memory) on a large droplet
        _case("droplet_1024_in_place", "droplet", 1024, 1024, 50, tau=0.8, eos="vdw", Tr=0.85, k=0.01, lag=True),
        # hundreds of small independent domains of uneven sizes and parameters, stepped together
        _case("batch_256", "batch", 32, 256, 100, domains=256, layout=0),
        # the 3D forward step
        _case("taylor_green_128", "taylor_green", 128, 128, 50, nz=128, tau=0.6),
        # the gradient with respect to a body-force field: forward with checkpoints, recompute, reverse
        _case("adjoint_64", "adjoint", 64, 64, 50, nz=64, tau=0.6, every=10),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of its range, odd ones and multiples of 32 among them."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, n // 32 * 32) if rng.random() < 0.35 else n


def draw(rng):
    family = rng.choice(["kolmogorov", "thermal", "thermal", "droplet", "droplet", "benard", "couette", "batch",
                         "taylor_green", "adjoint"])
    c = dict(family=family, nx=0, ny=0, nz=1, steps=0, storage=rng.choice(["f32", "f32", "f16", "bf16"]))
    work = 6e7   # node updates of a pass, about
    if family in ("kolmogorov", "thermal"):
        c.update(nx=_size(rng, 32, 2048), ny=_size(rng, 32, 2048), tau=round(rng.uniform(0.6, 1.0), 3))
    elif family == "droplet":
        eos = rng.choice(["vdw", "vdw", "cs"])
        c.update(nx=_size(rng, 64, 1024), ny=_size(rng, 64, 1024), tau=round(rng.uniform(0.75, 1.0), 3), eos=eos,
                 Tr=rng.choice(sorted(COEXIST[eos])), k=0.01 if eos == "vdw" else 3.02, lag=rng.random() < 0.4)
    elif family == "benard":
        c.update(nx=_size(rng, 64, 1024), ny=_size(rng, 52, 1026), Pr=round(rng.uniform(0.71, 1.41), 3), storage="f32")
    elif family == "couette":
        c.update(nx=_size(rng, 50, 512), ny=_size(rng, 56, 256), Pr=round(rng.uniform(0.71, 1.41), 3), storage="f32")
        work = 2e7
    elif family == "batch":
        c.update(nx=32, ny=rng.choice([128, 192, 256]), domains=rng.randrange(24, 257), layout=rng.randrange(1, 1 << 20), steps=50)
    else:
        top = 160 if family == "taylor_green" else 72
        c.update(nx=_size(rng, 24, top), ny=_size(rng, 24, top), nz=_size(rng, 24, top), tau=round(rng.uniform(0.6, 0.9), 3))
        if family == "adjoint":
            if rng.random() < 0.4:
                c.update(nx=_size(rng, 64, 512), ny=_size(rng, 64, 512), nz=1)
            c.update(every=rng.choice([1, 5, 10, 50]), storage="f32")
            work = 1e7
    if not c["steps"]:
        n = c["nx"] * c["ny"] * c["nz"]
        c["steps"] = max(10, min(400 if family != "adjoint" else 60, int(work / n)))
    return c


# ------------------------------------------------------------------------------------ the inputs
def _lattice(c):
    return "D3Q39" if c["nz"] > 1 else "D2Q37"


def _axes(*shape):
    return torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device="cuda") for n in shape), indexing="ij")


def _noise(gen, shape):
    return 2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0


def _domain(c, seed):
    """One domain: its parameters (hlbm_source_params as a dict), tau^, initial fields (float32), and its
    acceleration ("profile" [D, ny], "field" [D, ...], or None)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    nx, ny, nz, family = c["nx"], c["ny"], c["nz"], c["family"]
    turn = 2.0 * math.pi * torch.rand(3, dtype=torch.float64, device="cuda", generator=gen)   # phases
    shape = (ny, nx) if nz == 1 else (nz, ny, nx)
    D = len(shape)
    rho = torch.ones(shape, dtype=torch.float64, device="cuda")
    theta = torch.ones_like(rho)
    u = torch.zeros((D,) + shape, dtype=torch.float64, device="cuda")
    force, kind, tau = None, None, c.get("tau")
    p = dict(rho0=1.0)
    if family == "kolmogorov":
        # from rest under g_x = g0 sin(2 pi y / ny + phase), the density with noise
        y, _ = _axes(ny, nx)
        p.update(force=True, H=bool(c.get("H", False)), Pr=c.get("Pr", 1.0))
        force, kind = torch.zeros((2, ny), dtype=torch.float64, device="cuda"), "profile"
        force[0] = c.get("g0", 1e-5) * torch.sin(2 * math.pi * y[:, 0] / ny + turn[0])
        rho = rho + 1e-4 * _noise(gen, shape)
    elif family == "thermal":
        y, x = _axes(ny, nx)
        p.update(H=True, Pr=0.71)
        theta = 1.0 + 0.01 * torch.sin(2 * math.pi * x / nx + turn[0])
        rho = 1.0 / theta + 1e-6 * _noise(gen, shape)
        u[0] = 0.01 * torch.sin(2 * math.pi * y / ny + turn[1])
    elif family == "droplet":
        y, x = _axes(ny, nx)
        a, b, tc = EOS[c["eos"]]
        gas, liquid = COEXIST[c["eos"]][c["Tr"]]
        p.update(SC=True, P=True, isothermal=True, eos=c["eos"], eos_a=a, eos_b=b, eos_T=c["Tr"] * tc, k=c["k"], rho0=gas,
                 lag=c["lag"])
        x0, y0 = nx * (0.5 + 0.05 * torch.sin(turn[0])), ny * (0.5 + 0.05 * torch.sin(turn[1]))
        r = torch.sqrt((x - x0) ** 2 + (y - y0) ** 2)
        rho = 0.5 * (liquid + gas) - 0.5 * (liquid - gas) * torch.tanh(2.0 * (r - 0.22 * min(nx, ny)) / 5.0)
    elif family == "benard":
        # hot below, cold above; gravity from the Rayleigh number; a pair of weak rolls
        y, x = _axes(ny, nx)
        H, nu, hot, cold, Ra = ny - 2, 0.04, 1.4, 1.0, 1e4
        g = Ra * nu * nu * (hot + cold) / (2.0 * c["Pr"] * (hot - cold) * H ** 3)
        tau = 0.5 + nu / (CS2["D2Q37"] * 0.5 * (hot + cold))
        p.update(walls=True, wall_u=((0.0,) * 3, (0.0,) * 3), wall_theta=(hot, cold), force=True, g=(0.0, -g, 0.0), H=True,
                 Pr=c["Pr"], rho0=1.0 / cold)
        y = y - 0.5
        theta = hot - (hot - cold) * y / H + 0.004 * torch.sin(2 * math.pi * x / nx + turn[0]) * torch.sin(math.pi * y / H)
        kx, ky = 2 * math.pi / nx, math.pi / H
        u[0] = 0.01 * torch.sin(kx * x + turn[1]) * torch.cos(ky * y)
        u[1] = -0.01 * (kx * H / math.pi) * torch.cos(kx * x + turn[1]) * torch.sin(ky * y)
        rho = 1.0 / theta
    elif family == "couette":
        # thermal Couette flow: the upper wall moves, a linear profile with a disturbance
        y, x = _axes(ny, nx)
        H, nu, top, Ec = ny - 2, 0.01, 0.8, 10.0
        u0 = 100.0 * nu / H
        dth = u0 * u0 / (2.0 * CS2["D2Q37"] * Ec)
        tau = 0.5 + nu / CS2["D2Q37"]
        p.update(walls=True, wall_u=((0.0,) * 3, (u0, 0.0, 0.0)), wall_theta=(top - dth, top), H=True, Pr=c["Pr"])
        s = (y - 0.5) / H
        theta = top - dth * (1.0 - s) + 1e-3 * torch.sin(2 * math.pi * x / nx + turn[0]) * torch.sin(math.pi * s)
        u[0] = u0 * s
        rho = top / theta
    else:   # Taylor-Green vortex, Ma 0.3 (in 2D one of its planes); the adjoint's force is a weak smooth field
        lat = _lattice(c)
        U = 0.3 * math.sqrt(CS2[lat] * (D + 2.0) / D)
        if D == 3:
            z, y, x = (2 * math.pi * q / n + t for q, n, t in zip(_axes(nz, ny, nx), shape, turn))
            u[0], u[1] = U * torch.sin(x) * torch.cos(y) * torch.cos(z), -U * torch.cos(x) * torch.sin(y) * torch.cos(z)
            rho = 1.0 + U * U / (16.0 * CS2[lat]) * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)
        else:
            y, x = (2 * math.pi * q / n + t for q, n, t in zip(_axes(ny, nx), shape, turn))
            u[0], u[1] = U * torch.sin(x) * torch.cos(y), -U * torch.cos(x) * torch.sin(y)
            rho = 1.0 + U * U / (4.0 * CS2[lat]) * (torch.cos(2 * x) + torch.cos(2 * y))
        p.update(force=True)
        force, kind = torch.zeros((D,) + shape, dtype=torch.float64, device="cuda"), "field"
        force[0] = 1e-4 * torch.sin(y)
        force[D - 1] += 5e-5 * torch.cos(x)
    f32 = [t.to(torch.float32).contiguous() for t in (rho, u, theta)]
    return p, tau, f32, None if force is None else force.to(torch.float32).contiguous(), kind


def _members(c):
    """The domains of a batch: Kolmogorov flow with the Prandtl source and droplets in turn, of uneven sides,
    relaxation times, forces and temperatures.  Their sizes and parameters belong to the case, not to the seed."""
    r = random.Random(c["layout"])
    out = []
    for i in range(c["domains"]):
        n = r.randint(c["nx"], c["ny"])
        m = dict(nx=n, ny=n, nz=1, steps=c["steps"], storage=c["storage"])
        if i % 2 == 0:
            m.update(family="kolmogorov", tau=r.uniform(0.55, 1.2), g0=10.0 ** r.uniform(-6.0, -4.0), H=True, Pr=r.uniform(0.71, 1.41))
        else:
            m.update(family="droplet", tau=r.uniform(0.75, 1.2), eos="vdw", Tr=r.choice([0.85, 0.9, 0.95]), k=0.01, lag=False)
        out.append(m)
    return out


# ---------------------------------------------------------------------------------- the passes
def _solver(c, seed):
    from paper_2411_10751_gb300.solver import HLBM
    p, tau, fields, force, kind = _domain(c, seed)
    s = HLBM(_lattice(c), c["nx"], c["ny"], c["nz"], tau, p, storage=c["storage"])
    return s, fields, force, kind


def prepare(case, seed):
    if case["family"] == "batch":
        from paper_2411_10751_gb300.solver import Batch
        solvers = []
        for i, m in enumerate(_members(case)):
            s, fields, force, kind = _solver(m, seed * 1009 + i)
            s.init(*fields)
            if force is not None:
                s.set_force_field(force, kind)
            solvers.append(s)
        return dict(case=case, solvers=solvers, batch=Batch(solvers))
    s, fields, force, kind = _solver(case, seed)
    if case["family"] == "adjoint":
        return dict(case=case, solver=s, fields=fields, g=force.requires_grad_())
    s.init(*fields)
    if force is not None:
        s.set_force_field(force, kind)
    return dict(case=case, solver=s)


def run(state):
    c = state["case"]
    if c["family"] == "adjoint":
        from paper_2411_10751_gb300.solver import KineticEnergy
        g = state["g"]
        loss = KineticEnergy.apply(g, state["solver"], *state["fields"], c["steps"], c["every"])
        grad, = torch.autograd.grad(loss, g)
        return {"loss": loss.detach(), "grad": grad}
    if c["family"] == "batch":
        state["batch"].step(c["steps"])
        fields = [s.moments() for s in state["solvers"]]
        return {k: torch.cat([f[i].reshape(-1) for f in fields]) for i, k in enumerate(("rho", "u", "theta"))}
    s = state["solver"]
    s.step(c["steps"])
    rho, u, theta = s.moments()
    return {"rho": rho, "u": u, "theta": theta}


def _nodes(c):
    return sum(m["nx"] * m["ny"] for m in _members(c)) if c["family"] == "batch" else c["nx"] * c["ny"] * c["nz"]


def work(case):
    """A step reads and writes every population once (the in-place step a neighbour field too, the wall-bounded
    step its previous moments); the readout reads them and writes the fields.  The adjoint's forward steps are taken
    once, and a reverse step reads lambda, the forward state and g, writes lambda and adds to dL/dg.  Operations per
    node and step: about 12 per velocity for the moments and the collision."""
    n, D = _nodes(case), 3 if case["nz"] > 1 else 2
    q = 39 if D == 3 else 37
    elem = 4 if case["storage"] == "f32" else 2
    step = 2 * q * elem
    if case["family"] == "droplet" and case["lag"]:
        step += 8
    if case["family"] in ("benard", "couette"):
        step += 32
    if case["family"] == "adjoint":
        per = (step + 4 * D) + (2 * q * 4 + q * elem + 12 * D)
        return {"bytes": float(n) * case["steps"] * per, "flops": float(n) * case["steps"] * 30 * q}
    return {"bytes": float(n) * (case["steps"] * step + q * elem + 4 * (D + 2)), "flops": float(n) * (case["steps"] + 1) * 12 * q}


# ------------------------------------------------------------- the same in 64 bits, by plain torch
@functools.lru_cache(None)
def _quadrature(lat):
    """(c [Q, D], w [Q], c0^2).  D2Q37: the nine even moment conditions up to degree 8 on the velocity shells
    |c|^2 in {0, 1, 2, 4, 5, 8, 9, 10} give the eight weights and c0^2."""
    if lat == "D3Q39":
        groups = [((0, 0, 0), 1 / 12), ((1, 0, 0), 1 / 12), ((1, 1, 1), 1 / 27), ((2, 0, 0), 2 / 135), ((2, 2, 0), 1 / 432),
                  ((3, 0, 0), 1 / 1620)]
        cs2 = 2.0 / 3.0
    else:
        reps = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 1)]
        odd = {0: 1, 2: 1, 4: 3, 6: 15, 8: 105}
        conds = [(0, 0), (2, 0), (4, 0), (2, 2), (6, 0), (4, 2), (6, 2), (4, 4), (8, 0)]
        rows = np.array([[sum(c[0] ** p * c[1] ** q for c in _orbit(r)) for r in reps] for p, q in conds], dtype=np.float64)

        def solve(cs2):
            rhs = np.array([odd[p] * odd[q] * cs2 ** ((p + q) // 2) for p, q in conds])
            w = np.linalg.solve(rows[:8], rhs[:8])
            return w, float(rows[8] @ w - rhs[8])

        lo, hi = 0.69, 0.71   # the root with all weights positive
        assert solve(lo)[1] * solve(hi)[1] < 0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (lo, mid) if solve(lo)[1] * solve(mid)[1] <= 0 else (mid, hi)
        cs2 = 0.5 * (lo + hi)
        groups = list(zip(reps, solve(cs2)[0]))
    c = [v for r, _ in groups for v in _orbit(r)]
    w = [x for r, x in groups for _ in _orbit(r)]
    return np.array(c, dtype=np.int64), np.array(w, dtype=np.float64), cs2


def _orbit(rep):
    """Every vector that permutations and signs make of `rep`."""
    import itertools
    return sorted({tuple(s * v for s, v in zip(sign, perm)) for perm in itertools.permutations(rep)
                   for sign in itertools.product((1, -1), repeat=len(rep))})


class _Exact:
    """The scheme in 64 bits: f_i(x, t), Hermite coefficients per monomial order, streaming by index."""

    def __init__(self, c, p, tau, force, kind):
        self.p, self.tau = p, tau
        self.shape = (c["ny"], c["nx"]) if c["nz"] == 1 else (c["nz"], c["ny"], c["nx"])
        D = self.D = len(self.shape)
        cv, w, self.cs2 = _quadrature(_lattice(c))
        self.Q, self.N, self.order = len(w), int(np.prod(self.shape)), 4 if D == 2 else 3
        dev = dict(dtype=torch.float64, device="cuda")
        self.cv = cv
        self.w = torch.tensor(w, **dev)
        cf = torch.tensor(cv, **dev)
        self.moment = torch.stack([torch.ones(self.Q, **dev)] + [cf[:, d] for d in range(D)] + [(cf * cf).sum(1)])
        xi = cf / math.sqrt(self.cs2)
        he = [torch.ones_like(xi), xi, xi ** 2 - 1, xi ** 3 - 3 * xi, xi ** 4 - 6 * xi ** 2 + 3]
        self.index = [i for i in np.ndindex(*(self.order + 1,) * D) if sum(i) <= self.order]
        cols = []
        for i in self.index:   # He_i(xi) / i!
            col = torch.ones(self.Q, **dev)
            for d in range(D):
                col = col * he[i[d]][:, d] / math.factorial(i[d])
            cols.append(col)
        self.poly = torch.stack(cols, 1)                       # [Q, monomials]
        self.basis = self.w[:, None] * self.poly
        grid = np.indices(self.shape).reshape(D, -1)           # slowest axis first
        self.grid = grid
        src = []
        for v in cv:   # x - c_i, the velocity's components in x, y (, z) order
            at = [(grid[d] - v[D - 1 - d]) % self.shape[d] for d in range(D)]
            src.append(np.ravel_multi_index(at, self.shape))
        self.src = torch.tensor(np.array(src), device="cuda")
        self.g = None
        if p.get("force"):
            if force is None:
                self.g = torch.tensor(list(p.get("g", (0.0,) * 3))[:D], **dev)[:, None].expand(D, self.N).contiguous()
            elif kind == "profile":
                self.g = force.double()[:, :, None].expand(2, *self.shape).reshape(2, -1)
            else:
                self.g = force.double().reshape(D, -1)

    def shift(self, a, *by):
        """a at x + by (components in x, y (, z) order)."""
        v = a.reshape(self.shape)
        return torch.roll(v, [-b for b in reversed(by)], dims=list(range(self.D))).reshape(-1)

    def products(self, u, tb):
        """m_i = prod_d m_{i_d}(u_d / c0) of every Hermite index, m_k the Gaussian moments of variance 1 + tb."""
        one, c0 = [], math.sqrt(self.cs2)
        for d in range(self.D):
            x = u[d] / c0
            one.append([torch.ones_like(x), x, x * x + tb, x ** 3 + 3 * x * tb, x ** 4 + 6 * x * x * tb + 3 * tb * tb])
        m = {}
        for i in self.index:
            v = one[0][i[0]]
            for d in range(1, self.D):
                v = v * one[d][i[d]]
            m[i] = v
        return m

    def equilibrium(self, rho, u, theta):
        m = self.products(u, theta - 1)
        return self.basis @ torch.stack([rho * m[i] for i in self.index])

    def psi(self, rho):
        p = self.p
        e = p["eos_b"] * rho if p["eos"] == "vdw" else 0.25 * p["eos_b"] * rho
        z = 1 / (1 - e) if p["eos"] == "vdw" else (1 + e + e * e - e ** 3) / (1 - e) ** 3
        pressure = rho * p["eos_T"] * z - p["eos_a"] * rho * rho
        return torch.sqrt(torch.clamp(2 * rho - 2 * pressure / self.cs2, min=0))

    def macro(self, f, psi=None):
        """rho, u, theta, F, sigma of populations f; psi: the pseudopotential to use (None: that of f's density)."""
        D = self.D
        m = self.moment @ f
        rho = m[0]
        F = rho * self.g if self.g is not None else torch.zeros_like(m[1:1 + D])
        sigma = torch.zeros_like(rho)
        if self.p.get("SC"):
            psi = self.psi(rho) if psi is None else psi
            fs = torch.zeros_like(F)
            for v, w in zip(self.cv, self.w):
                if any(v):
                    t = w * self.shift(psi, *v)
                    for d in range(D):
                        if v[d]:
                            fs[d] += float(v[d]) * t
            fs = psi * fs
            F = F + fs
            if self.p.get("P"):
                coef = self.p["k"] * self.cs2 / (D * (self.tau - 0.5))
                sigma = torch.where(psi > 0, coef * (fs * fs).sum(0) / torch.clamp(psi * psi, min=1e-300), sigma)
        u = (m[1:1 + D] + 0.5 * F) / rho
        G2 = 2 * (u * F).sum(0) + D * self.cs2 * sigma
        theta = (m[1 + D] - rho * (u * u).sum(0) + 0.5 * G2) / (rho * D * self.cs2)
        return rho, u, theta, F, sigma

    def grad_theta(self, theta):
        gx = 0.5 * (self.shift(theta, 1, 0) - self.shift(theta, -1, 0))
        gy = 0.5 * (self.shift(theta, 0, 1) - self.shift(theta, 0, -1))
        if self.p.get("walls"):
            t, g = theta.reshape(self.shape), gy.reshape(self.shape)
            g[0] = 0.5 * (-3 * t[0] + 4 * t[1] - t[2])
            g[-1] = -0.5 * (-3 * t[-1] + 4 * t[-2] - t[-3])
        return gx, gy

    def collide(self, f, fields):
        rho, u, theta, F, sigma = fields
        omega, beta, c0, D = 1 / self.tau, 1 - 0.5 / self.tau, math.sqrt(self.cs2), self.D
        tb = torch.zeros_like(rho) if self.p.get("isothermal") else theta - 1
        m = self.products(u, tb)
        B = {i: omega * rho * m[i] for i in self.index}
        for i in self.index:   # body force: orders 1 to 3
            if 1 <= sum(i) <= 3:
                for d in range(D):
                    if i[d]:
                        low = tuple(i[e] - (e == d) for e in range(D))
                        B[i] = B[i] + beta * F[d] / c0 * i[d] * m[low]
        if D == 2:
            if self.p.get("P"):
                B[2, 0], B[0, 2] = B[2, 0] + beta * sigma, B[0, 2] + beta * sigma
            if self.p.get("H"):
                gx, gy = self.grad_theta(theta)
                h = beta * rho * theta * (1 - 1 / self.p["Pr"]) * c0
                B[3, 0], B[1, 2] = B[3, 0] + 3 * h * gx, B[1, 2] + h * gx
                B[0, 3], B[2, 1] = B[0, 3] + 3 * h * gy, B[2, 1] + h * gy
        return (1 - omega) * f + self.basis @ torch.stack([B[i] for i in self.index])

    def stream(self, f):
        return torch.gather(f, 1, self.src)

    # walls: the populations after streaming from the post-collision state S and the previous moments
    def wall_stream(self, S, prev):
        ny, nx = self.shape
        f = self.stream(S).reshape(self.Q, ny, nx)
        S = S.reshape(self.Q, ny, nx)
        opp = [int(np.where((self.cv == -v).all(1))[0][0]) for v in self.cv]
        rho_p, u_p, th_p = prev[0].reshape(ny, nx), prev[1].reshape(2, ny, nx), prev[2].reshape(ny, nx)
        for side in (0, 1):
            uw = torch.tensor(self.p["wall_u"][side][:2], dtype=torch.float64, device="cuda")[:, None]
            tw = float(self.p["wall_theta"][side])
            first = 1 if side == 0 else ny - 2
            for r in range(3):
                y = r if side == 0 else ny - 1 - r
                unknown = [i for i, v in enumerate(self.cv) if not 0 <= y - v[1] < ny]
                mp = self.products(u_p[:, y], th_p[y] - 1)
                Pp = self.poly @ torch.stack([mp[i] for i in self.index])       # [Q, nx]
                target = {}
                for a in sorted({abs(int(self.cv[i][1])) for i in unknown}):
                    k = 2.0 * (0.5 - (r - a / 2.0))                             # from the interface outwards, per half cell
                    ut, tt = uw + k * (uw - u_p[:, first]), tw + k * (tw - th_p[first])
                    mt = self.products(ut, tt - 1)
                    target[a] = self.poly @ torch.stack([mt[i] for i in self.index])
                out = sum(self.w[i] * Pp[opp[i]] for i in unknown)
                back = sum(self.w[i] * target[abs(int(self.cv[i][1]))][i] for i in unknown)
                for i in unknown:
                    f[i, y] = S[opp[i], y] + self.w[i] * rho_p[y] * (
                        out / back * target[abs(int(self.cv[i][1]))][i] - Pp[opp[i]])
        return f.reshape(self.Q, -1)


def _exact_forward(c, seed):
    p, tau, (rho, u, theta), force, kind = _domain(c, seed)
    E = _Exact(c, p, tau, force, kind)
    rho, u, theta = rho.double().reshape(-1), u.double().reshape(E.D, -1), theta.double().reshape(-1)
    f = E.equilibrium(rho, u, theta)
    walls, lag = p.get("walls"), p.get("lag")
    psi = E.psi(rho) if lag else None
    if walls:   # the state before the first streaming, periodic in y
        S, prev = torch.empty_like(f).scatter_(1, E.src, f), (rho, u, theta)
        f = E.wall_stream(S, prev)
    for _ in range(c["steps"]):
        m = E.macro(f, psi)
        S = E.collide(f, m)
        if lag and p.get("SC"):
            psi = E.psi(m[0])
        f = E.wall_stream(S, m[:3]) if walls else E.stream(S)
    rho, u, theta = E.macro(f, psi)[:3]
    return rho.reshape(E.shape), u.reshape(E.D, *E.shape), theta.reshape(E.shape)


def exact(case, seed):
    c = case
    if c["family"] == "batch":
        fields = [_exact_forward(m, seed * 1009 + i) for i, m in enumerate(_members(c))]
        return {k: torch.cat([f[i].reshape(-1) for f in fields]) for i, k in enumerate(("rho", "u", "theta"))}
    if c["family"] == "adjoint":
        p, tau, (rho, u, theta), force, kind = _domain(c, seed)
        E = _Exact(c, p, tau, force, kind)
        g = E.g = E.g.clone().requires_grad_()
        f = E.equilibrium(rho.double().reshape(-1), u.double().reshape(E.D, -1), theta.double().reshape(-1))
        for _ in range(c["steps"]):
            f = E.stream(E.collide(f, E.macro(f)))
        r, v = E.macro(f)[:2]
        loss = 0.5 * (r * (v * v).sum(0)).sum()
        grad, = torch.autograd.grad(loss, g)
        return {"loss": loss.detach(), "grad": grad.reshape(E.D, *E.shape)}
    rho, u, theta = _exact_forward(c, seed)
    return {"rho": rho, "u": u, "theta": theta}
