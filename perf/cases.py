"""The calls a user of this library has it do, as cases that can be timed and compared.

A case is one run through the public entry points: from given initial fields (or from rest), advance the handle's
medium by `steps` steps and read the fields, and the receiver traces where there are receivers.  `prepare` holds what
a program sets up once (handle, medium, sources, receivers, initial fields); `run` is what it repeats per shot.
`exact` is the same scheme in 64-bit torch operations, written without the library.
"""
import math

import numpy as np
import torch

from paper_1108_2651_gb300 import autograd, lbem, workloads

C_REF2 = {2: 0.5, 3: 1.0 / 6.0}
MU_TENSOR = (2.0, 1.0)  # the uniaxial medium's diag(mu_xx, mu_yy)
LAYER, GAMMA_MAX = 32, 0.2  # the walled box's absorbing layer
WP2, GAMMA = 0.5, 0.01  # the Drude cylinder's pole


def listed():
    return [
        # a homogeneous pulse on a small grid: the scheme's basic validation run, many short launches
        dict(name="pulse2d_128", dim=2, medium="homogeneous", storage="f32", nx=128, ny=128, nz=1, steps=500, nrec=0),
        # a snapshot loop on a small medium: a few steps, then fields, energy density and Poynting vector
        dict(name="snapshot2d_256", dim=2, medium="eps", storage="f32", nx=256, ny=256, nz=1, steps=20, nrec=0,
             flux=True),
        # the 1024^2 heterogeneous medium with a Ricker source and 64 receivers
        dict(name="het2d_1024", dim=2, medium="eps", storage="f32", nx=1024, ny=1024, nz=1, steps=1000, nrec=64),
        # a medium of a user's own size: odd width, height and step count
        dict(name="het2d_1501x1999", dim=2, medium="eps", storage="f32", nx=1501, ny=1999, nz=1, steps=333, nrec=40),
        # the 4096^2 heterogeneous medium of the benchmark
        dict(name="het2d_4096", dim=2, medium="eps", storage="f32", nx=4096, ny=4096, nz=1, steps=400, nrec=64),
        # the same in the 16-bit storage that keeps 1e-3 accuracy
        dict(name="het2d_4096_i16b", dim=2, medium="eps", storage="i16b", nx=4096, ny=4096, nz=1, steps=400, nrec=64),
        # heterogeneous permeability (the B x grad ln mu source)
        dict(name="mu2d_2048", dim=2, medium="mu", storage="f32", nx=2048, ny=2048, nz=1, steps=400, nrec=64),
        # an open domain: PEC box with an absorbing layer
        dict(name="walls2d_4096", dim=2, medium="walls", storage="f32", nx=4096, ny=4096, nz=1, steps=200, nrec=64),
        # a dispersive scatterer (lossy Drude cylinder)
        dict(name="drude2d_2048", dim=2, medium="drude", storage="f32", nx=2048, ny=2048, nz=1, steps=200, nrec=64),
        # 256 independent media of uneven sizes stepped as one batch (a training set of simulations)
        dict(name="batch2d_256", dim=2, medium="batch", storage="f32", nx=512, ny=64, nz=1, count=256, steps=400,
             nrec=8),
        # the 3D forward run
        dict(name="het3d_192", dim=3, medium="eps", storage="f32", nx=192, ny=192, nz=192, steps=100, nrec=128),
        # inversion: receiver traces of a 3D medium, their misfit and its gradient with respect to eps
        dict(name="adjoint3d_96", dim=3, medium="adjoint", storage="f32", nx=96, ny=96, nz=96, steps=40, nrec=128,
             every=10),
    ]


def draw(rng):
    """One more case of the same ranges: grids of 64^2 .. 4096^2 and 24^3 .. 192^3, every medium and storage."""
    def size(lo, hi, q=1):
        return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / q)) * q)

    kind = rng.choice(["eps", "eps", "eps", "f16", "bf16", "i16b", "mu", "walls", "drude", "aniso", "batch", "3d",
                       "3d", "adjoint"])
    nrec = rng.randint(1, 64)
    if kind == "batch":
        return dict(dim=2, medium="batch", storage="f32", nx=size(96, 512), ny=rng.randint(48, 80), nz=1,
                    count=rng.randint(8, 256), steps=rng.randint(50, 400), nrec=rng.randint(1, 8))
    if kind == "adjoint":
        n = size(24, 96)
        return dict(dim=3, medium="adjoint", storage="f32", nx=n, ny=min(96, n + rng.randint(0, 9)), nz=n,
                    steps=rng.randint(10, 40), nrec=nrec, every=rng.randint(3, 12))
    if kind == "3d":
        return dict(dim=3, medium=rng.choice(["eps", "walls"]), storage="f32", nx=size(24, 192), ny=size(24, 192),
                    nz=size(24, 192), steps=rng.randint(10, 100), nrec=nrec)
    storage = kind if kind in ("f16", "bf16", "i16b") else "f32"
    q = 4 if storage != "f32" else 1  # 16-bit states step in pairs where rows are whole groups of four sites
    nx, ny = size(80, 4096, q), size(80, 4096)
    # fewer steps on the larger grids, up to the work of the largest listed run
    most = int(min(800, 6.7e9 / (nx * ny))) if kind not in ("walls", "drude") else int(min(400, 3.3e9 / (nx * ny)))
    return dict(dim=2, medium="eps" if storage != "f32" else kind, storage=storage, nx=nx, ny=ny, nz=1,
                steps=rng.randint(20, max(21, most)), nrec=nrec)


# ------------------------------------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(shape, sigma, gen, unit=True):
    """A periodic Gaussian-smoothed uniform random field (std sigma cells), scaled to [0, 1] or to max |.| = 1."""
    u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    k2 = torch.zeros((), device="cuda")
    for ax, n in enumerate(shape):
        k = (torch.fft.rfftfreq(n, device="cuda") if ax == len(shape) - 1 else torch.fft.fftfreq(n, device="cuda"))
        k2 = k2 + (k ** 2).reshape([-1 if a == ax else 1 for a in range(len(shape))])
    s = torch.fft.irfftn(torch.fft.rfftn(u) * torch.exp(-2.0 * math.pi ** 2 * sigma ** 2 * k2), s=shape)
    if unit:
        return (s - s.min()) / (s.max() - s.min())
    s = s - s.mean()
    return s / s.abs().max()


def _grid(case):
    return (case["ny"], case["nx"]) if case["dim"] == 2 else (case["nz"], case["ny"], case["nx"])


def _medium(shape, dim, kind, gen):
    """eps_r, mu_r (or None) and the pole's wp^2 and gamma (or None), float32 on the GPU."""
    if kind == "homogeneous":
        return torch.ones(shape, device="cuda"), None, None, None
    sigma = min(20.0 if dim == 2 else 12.0, min(shape) / 8.0)
    eps = (1.0 + 2.0 * _smooth(shape, sigma, gen)) ** 2
    if kind == "mu":
        mu = 1.0 + _smooth(shape, sigma, gen)
        return eps / mu * (1.0 + 1e-6), mu, None, None
    if kind == "drude":
        ny, nx = shape
        y = torch.arange(ny, device="cuda").reshape(-1, 1)
        x = torch.arange(nx, device="cuda").reshape(1, -1)
        r = min(shape) / 8.0
        disk = ((x - 3 * nx // 4) ** 2 + (y - ny // 2) ** 2).float() <= r * r
        eps = torch.where(disk, eps.clamp(min=2.25), eps)
        return eps, None, torch.where(disk, WP2, 0.0).float(), torch.where(disk, GAMMA, 0.0).float()
    return eps, None, None, None


def _events(shape, dim, nrec, steps, gen):
    """A Ricker source at the centre and receivers at seeded sites: E_z, some of them a component of B."""
    n = int(np.prod(shape))
    centre = workloads.flat_index(shape, [k // 2 for k in shape])
    amp = workloads.ricker(steps, math.sqrt(C_REF2[dim]) / 40.0).astype(np.float32)[None, :]
    rec = torch.randint(0, n, (nrec,), generator=gen, device="cuda").cpu().numpy().astype(np.int64)
    comp = np.where(np.arange(nrec) % 4 == 3, 4, 2).astype(np.int32)
    return np.array([centre], np.int64), np.array([2], np.int32), amp, rec, comp


def _fields0(shape, dim, gen):
    """A smooth random electric field ([3][nsite], only E_z in 2D) and no magnetic one."""
    E = torch.zeros((3,) + shape, device="cuda")
    for c in ([2] if dim == 2 else range(3)):
        E[c] = _smooth(shape, min(6.0, min(shape) / 8.0), gen, unit=False)
    return E


def _batch_shapes(case):
    """Square grids of log-uniform size ny .. nx."""
    rng = np.random.Generator(np.random.PCG64(3))
    lo, hi = math.log(case["ny"]), math.log(case["nx"])
    return [(s, s) for s in (int(round(math.exp(rng.uniform(lo, hi)))) for _ in range(case["count"]))]


def _walls(case):
    """Walls on every axis (PEC) and the layer's width: up to LAYER sites, a quarter of the shortest axis."""
    layer = min(LAYER if case["dim"] == 2 else LAYER // 2, min(_grid(case)) // 4)
    return [lbem.BC_PEC] * case["dim"], layer


def _inputs(case, seed):
    """What one handle's run starts from."""
    shape, dim, gen = _grid(case), case["dim"], _generator(seed)
    d = dict(shape=shape)
    d["eps"], d["mu"], d["wp2"], d["gamma"] = _medium(shape, dim, case["medium"], gen)
    if case["medium"] != "homogeneous" and not case.get("flux"):
        d["src"], d["scomp"], d["amp"], d["rec"], d["rcomp"] = _events(shape, dim, case["nrec"], case["steps"], gen)
    if case["medium"] == "homogeneous":
        y, x = (torch.arange(n, device="cuda").float() for n in shape)
        cy, cx = (float(v) for v in (torch.rand(2, generator=gen, device="cuda") * torch.tensor(shape, device="cuda")))
        wrap = lambda v, n: (v + n / 2) % n - n / 2  # noqa: E731
        E = torch.zeros((3,) + shape, device="cuda")
        E[2] = torch.exp(-(wrap(y - cy, shape[0])[:, None] ** 2 + wrap(x - cx, shape[1])[None, :] ** 2) / 72.0)
        d["E0"] = E
    elif case["medium"] != "adjoint":
        d["E0"] = _fields0(shape, dim, gen)
    return d


def _batch_inputs(case, seed):
    out = []
    for k, shape in enumerate(_batch_shapes(case)):
        gen = _generator(seed * 1000003 + k)
        d = dict(shape=shape)
        d["eps"], _, _, _ = _medium(shape, 2, "eps", gen)
        d["src"], d["scomp"], d["amp"], d["rec"], d["rcomp"] = _events(shape, 2, case["nrec"], case["steps"], gen)
        out.append(d)
    return out


# ------------------------------------------------------------------------------------------------ the framework

def _solver(case, d, stream=None):
    s = lbem.Solver(d["shape"], storage=case["storage"], stream=stream)
    if case["medium"] == "aniso":
        lbem.lbem_set_medium_aniso(s.h, d["eps"].reshape(-1), *MU_TENSOR)
    else:
        lbem.lbem_set_medium(s.h, d["eps"].reshape(-1), None if d.get("mu") is None else d["mu"].reshape(-1))
    if d.get("wp2") is not None:
        lbem.lbem_set_dispersion(s.h, d["wp2"].reshape(-1), None, d["gamma"].reshape(-1))
    if case["medium"] == "walls":
        kind, layer = _walls(case)
        lbem.lbem_set_boundaries(s.h, kind, layer, GAMMA_MAX)
    if "src" in d:
        lbem.lbem_set_sources(s.h, d["src"], d["scomp"], d["amp"])
        lbem.lbem_set_receivers(s.h, d["rec"], d["rcomp"], case["steps"])
    return s


class _Batch:
    """The members, the batch handle (its launch shape timed once, as a program that repeats runs does; on a stream
    of its own, so that its launches are captured into a graph) and one buffer each for all members' E, B and
    traces."""

    def __init__(self, case, seed):
        inputs = _batch_inputs(case, seed)
        torch.cuda.synchronize()  # the members read the inputs on the batch's stream
        self.stream = torch.cuda.Stream()
        self.solvers = [_solver(case, d, self.stream.cuda_stream) for d in inputs]
        for s in self.solvers:
            lbem.lbem_set_fields(s.h)
        self.b = lbem.lbem_batch_create([s.h for s in self.solvers], self.stream.cuda_stream)
        lbem.lbem_batch_autotune(self.b, 100)
        self.at = np.concatenate([[0], np.cumsum([3 * s.nsite for s in self.solvers])])
        self.E = torch.empty(int(self.at[-1]), device="cuda")
        self.B = torch.empty_like(self.E)
        self.traces = torch.empty((case["count"], case["nrec"], case["steps"]), device="cuda")

    def run(self, steps):
        for s in self.solvers:
            lbem.lbem_set_fields(s.h)
        lbem.lbem_batch_step(self.b, steps)
        for k, s in enumerate(self.solvers):
            lbem.lbem_fields(s.h, self.E[self.at[k]:self.at[k + 1]], self.B[self.at[k]:self.at[k + 1]])
            lbem.lbem_traces(s.h, self.traces[k])
        torch.cuda.current_stream().wait_stream(self.stream)
        return dict(E=self.E, B=self.B, traces=self.traces)

    def __del__(self):
        if getattr(self, "b", None):
            lbem.lbem_batch_destroy(self.b)


def prepare(case, seed):
    if case["medium"] == "batch":
        return case, _Batch(case, seed), None
    d = _inputs(case, seed)
    if case["medium"] == "adjoint":
        p = workloads.Problem("adjoint", 3, d["shape"], None, None, case["steps"])
        p.src_site, p.src_comp, p.src_amp, p.rec_site, p.rec_comp = d["src"], d["scomp"], d["amp"], d["rec"], d["rcomp"]
        d["problem"] = p
        # the traces that were observed: of the same order as the run's own
        d["obs"] = 1e-3 * torch.randn((case["nrec"], case["steps"]), generator=_generator(seed + 77), device="cuda")
        return case, lbem.Solver(d["shape"]), d
    return case, _solver(case, d), d


def run(state):
    case, s, d = state
    if case["medium"] == "batch":
        return s.run(case["steps"])
    if case["medium"] == "adjoint":
        eps = d["eps"].detach().clone().requires_grad_(True)
        traces = autograd.receiver_traces(eps, s, d["problem"], checkpoint_every=case["every"])
        loss = autograd.misfit(traces, d["obs"])
        loss.backward()
        return dict(traces=traces.detach(), loss=loss.detach(), grad=eps.grad)
    lbem.lbem_set_fields(s.h, d["E0"].view(-1))
    s.step(case["steps"])
    E, B = s.fields()
    out = dict(E=E, B=B)
    if case.get("flux"):
        out["u"] = torch.empty(s.nsite, device="cuda")
        out["P"] = torch.empty(3 * s.nsite, device="cuda")
        lbem.lbem_energy_flux(s.h, out["u"], out["P"])
    if case["nrec"]:
        out["traces"] = s.traces(case["nrec"])
    return out


def work(case):
    """Each input read once, each output written once; per site and step the update's additions and products."""
    if case["medium"] == "batch":
        lo, hi = math.log(case["ny"]), math.log(case["nx"])
        mean = (math.exp(2 * hi) - math.exp(2 * lo)) / (2 * (hi - lo)) if hi > lo else case["nx"] ** 2
        n = case["count"] * mean
        return dict(bytes=n * (4 + 24) + 4.0 * case["count"] * case["steps"] * (case["nrec"] + 1),
                    flops=12.0 * n * case["steps"])
    n = float(np.prod(_grid(case)))
    t = case["steps"] * 4.0 * (case["nrec"] + 1)
    if case["medium"] == "adjoint":  # eps and the observations in, traces and gradient out; forward and reverse
        return dict(bytes=8 * n + 2 * t, flops=(70.0 + 90.0) * n * case["steps"])
    planes = {"mu": 2, "drude": 3}.get(case["medium"], 1)
    per = {"mu": 20.0, "drude": 22.0, "aniso": 16.0, "walls": 17.0}.get(case["medium"], 12.0)
    if case["dim"] == 3:
        per = 70.0 if case["medium"] != "walls" else 91.0
    out = 24 + (16 if case.get("flux") else 0)
    return dict(bytes=n * (4.0 * planes + 12 + out) + t, flops=per * n * case["steps"])


# ------------------------------------------------------------------------------------------------ in 64 bits

# D2Q5 (x, y) and D3Q7 (x, y, z) velocities
_C = {2: [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1)],
      3: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (-1, 0, 0), (0, -1, 0), (0, 0, -1)]}


def _dlog(mu, dim):
    """grad ln mu by periodic central differences, per axis x, y[, z]."""
    m = mu.log()
    return [0.5 * (torch.roll(m, -1, ax) - torch.roll(m, 1, ax)) for ax in (range(dim - 1, -1, -1))]


def _layer_factor(case, shape):
    if case["medium"] != "walls":
        return None
    _, layer = _walls(case)
    f = torch.ones(shape, dtype=torch.float64, device="cuda")
    for ax, n in enumerate(shape):
        i = torch.arange(n, device="cuda")
        i = torch.minimum(i, n - 1 - i).double()
        v = torch.where(i < layer, 1.0 - GAMMA_MAX * ((layer - i) / layer) ** 2, torch.ones_like(i))
        f = f * v.reshape([-1 if a == ax else 1 for a in range(len(shape))])
    return f


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


class _Exact:
    """The scheme with the pseudo-vector components kept per direction: g[i] is a list of the components (E_z's in 2D,
    three in 3D), at the site, before the collision.  Written out of place, so that torch can differentiate it."""

    def __init__(self, case, d):
        self.case, self.dim, self.shape = case, case["dim"], d["shape"]
        self.comps = [2] if self.dim == 2 else [0, 1, 2]
        eps = d["eps"].double()
        self.mu = None if d.get("mu") is None else d["mu"].double()
        self.r, self.mubar = 1.0, 1.0
        if case["medium"] == "aniso":
            self.r, self.mubar = math.sqrt(MU_TENSOR[0] / MU_TENSOR[1]), math.sqrt(MU_TENSOR[0] * MU_TENSOR[1])
        self.eps_mu = eps if self.mu is None else eps * self.mu
        self.cL2 = (self.dim - 1) * C_REF2[self.dim] / (self.eps_mu * self.mubar)
        self.dl = None if self.mu is None else _dlog(self.mu, self.dim)
        self.fac = _layer_factor(case, self.shape)
        self.wp2 = None if d.get("wp2") is None else d["wp2"].double()
        self.gam = None if d.get("gamma") is None else d["gamma"].double()
        if self.wp2 is not None:
            self.P = torch.zeros_like(self.cL2)
            self.J = torch.zeros_like(self.cL2)
        # the equilibrium's weights w_i / c_L^2, per direction
        r = (self.r, 1.0 / self.r, 1.0)
        self.axis_r = [None] + [r[max(range(self.dim), key=lambda a: abs(c[a]))] for c in _C[self.dim][1:]]
        self.fsum = self.r + 1.0 / self.r if self.dim == 2 else 3.0
        self.src = None
        if "src" in d:
            self.src = (torch.as_tensor(d["src"], device="cuda"), torch.as_tensor(d["amp"], device="cuda").double())
            self.rec = [(torch.as_tensor(d["rec"][d["rcomp"] == c], device="cuda"), int(c),
                         np.nonzero(d["rcomp"] == c)[0]) for c in np.unique(d["rcomp"])]
            self.nrec = len(d["rec"])
        E0 = d.get("E0")
        E = [torch.zeros_like(self.cL2) if E0 is None else E0[c].double() for c in self.comps]
        w0 = 1.0 - self.fsum * self.cL2
        self.g = [[-e * (w0 / self.cL2 if i == 0 else 0.5 * self.axis_r[i]) for e in E] for i in range(2 * self.dim + 1)]

    def moments(self):
        g, r = self.g, self.r
        if self.dim == 2:
            s = [sum(g[i][0] for i in range(5))]
            return s, [r * (g[4][0] - g[2][0]), (g[1][0] - g[3][0]) / r, torch.zeros_like(self.cL2)]
        s = [sum(g[i][c] for i in range(7)) for c in range(3)]
        B = [0.0, 0.0, 0.0]
        for i, c in enumerate(_C[3]):
            if i:
                x = _cross(g[i], c)
                B = [b + v for b, v in zip(B, x)]
        return s, B

    def E(self, s):
        E = [-self.cL2 * v for v in s]
        if self.wp2 is not None:
            E = [E[0] - self.P]
        return E

    def sample(self):
        s, B = self.moments()
        E = self.E(s)
        out = [None] * self.nrec
        for site, c, at in self.rec:
            f = (E[0] if self.dim == 2 else E[c]) if c < 3 else B[c - 3]
            v = f.reshape(-1)[site]
            for j, k in enumerate(at):
                out[k] = v[j]
        return torch.stack(out)

    def step(self, t):
        dim, g = self.dim, self.g
        s, B = self.moments()
        S = [torch.zeros_like(self.cL2) for _ in self.comps]  # Eq. 3's source over c_eff^2
        if self.dl is not None:
            S = [B[0] * self.dl[1] - B[1] * self.dl[0]] if dim == 2 else _cross(B, self.dl)
        if self.src is not None:
            site, amp = self.src
            if t < amp.shape[1]:
                m = self.mubar if self.mu is None else self.mu.reshape(-1)[site]
                c = 0 if dim == 2 else 2
                S[c] = S[c].reshape(-1).index_add(0, site, -(m * amp[:, t])).reshape(self.shape)
        lam = [self.cL2 * v for v in s]
        w0 = 1.0 - self.fsum * self.cL2
        P = 0.0
        if self.wp2 is not None:
            P, E = self.P, self.E(s)[0]
            h = 0.5 * self.gam
            self.J = ((1.0 - h) * self.J + self.wp2 * E) / (1.0 + h)
            self.P = P + self.J
        k = 1.0 if dim == 2 else 0.5  # c_eff^2 / c_L^2
        new = []
        for i, c in enumerate(_C[dim]):
            if i == 0:
                out = [2.0 * w0 * a - b - 2.0 * self.fsum * P - w0 * k * z for a, b, z in zip(s, g[0], S)]
            else:
                a = self.axis_r[i]
                if dim == 2:
                    # the opposite population: 2 g^(0) - g with g^(0) = Lambda/2 + c . (B_y, -B_x) / 2
                    o = g[{1: 3, 2: 4, 3: 1, 4: 2}[i]][0]
                    out = [a * (lam[0] + P) - o - 0.5 * a * self.cL2 * S[0]]
                else:
                    x = _cross(c, B)
                    out = [l + 0.5 * v - b - 0.5 * self.cL2 * k * z for l, v, b, z in zip(lam, x, g[i], S)]
            new.append(out if self.fac is None else [v * self.fac for v in out])
        self.g = [[self.pull(new, i, c, n) for n in range(len(self.comps))] for i, c in enumerate(_C[dim])]

    def pull(self, new, i, c, n):
        """Population i arriving at each site; across a wall the site's own opposite one times the wall's sign."""
        if i == 0:
            return new[0][n]
        a = max(range(self.dim), key=lambda k: abs(c[k]))
        ax = self.dim - 1 - a
        v = torch.roll(new[i][n], c[a], ax)
        if self.case["medium"] != "walls":
            return v
        back = new[i + self.dim if i <= self.dim else i - self.dim][n]
        sign = -1.0 if self.dim == 2 or n != a else 1.0
        at = 0 if c[a] > 0 else self.shape[ax] - 1
        v.select(ax, at).copy_(sign * back.select(ax, at))
        return v

    def fields(self):
        s, B = self.moments()
        E = self.E(s)
        zero = torch.zeros_like(self.cL2)
        return torch.stack([zero, zero, E[0]] if self.dim == 2 else E), torch.stack(B)


def _exact_run(case, d):
    x = _Exact(case, d)
    traces = []
    for t in range(case["steps"]):
        if x.src is not None:
            traces.append(x.sample())
        x.step(t)
    return x, (torch.stack(traces, 1) if traces else None)


def exact(case, seed):
    if case["medium"] == "batch":
        if case["count"] * case["steps"] > 3e4:  # thousands of small runs: a sample of members is not the whole
            return None
        runs = [_exact_run(case, d) for d in _batch_inputs(case, seed)]
        EB = [x.fields() for x, _ in runs]
        return dict(E=torch.cat([e.reshape(-1) for e, _ in EB]), B=torch.cat([b.reshape(-1) for _, b in EB]),
                    traces=torch.stack([t for _, t in runs]))
    d = _inputs(case, seed)
    if case["medium"] == "adjoint":
        obs = 1e-3 * torch.randn((case["nrec"], case["steps"]), generator=_generator(seed + 77), device="cuda")
        d["eps"] = d["eps"].double().requires_grad_(True)
        _, traces = _exact_run(case, d)
        # the misfit's cotangent is the run's own traces minus the observed ones
        loss = 0.5 * ((traces - obs.double()) ** 2).sum()
        loss.backward()
        return dict(traces=traces.detach(), loss=loss.detach(), grad=d["eps"].grad)
    with torch.no_grad():
        x, traces = _exact_run(case, d)
        E, B = x.fields()
        out = dict(E=E, B=B)
        if case.get("flux"):
            c2 = C_REF2[case["dim"]] / x.eps_mu
            out["u"] = ((B ** 2).sum(0) + (E ** 2).sum(0) / c2).reshape(-1)
            out["P"] = torch.stack(_cross(list(E), list(B))).reshape(-1)
        if traces is not None:
            out["traces"] = traces
    return out
