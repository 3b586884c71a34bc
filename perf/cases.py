"""What a user of the library has it do, as timed cases.

Each case is one call pattern of a user's program, through the public binding:

* ``step``: a handle that was set up once integrates a chunk of steps (RK4) or
  attempts (Dormand-Prince), then the cavity amplitudes and the magnetisation
  of every instance are read out into tensors that the program keeps;
* ``map``: several handles of mixed grids stepped together as one group;
* ``field``: one evaluation of the effective field of the current state;
* ``gradient``: an objective and its backward pass through the autograd wrapper.

``exact`` gives the same results in 64 bits, from plain torch: the Newell
tensor, the zero-padded convolution with torch.fft, the local fields, the
Runge-Kutta steps with the cavity equations, and autograd for the gradients.
"""
import math
import random

import torch

import paper_2410_00966_gb300 as pkg

GAMMA, MU0, HBAR = 1.7595e11, 4e-7 * math.pi, 1.05457182e-34
TWOPI = 2.0 * math.pi
MATERIALS = {
    # Ms (A/m), Aex (J/m), alpha, Ku (J/m^3), cell (m)
    "permalloy": dict(Ms=8e5, Aex=1.3e-11, alpha=0.01, Ku=0.0, d=4e-9),
    "yig": dict(Ms=1.4e5, Aex=3.65e-12, alpha=1e-4, Ku=1e3, d=5e-9),
    "vortex": dict(Ms=8e5, Aex=1.3e-11, alpha=0.02, Ku=0.0, d=2e-9),
}
DT_RK4 = 5e-14        # the fixed step of the anticrossing map and of the gradient runs
DT_FIRST = 2e-15      # first Dormand-Prince trial step, careful: the controller grows it by 5 at a time


def _step(name, nx, ny, nz, batch, steps, *, material="permalloy", kind="rk4", cavity="E", modes=1, profile="uniform",
          mask="full", drive=False, tuned=False):
    return dict(name=name, what="step", nx=nx, ny=ny, nz=nz, batch=batch, steps=steps, material=material, kind=kind,
                cavity=cavity, modes=modes, profile=profile, mask=mask, drive=drive, tuned=tuned)


def listed():
    return [
        # the smallest call: the field of a small film, looked at once
        dict(name="field of a film", what="field", nx=32, ny=32, nz=1, material="permalloy"),
        # the small film at a fixed step, read out every 50 steps: launches and latency are all there is
        _step("film ring-down", 32, 32, 1, 1, 50),
        # a bias sweep of a thin film of no particular size, one launch for all its values
        _step("film bias sweep", 100, 75, 1, 16, 20),
        # an extended thin film, driven by a sinc pulse and recorded, for its broadband response
        _step("wide film spectroscopy", 1000, 600, 1, 1, 4, drive=True),
        # a strip over a coplanar waveguide: coupling falls off across it; adaptive steps
        _step("strip on a waveguide", 300, 120, 5, 1, 3, kind="dp45", profile="lorentzian"),
        # a YIG sphere with two cavity modes and the memory sums as the paper writes them
        _step("sphere, two modes", 50, 50, 50, 1, 5, material="yig", cavity="P", modes=2, mask="ellipsoid"),
        # the YIG wire, omega_c swept through its uniform mode in 21 values, tuned once by the program
        _step("wire sweep", 256, 64, 16, 21, 2, material="yig", kind="dp45", tuned=True),
        # the largest grid: a film over a waveguide, 8.4 million cells, adaptive steps, tuned once
        _step("large film on a waveguide", 1024, 1024, 8, 1, 2, kind="dp45", profile="lorentzian", tuned=True),
        # an anticrossing map: 64 instances of four grid sizes in one captured group
        dict(name="anticrossing map", what="map", n=32, instances=64, steps=16, material="permalloy"),
        # gradients of the photon number of a vortex disk with respect to its parameters and its Ms map
        dict(name="vortex disk gradient", what="gradient", nx=128, ny=128, nz=4, steps=16, ckpt=8, material="vortex"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(("step", "step", "step", "step", "map", "field", "gradient"))
    if what == "map":
        case = dict(what="map", n=size(16, 32), instances=size(8, 64), steps=16, material="permalloy")
        while work(case)["flops"] > 3.3e11:
            case["steps"] -= 3
        return case
    if what == "gradient":
        return dict(what="gradient", nx=size(32, 128), ny=size(32, 128), nz=rng.choice((1, 2, 3, 4)),
                    steps=rng.choice((8, 12, 16)), ckpt=rng.choice((4, 8)), material="vortex")
    family = rng.choice(("film", "slab", "block"))
    if family == "film":
        nx, ny, nz = size(16, 1024), size(16, 1024), 1
    elif family == "slab":
        nx, ny, nz = size(24, 1024), size(24, 1024), rng.randint(2, 8)
    else:
        nx, ny, nz = size(16, 256), size(16, 128), size(9, 64)
    cells = nx * ny * nz
    material = rng.choice(("permalloy", "yig"))
    if what == "field":
        return dict(what="field", nx=nx, ny=ny, nz=nz, material=material)
    kind = rng.choice(("rk4", "dp45"))
    batch = max(1, min(size(1, 21), 4_000_000 // cells))
    steps = max(2, min(40, 8_000_000 // (cells * batch))) if kind == "rk4" else 2
    case = dict(what="step", nx=nx, ny=ny, nz=nz, batch=batch, steps=steps, material=material, kind=kind,
                cavity=rng.choice(("E", "E", "P")), modes=rng.choice((1, 1, 1, 2)),
                profile=rng.choice(("uniform", "lorentzian")), mask=rng.choice(("full", "full", "ellipsoid")),
                drive=rng.random() < 0.25, tuned=rng.random() < 0.3)
    while case["batch"] > 1 and work(case)["flops"] > 1.5e11:     # padding can cost eight times the cells
        case["batch"] = (case["batch"] + 1) // 2
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _centres(nx, ny, nz):
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5 - nx / 2)[None, None, :]
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5 - ny / 2)[None, :, None]
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5 - nz / 2)[:, None, None]
    return x, y, z


def _tilted(batch, cells, g):
    """Magnetisation turned away from x by a pulse (0.1 to 0.3 rad), with a random tilt of each cell; (batch, cells, 3)."""
    turn = 0.1 + 0.2 * torch.rand(batch, 2, generator=g, device="cuda")
    m = 0.05 * (2.0 * torch.rand(batch, cells, 3, generator=g, device="cuda") - 1.0)
    m[..., 0] += 1.0
    m[..., 1] += turn[:, None, 0]
    m[..., 2] += 0.5 * turn[:, None, 1]
    return m / m.norm(dim=-1, keepdim=True)


def _ms_map(case, Ms, g):
    """Ms of each cell (float32): the whole grid, or the ellipsoid inscribed in it."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case.get("mask", "full") == "full":
        return torch.full((nx * ny * nz,), Ms, device="cuda", dtype=torch.float32)
    x, y, z = _centres(nx, ny, nz)
    inside = (2 * x / nx) ** 2 + (2 * y / ny) ** 2 + (2 * z / nz) ** 2 <= 1.0
    return torch.where(inside, Ms, 0.0).to(torch.float32).reshape(-1).contiguous()


def _profile(case):
    """Coupling shape of each cell along y (float32 numpy), or None for a uniform one."""
    if case.get("profile", "uniform") == "uniform":
        return None
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x, _, _ = _centres(nx, ny, nz)
    p = torch.zeros(nz, ny, nx, 3, device="cuda", dtype=torch.float32)
    p[..., 1] = (1.0 / (1.0 + (x / max(4.0, nx / 8)) ** 2)).float()
    return p.reshape(-1, 3).cpu().numpy()


def _instances(case, batch, seed):
    """Bias and cavity of each instance: a sweep of omega_c or of the bias around seeded values."""
    r = random.Random(int(seed) * 31 + 5)
    b0, f0 = r.uniform(0.05, 0.1), r.uniform(5e9, 8e9)
    return [dict(bias=(b0 * (1.0 + 0.02 * b), 0.0, 0.0), omega=TWOPI * f0 * (1.0 + 0.01 * b), kappa=TWOPI * 10e6,
                 g=TWOPI * 100e6) for b in range(batch)]


def _map_grids(case):
    """The grids of a map and how many instances each has (the same for every seed)."""
    n, r = case["n"], random.Random(case["instances"])
    grids = [(n, n, 1), (2 * n, 2 * n, 2), (4 * n, 4 * n, 2), (8 * n, 8 * n, 4)]
    count = [0, 0, 0, 0]
    for _ in range(case["instances"]):
        count[r.randrange(4)] += 1
    return [(g, c) for g, c in zip(grids, count) if c]


def _inputs(case, seed):
    """Everything the calls of a step or field case are given, as plain tensors and numbers."""
    mat = MATERIALS[case["material"]]
    batch, cells = case.get("batch", 1), case["nx"] * case["ny"] * case["nz"]
    g = _gen(seed)
    ms = _ms_map(case, mat["Ms"], g)
    m0 = _tilted(batch, cells, g) * (ms > 0)[None, :, None]
    return dict(mat=mat, ms=ms, m0=m0.contiguous(), profile=_profile(case), inst=_instances(case, batch, seed))


def _handle(case, x):
    """A configured handle: material, state, bias and cavity modes of every instance."""
    mat, batch = x["mat"], case.get("batch", 1)
    sim = pkg.Sim(case["nx"], case["ny"], case["nz"], mat["d"], mat["d"], mat["d"], mat["Ms"], mat["Aex"],
                  mat["alpha"], Ku=mat["Ku"], batch=batch)
    torch.cuda.synchronize()
    if case.get("mask", "full") != "full":
        sim.set_ms_map(x["ms"])
    for b, q in enumerate(x["inst"]):
        sim.set_m(x["m0"][b], inst=b)
        sim.set_bias(q["bias"], inst=b)
    for k in range(case.get("modes", 1)):
        if x["profile"] is not None:
            q = x["inst"][0]
            sim.set_cavity_mode(k, q["omega"], q["kappa"], q["g"], profile=x["profile"])
        for b, q in enumerate(x["inst"]):
            sim.set_cavity_mode(k, q["omega"] * (1.0 + 0.2 * k), q["kappa"], q["g"], inst=b)
    sim.set_cavity_init(2.0, 0.0)
    if case.get("drive"):
        sim.set_drive(1e3, TWOPI * 20e9, 1e-12)
        sim.set_recording(1)
    dp = case.get("kind") == "dp45"
    sim.set_integrator(pkg.MMCQ_DP45 if dp else pkg.MMCQ_RK4, 1e-6,
                       pkg.MMCQ_CAVITY_P if case.get("cavity") == "P" else pkg.MMCQ_CAVITY_E)
    if case.get("tuned"):
        sim.autotune()
    return sim


def _vortex(case, seed):
    """A displaced vortex in a disk with a random Ms map, and the parameters as a differentiable program holds them."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    mat, g = MATERIALS["vortex"], _gen(seed)
    r = random.Random(int(seed))
    x, y, _ = _centres(nx, ny, nz)
    x, y = x.expand(nz, ny, nx), y.expand(nz, ny, nx)
    rad = 0.39 * min(nx, ny)
    ms = 7.5e5 + 1e5 * torch.rand(nz, ny, nx, generator=g, device="cuda", dtype=torch.float64)
    ms = torch.where(x * x + y * y <= max(rad, 4.0) ** 2, ms, 0.0)
    cx, cy, chir = r.uniform(0.2, 0.4) * rad, r.uniform(0.2, 0.4) * rad, r.choice((-1.0, 1.0))
    rr = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2) + 1e-3
    mz = torch.exp(-((rr / 5.0) ** 2))
    ip = torch.sqrt(1.0 - mz * mz)
    m = torch.stack([-chir * ip * (y - cy) / rr, chir * ip * (x - cx) / rr, mz], -1)
    m = (m * (ms > 0)[..., None]).reshape(1, -1, 3).float().cpu().numpy()
    p = torch.tensor([[0.005, 0.002, 0.0, TWOPI * 200e6, TWOPI * 1.3e9, TWOPI * 10e6]], dtype=torch.float32)
    return mat, m, ms.reshape(-1).float().cpu(), p


def prepare(case, seed):
    what = case["what"]
    if what == "gradient":
        mat, m0, ms, p = _vortex(case, seed)
        sim = pkg.Sim(case["nx"], case["ny"], case["nz"], mat["d"], mat["d"], mat["d"], mat["Ms"], mat["Aex"],
                      mat["alpha"])
        return dict(case=case, sim=sim, m0=m0, ms=ms.requires_grad_(), p=p.requires_grad_())
    if what == "map":
        sims, out = [], []
        for k, (grid, count) in enumerate(_map_grids(case)):
            sub = dict(case, nx=grid[0], ny=grid[1], nz=grid[2], batch=count, tuned=True)
            sims.append(_handle(sub, _inputs(sub, seed + 1000 * k)))
            out.append(torch.empty(count, sims[-1].n, 3, device="cuda"))
        torch.cuda.synchronize()
        return dict(case=case, sims=sims, group=pkg.Group(sims, chunk=8), out=out)
    sim = _handle(case, _inputs(case, seed))
    out = torch.empty(case.get("batch", 1), sim.n, 3, device="cuda")
    torch.cuda.synchronize()
    return dict(case=case, sim=sim, out=out, first=DT_FIRST)


def _read(sim, out, modes):
    """Amplitudes (batch, modes, 2) and magnetisation (batch, cells, 3) of every instance."""
    cav = [sim.cavity(-1, mode=k) for k in range(modes)]
    for b in range(sim.batch):
        sim.get_m(b, out=out[b])
    alpha = [[[cav[k][b]["re_alpha"], cav[k][b]["im_alpha"]] for k in range(modes)] for b in range(sim.batch)]
    return {"alpha": torch.tensor(alpha, dtype=torch.float32), "m": out}


def run(state):
    case = state["case"]
    what = case["what"]
    if what == "field":
        return state["sim"].eval_field(out=state["out"])
    if what == "gradient":
        state["p"].grad = state["ms"].grad = None
        J = pkg.cavity_objective(state["sim"], state["m0"], state["p"], case["steps"], DT_RK4, wn=1.0, wavg=1.0,
                                 window=case["steps"] // 2, ckpt_every=case["ckpt"], ms=state["ms"])
        J.sum().backward()
        return {"J": J.detach(), "p": state["p"].grad, "ms": state["ms"].grad}
    if what == "map":
        state["group"].step(case["steps"], DT_RK4)
        return [_read(s, o, 1) for s, o in zip(state["sims"], state["out"])]
    sim = state["sim"]
    if case["kind"] == "dp45":
        dt, state["first"] = state["first"], 0.0      # later calls continue with the controller's step
    else:
        dt = DT_RK4
    sim.step(case["steps"], dt)
    return _read(sim, state["out"], case["modes"])


# ---------------------------------------------------------------------------
# bytes and operations
# ---------------------------------------------------------------------------
def _pad(n):
    p = 1
    while p < 2 * n - 1:
        p *= 2
    return p


def _field_work(nx, ny, nz):
    """(flops, tensor bytes) of one field evaluation: the pruned transforms, the product, and the cell's own terms."""
    px, py, pz = max(2, _pad(nx)), _pad(ny), _pad(nz)
    hx = px // 2 + 1
    lg = lambda p: math.log2(p) if p > 1 else 0.0  # noqa: E731
    fft = ny * nz * 2.5 * px * lg(px) + nz * hx * 5.0 * py * lg(py) + hx * py * 5.0 * pz * lg(pz)
    return 6.0 * fft + 30.0 * hx * py * pz + 150.0 * nx * ny * nz, 24.0 * hx * (py // 2 + 1) * (pz // 2 + 1)


def work(case):
    """Each stage reads the state and writes a torque (three floats a cell each); the tensor is read once a pass."""
    what = case["what"]
    if what == "map":
        parts = [(g, c, 4 * case["steps"]) for g, c in _map_grids(case)]
    else:
        evals = {"field": 1, "gradient": 16 * case.get("steps", 0),
                 "step": (4 if case.get("kind") == "rk4" else 6) * case.get("steps", 0)}[what]
        parts = [((case["nx"], case["ny"], case["nz"]), case.get("batch", 1), evals)]
    out = {"bytes": 0.0, "flops": 0.0}
    for (nx, ny, nz), b, evals in parts:
        fl, kern = _field_work(nx, ny, nz)
        out["flops"] += fl * b * evals
        out["bytes"] += kern + 24.0 * nx * ny * nz * b * evals
    return out


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _nf(x, y, z):
    """Newell, Williams and Dunlop (1993): f."""
    x2, y2, z2 = x * x, y * y, z * z
    R = torch.sqrt(x2 + y2 + z2)
    s = lambda v: torch.where(v > 0, v, 1.0)  # noqa: E731
    r = 0.5 * y * (z2 - x2) * torch.asinh(y / torch.sqrt(s(x2 + z2))) + 0.5 * z * (y2 - x2) * torch.asinh(
        z / torch.sqrt(s(x2 + y2)))
    return r - x * y * z * torch.atan(y * z / torch.where(x * R == 0, 1.0, x * R)) + (2 * x2 - y2 - z2) * R / 6


def _ng(x, y, z):
    """The same paper's g."""
    x2, y2, z2 = x * x, y * y, z * z
    R = torch.sqrt(x2 + y2 + z2)
    s = lambda v: torch.where(v > 0, v, 1.0)  # noqa: E731
    n = lambda v: torch.where(v == 0, 1.0, v)  # noqa: E731
    r = x * y * z * torch.asinh(z / torch.sqrt(s(x2 + y2))) + y / 6 * (3 * z2 - y2) * torch.asinh(
        x / torch.sqrt(s(y2 + z2))) + x / 6 * (3 * z2 - x2) * torch.asinh(y / torch.sqrt(s(x2 + z2)))
    return r - z2 * z / 6 * torch.atan(x * y / n(z * R)) - z * y2 / 2 * torch.atan(x * z / n(y * R)) - \
        z * x2 / 2 * torch.atan(y * z / n(x * R)) - x * y * R / 3


class _Exact:
    """Field and torque of `batch` instances on one grid, float64."""

    def __init__(self, nx, ny, nz, mat, ms, batch, profile, inst, modes):
        f64 = dict(device="cuda", dtype=torch.float64)
        self.n, self.mat, self.ms = (nz, ny, nx), mat, ms.to(**f64).reshape(nz, ny, nx)
        self.live = self.ms > 0
        self.safe = torch.where(self.live, self.ms, 1.0)
        self.pad = tuple(2 * n if n > 1 else 1 for n in self.n)
        self.N = self._tensor()
        self.batch, self.modes, self.vc = batch, modes, mat["d"] ** 3
        if profile is None:
            p = torch.zeros(nz, ny, nx, 3, **f64)
            p[..., 1] = 1.0
        else:
            p = torch.from_numpy(profile).to(**f64).reshape(nz, ny, nx, 3)
        self.p = p
        col = lambda k: torch.tensor([q[k] for q in inst], **f64)  # noqa: E731
        scale = torch.sqrt(2 * HBAR / (GAMMA * self.vc * self.ms.detach().sum()))
        self.bscale = col("g") * scale
        self.bias, self.kappa = col("bias"), col("kappa")
        self.omega = torch.stack([col("omega") * (1 + 0.2 * k) for k in range(modes)], 1)
        self.drive = None

    def _tensor(self):
        """The tensor of every offset on the padded grid (Newell near, point dipole beyond 16 cells), transformed."""
        f64 = dict(device="cuda", dtype=torch.float64)
        ax = []
        for n, p in zip(self.n, self.pad):
            k = torch.arange(p, **f64)
            ax.append(torch.where(k < n, k, k - p))
        Z, Y, X = torch.meshgrid(*ax, indexing="ij")
        r2 = X * X + Y * Y + Z * Z
        near = r2 <= 256.0
        far = torch.where(near, 1.0, r2)
        pre = 1.0 / (4 * math.pi * far * torch.sqrt(far))
        xn, yn, zn = X[near], Y[near], Z[near]
        out = []
        for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)):
            c = (X, Y, Z)
            t = pre * ((1.0 if a == b else 0.0) - 3 * c[a] * c[b] / far)
            acc = torch.zeros_like(xn)
            for i in (-1, 0, 1):
                for j in (-1, 0, 1):
                    for k in (-1, 0, 1):
                        w = (2 if i == 0 else -1) * (2 if j == 0 else -1) * (2 if k == 0 else -1)
                        v = (xn + i, yn + j, zn + k)
                        if a == b:
                            q = [v[a]] + [v[e] for e in range(3) if e != a]
                            acc += w * _nf(*q)
                        else:
                            acc += w * _ng(v[a], v[b], v[3 - a - b])
            t[near] = acc / (4 * math.pi)
            for n, p, dim in zip(self.n, self.pad, (0, 1, 2)):      # the offset -n is not reached
                if p > 1:
                    t.index_fill_(dim, torch.tensor([n], device="cuda"), 0.0)
            out.append(torch.fft.rfftn(t, dim=(0, 1, 2)).real)
        return out

    def demag(self, M):
        dims = (-3, -2, -1)
        xx, yy, zz, xy, xz, yz = self.N
        F = [torch.fft.rfftn(M[..., c], s=self.pad, dim=dims) for c in range(3)]
        H = (xx * F[0] + xy * F[1] + xz * F[2], xy * F[0] + yy * F[1] + yz * F[2], xz * F[0] + yz * F[1] + zz * F[2])
        cut = [torch.fft.irfftn(h, s=self.pad, dim=dims)[..., : self.n[0], : self.n[1], : self.n[2]] for h in H]
        return -MU0 * torch.stack(cut, -1)

    def brms(self):
        return self.bscale.reshape(-1, 1, 1, 1, 1) * self.p

    def field(self, m, Gam, t):
        """m (batch, nz, ny, nx, 3); Gam (batch, modes); t (batch,)."""
        mat, d2 = self.mat, self.mat["d"] ** 2
        B = self.demag(self.ms[..., None] * m)
        ex = torch.zeros_like(m)
        for dim in (1, 2, 3):
            if m.shape[dim] > 1:
                k = m.shape[dim] - 1
                lo, hi = m.narrow(dim, 0, k), m.narrow(dim, 1, k)
                both = (self.live.narrow(dim - 1, 0, k) & self.live.narrow(dim - 1, 1, k))[..., None]
                dif = torch.where(both, hi - lo, 0.0)
                shape = list(m.shape)
                shape[dim] = 1
                z = torch.zeros(shape, device=m.device, dtype=m.dtype)
                ex = ex + torch.cat([dif, z], dim) - torch.cat([z, dif], dim)
        B = B + (2 * mat["Aex"] / d2) * ex / self.safe[..., None]
        e = torch.tensor([1.0, 0.0, 0.0], device="cuda", dtype=torch.float64)
        B = B + 2 * mat["Ku"] * m[..., :1] / self.safe[..., None] * e
        B = B + self.bias.reshape(-1, 1, 1, 1, 3)
        G = Gam.sum(1)
        if self.drive is not None:
            amp, w, t0 = self.drive
            G = G + amp * torch.sinc(w * (t - t0) / math.pi)
        return torch.where(self.live[..., None], B + G.reshape(-1, 1, 1, 1, 1) * self.brms(), 0.0)

    def torque(self, m, Gam, t):
        B = self.field(m, Gam, t)
        c = torch.cross(m, B, dim=-1)
        k = -GAMMA / (1 + self.mat["alpha"] ** 2) * (c + self.mat["alpha"] * torch.cross(m, c, dim=-1))
        return torch.where(self.live[..., None], k, 0.0)

    def X(self, m):
        return self.vc * (self.ms[..., None] * m * self.brms()).sum((1, 2, 3, 4))

    def unit(self, m):
        r = m.norm(dim=-1, keepdim=True)
        return m / torch.where(r > 0, r, 1.0)


_DP = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
       [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
       [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
       [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]
_DP_E = [35 / 384 - 5179 / 57600, 0, 500 / 1113 - 7571 / 16695, 125 / 192 - 393 / 640, -2187 / 6784 + 92097 / 339200,
         11 / 84 - 187 / 2100, -1 / 40]
_DP_C = [0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1, 1]
_RK = [[], [0.5], [0, 0.5], [0, 0, 1.0]]
_RK_B = [1 / 6, 1 / 3, 1 / 3, 1 / 6]
_RK_C = [0, 0.5, 0.5, 1]


def _integrate(E, m, a, steps, dt0, dp, pmode):
    """`steps` steps or attempts from (m, a); a (batch, modes) complex128, a(0) at t = 0.  Yields (m, a) after each."""
    A, C = (_DP, _DP_C) if dp else (_RK, _RK_C)
    B = E.batch
    t = torch.zeros(B, device="cuda", dtype=torch.float64)
    dt = torch.full((B,), dt0, device="cuda", dtype=torch.float64)
    a0 = a
    S, Cs = torch.zeros_like(a.real), torch.zeros_like(a.real)
    lam = -(E.kappa[:, None] + 1j * E.omega)

    def rebuilt(tt):
        return torch.exp(lam * tt[:, None]) * (a0 + (-S + 1j * Cs) / HBAR)

    col = lambda v: v.reshape(-1, 1, 1, 1, 1)  # noqa: E731
    for _ in range(steps):
        km, ka = [], []
        ms, al = m, a
        for s in range(7 if dp else 4):
            w = A[s]
            ms = m + sum(col(dt) * w[j] * km[j] for j in range(s) if w[j]) if s else m
            if dp and s == 6:
                ms = E.unit(ms)
            al = a + sum(dt[:, None] * w[j] * ka[j] for j in range(s) if w[j]) if s else a
            ts = t + C[s] * dt
            km.append(E.torque(ms, 2 * (rebuilt(ts) if pmode else al).real, ts))
            X = E.X(ms)[:, None]
            ka.append(lam * al + 1j * X / HBAR)
        if dp:
            e = sum(col(dt) * _DP_E[j] * km[j] for j in range(7) if _DP_E[j])
            err = e.norm(dim=-1).amax((1, 2, 3))
            ok = err <= 1e-6
            new, nal = ms, al
        else:
            ok = torch.ones(B, device="cuda", dtype=torch.bool)
            new = E.unit(m + sum(col(dt) * _RK_B[j] * km[j] for j in range(4)))
            nal = a + sum(dt[:, None] * _RK_B[j] * ka[j] for j in range(4))
        m = torch.where(col(ok), new, m)
        t = torch.where(ok, t + dt, t)
        if pmode:
            X = E.X(m)[:, None]
            ph = torch.exp(E.kappa * t)[:, None] * X * (dt * ok)[:, None]
            S = S + ph * torch.sin(E.omega * t[:, None])
            Cs = Cs + ph * torch.cos(E.omega * t[:, None])
            a = rebuilt(t)
        else:
            a = torch.where(ok[:, None], nal, a)
        if dp:
            dt = dt * (0.9 * (1e-6 / err) ** 0.2).clamp(0.2, 5.0)
        yield m, a


def _exact_step(case, seed):
    x = _inputs(case, seed)
    batch, modes = case.get("batch", 1), case.get("modes", 1)
    E = _Exact(case["nx"], case["ny"], case["nz"], x["mat"], x["ms"], batch, x["profile"], x["inst"], modes)
    if case.get("drive"):
        E.drive = (1e3, TWOPI * 20e9, 1e-12)
    m = E.unit(x["m0"].double()).reshape((batch,) + E.n + (3,))
    a = torch.zeros(batch, modes, device="cuda", dtype=torch.complex128)
    a[:, 0] = 1.0
    if case["what"] == "field":
        t = torch.zeros(batch, device="cuda", dtype=torch.float64)
        return E.field(m, 2 * a.real, t).reshape(-1, 3)
    dp = case.get("kind") == "dp45"
    for m, a in _integrate(E, m, a, case["steps"], DT_FIRST if dp else DT_RK4, dp, case.get("cavity") == "P"):
        pass
    return {"alpha": torch.stack([a.real, a.imag], -1), "m": m.reshape(batch, -1, 3)}


def _exact_gradient(case, seed):
    mat, m0, ms, p = _vortex(case, seed)
    ms = ms.double().cuda().requires_grad_()
    p = p.double().cuda().requires_grad_()
    nx, ny, nz, steps = case["nx"], case["ny"], case["nz"], case["steps"]
    one = dict(bias=(0.0, 0.0, 0.0), omega=0.0, kappa=0.0, g=0.0)
    E = _Exact(nx, ny, nz, mat, ms, 1, None, [one], 1)
    E.bias, E.omega, E.kappa = p[:, :3], p[:, 4:5], p[:, 5]
    E.bscale = p[:, 3] * torch.sqrt(2 * HBAR / (GAMMA * E.vc * ms.detach().sum()))
    m = E.unit(torch.from_numpy(m0).double().cuda()).reshape((1,) + E.n + (3,))
    a = torch.zeros(1, 1, device="cuda", dtype=torch.complex128)
    J, window = 0.0, steps // 2
    for q, (m, a) in enumerate(_integrate(E, m, a, steps, DT_RK4, False, False)):
        if q >= steps - window:
            J = J + (a.abs() ** 2).sum(1) / window
    J = J + (a.abs() ** 2).sum(1)
    J.sum().backward()
    return {"J": J.detach(), "p": p.grad, "ms": ms.grad}


def exact(case, seed):
    what = case["what"]
    if what == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if what != "map":
            return _exact_step(case, seed)
        out = []
        for k, (grid, count) in enumerate(_map_grids(case)):
            sub = dict(case, what="step", nx=grid[0], ny=grid[1], nz=grid[2], batch=count)
            out.append(_exact_step(sub, seed + 1000 * k))
        return out
