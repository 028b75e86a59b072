"""What this library is measured on: whole pieces of work as a user's program has it do them.

Every case is a dict of plain values; prepare() makes the inputs and the context a program keeps, run() is one
pass through the public entry points (paper_1206_0389_gb300.lbm, .autograd), exact() is the same in plain
float64 torch operations.  The sizes are those of this repository's own workloads (the 32^3 Taylor-Green run,
the 256^3 decaying turbulence, the 2- and 3-level jets, the jet in the tank, the 96^3 adjoint), or ragged ones
of the same ranges.  A pass ends with what such a run reads back: density and velocity fields, time statistics
and ring profiles, probed cells, audits, gradients.  Fields and logs are kept in the precision of the run's
storage, as a program that writes them to files does (the calls return float64).
"""
import math

import numpy as np
import torch

from paper_1206_0389_gb300 import lbm
from paper_1206_0389_gb300.autograd import forced_fclb

U_IN = 0.05      # inflow velocity of the jets
SEED_STEP = 7919
E27 = ((0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, 1, -1, -1, 1, -1),
       (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1, 1, 1, -1, 1, -1, 1, -1, -1),
       (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1, 1, 1, 1, -1, 1, -1, -1, -1))
W19 = (1 / 3, 1 / 18, 1 / 36)
W27 = (8 / 27, 2 / 27, 1 / 54, 1 / 216)


# ------------------------------------------------------------------------------------------------- the cases
def _uniform(name, model, storage, nb, steps, nu=1e-4, cs=0.0, walls=0, slip=0, flow="turbulence", restart=False,
             monitor="", every=0):
    return dict(name=name, kind="uniform", model=model, storage=storage, nbx=nb[0], nby=nb[1], nbz=nb[2],
                steps=steps, nu=nu, cs=cs, walls=walls, slip=slip, flow=flow, restart=restart, monitor=monitor,
                every=every)


def _jet(name, model, storage, nb, steps, D, levels=2, radius=0.0, tank=False, cs=0.0, sample=0, read=1, rest=True):
    return dict(name=name, kind="jet", model=model, storage=storage, nbx=nb[0], nby=nb[1], nbz=nb[2], steps=steps,
                D=D, levels=levels, radius=radius, tank=tank, cs=cs, sample=sample, read=read, rest=rest)


def _adjoint(name, storage, nb, steps, every):
    return dict(name=name, kind="adjoint", model="d3q27", storage=storage, nbx=nb[0], nby=nb[1], nbz=nb[2],
                steps=steps, every=every)


def listed():
    return [
        # a small verification run from start to end, as parameter studies do many of: upload, 200 steps, fields
        _uniform("tgv_32_d3q19_f64", "d3q19", "f64", (4, 4, 4), 200, nu=0.005, cs=0.1, flow="vortex", restart=True),
        # a small ragged box probed after every single step: latency of the shortest calls
        _uniform("probed_40x24x56_d3q27_f32", "d3q27", "f32", (5, 3, 7), 100, nu=1e-3, monitor="probes", every=1),
        # the headline workload between two field outputs
        _uniform("turbulence_256_d3q27_f32", "d3q27", "f32", (32, 32, 32), 400),
        # the same in half-precision storage
        _uniform("turbulence_256_d3q27_f16", "d3q27", "f16", (32, 32, 32), 400),
        # an ordinary LES run on a ragged box whose mass and momentum are watched
        _uniform("audited_184x136x104_d3q19_f32", "d3q19", "f32", (23, 17, 13), 400, cs=0.1, monitor="audit", every=20),
        # a double-precision reference run at half the headline's resolution
        _uniform("turbulence_128_d3q27_f64", "d3q27", "f64", (16, 16, 16), 40),
        # a walled channel (no-slip sides and bottom, free-slip top) in half-precision storage
        _uniform("channel_192x80x112_d3q19_f16", "d3q19", "f16", (24, 10, 14), 400, nu=1e-3, cs=0.1, walls=15, slip=8),
        # the 2-level LES jet whose statistics are sampled: the paper's first model and its evaluation quantities
        _jet("jet2_sampled_192_d3q19_f32", "d3q19", "f32", (24, 12, 12), 200, 8.0, radius=20.0, cs=0.18, sample=10, rest=False),
        # the paper's tank (walls, free-slip top, pressure outlet, nozzle) around a small 2-level jet
        _jet("tank2_192_d3q27_f32", "d3q27", "f32", (24, 12, 12), 400, 8.0, radius=20.0, tank=True, read=2, rest=False),
        # the 2-level jet at full size, from rest
        _jet("jet2_384_d3q27_f32", "d3q27", "f32", (48, 24, 24), 200, 16.0, radius=24.0),
        # the 3-level jet at the paper's scale (40 M active cells) in half-precision storage, from rest, sampled
        _jet("jet3_512_d3q27_f16", "d3q27", "f16", (64, 32, 32), 100, 32.0, levels=3, sample=20),
        # a gradient with respect to the body force, forward and backward
        _adjoint("adjoint_96_d3q27_f32", "f32", (12, 12, 12), 128, 0),
    ]


def draw(rng):
    kind = rng.choice(("uniform", "uniform", "uniform", "jet", "jet", "adjoint"))
    if kind == "adjoint":
        nb = tuple(rng.randint(2, 12) for _ in range(3))
        c = _adjoint("", rng.choice(("f32", "f32", "f64")), nb, 1, 0)
        c["steps"] = rng.randint(8, 24 if c["storage"] == "f64" else 128)
        c["every"] = rng.choice((0, 0, 1, rng.randint(2, 8)))
    elif kind == "jet":
        model = rng.choice(("d3q19", "d3q27"))
        storage = rng.choice(("f32", "f32", "f16"))
        cs = 0.18 if model == "d3q19" else 0.0
        sample = rng.choice((0, 5, 10))
        steps = rng.randrange(20, 200, 10)
        form = rng.choice(("jet", "jet", "tank", "three"))
        if form == "three":
            nb = (rng.randint(16, 40), 2 * rng.randint(7, 10), 2 * rng.randint(7, 10))
            c = _jet("", model, storage, nb, steps, 16.0, levels=3, cs=cs, sample=sample)
        elif form == "tank":
            nb = (rng.randint(12, 36), rng.randint(10, 18), rng.randint(10, 18))
            c = _jet("", model, storage, nb, steps, 8.0, radius=20.0, tank=True, cs=cs, sample=sample, rest=False,
                     read=rng.choice((1, 2)))
        else:
            nb = (rng.randint(8, 44), rng.randint(9, 24), rng.randint(9, 24))
            c = _jet("", model, storage, nb, steps, 8.0, radius=rng.uniform(12.0, 24.0), cs=cs, sample=sample,
                     rest=rng.choice((False, True)))
        if c["nbx"] * c["nby"] * c["nbz"] > 24 * 12 * 12:   # the dense fine level is set up from host arrays
            c["rest"], c["read"] = True, 1
    else:
        cells = math.exp(rng.uniform(math.log(16.0 ** 3), math.log(240.0 ** 3)))
        ax, ay = math.exp(rng.uniform(-0.5, 0.5)), math.exp(rng.uniform(-0.5, 0.5))
        side = cells ** (1 / 3) / 8
        nb = tuple(max(1, round(side * s)) for s in (ax, ay, 1 / (ax * ay)))
        model, storage = rng.choice(("d3q19", "d3q27")), rng.choice(("f32", "f32", "f16", "f64"))
        n = 512 * nb[0] * nb[1] * nb[2]
        steps = max(10, min(400, int((8e7 if storage == "f64" else 4e9) / n)))
        monitor = rng.choice(("", "", "audit", "probes"))
        walls, slip = rng.choice(((0, 0), (0, 0), (0, 0), (15, 8), (12, 0), (3, 1)))
        c = _uniform("", model, storage, nb, steps, nu=10 ** rng.uniform(-4, -2), cs=0.1 if model == "d3q19" else 0.0,
                     walls=walls, slip=slip, restart=rng.choice((False, True)), monitor=monitor,
                     every=rng.choice((1, 5, 20)) if monitor else 0)
        if c["every"]:
            c["steps"] = max(1, steps // c["every"]) * c["every"]
            if c["every"] == 1:
                c["steps"] = min(c["steps"], 100)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------- the inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * SEED_STEP + 1)
    return g


def _random_flow(shape, urms, seed):
    """A solenoidal random field (3, NZ, NY, NX) whose spectrum peaks near the fourth mode of the shortest axis."""
    NZ, NY, NX = shape
    dev = _device()
    a = torch.randn((3, NZ, NY, NX), generator=_generator(seed), device=dev, dtype=torch.float64)
    k = torch.meshgrid(*(torch.fft.fftfreq(n, 1.0 / n, device=dev, dtype=torch.float64) / n for n in shape), indexing="ij")
    kz, ky, kx = (v * min(shape) for v in k)
    kk = kx * kx + ky * ky + kz * kz
    amp = torch.where(kk > 0, kk.sqrt() * torch.exp(-kk / 16.0), torch.zeros_like(kk))
    a = [torch.fft.fftn(a[i]) * amp for i in range(3)]
    u = [1j * (ky * a[2] - kz * a[1]), 1j * (kz * a[0] - kx * a[2]), 1j * (kx * a[1] - ky * a[0])]
    u = torch.stack([torch.fft.ifftn(v).real for v in u])
    return u * (urms / math.sqrt(float((u * u).sum(0).mean()) / 3.0))


def _initial(case, seed):
    """(rho, u) of a uniform or adjoint case as float64 tensors."""
    shape = (8 * case["nbz"], 8 * case["nby"], 8 * case["nbx"])
    if case.get("flow") == "vortex":
        NZ, NY, NX = shape
        ph = torch.rand(3, generator=_generator(seed), device=_device(), dtype=torch.float64) * 2 * math.pi
        z, y, x = torch.meshgrid(*(2 * math.pi * (torch.arange(n, device=_device(), dtype=torch.float64) + 0.5) / n + ph[i]
                                   for i, n in enumerate(shape)), indexing="ij")
        u = 0.05 * torch.stack([x.sin() * y.cos() * z.cos(), -x.cos() * y.sin() * z.cos(), torch.zeros_like(x)])
        return torch.ones(shape, device=_device(), dtype=torch.float64), u
    u = _random_flow(shape, 0.04, seed)
    for c, drift in enumerate((0.02, 0.01, -0.01)):
        u[c] += drift
    return 1.001 + 0.02 * u[0], u


def _refine(case):
    """(refinement flags of each level but the finest, (y0, z0) of the axis)."""
    nb = (case["nbx"], case["nby"], case["nbz"])
    y0, z0 = 4.0 * nb[1], 4.0 * nb[2]

    def radial(scale, lo, hi, x1):
        h = 8.0 / scale
        x, y, z = ((np.arange(n * scale) + 0.5) * h for n in nb)
        r2 = (y[None, :] - y0) ** 2 + (z[:, None] - z0) ** 2
        return ((r2 >= lo * lo) & (r2 < hi * hi))[:, :, None] & (x < x1)[None, None, :]

    if case["levels"] == 2:
        # a cylinder around the axis along the whole domain (in the tank up to one block before the outlet)
        return [radial(1, 0.0, case["radius"], 8.0 * (nb[0] - 1) if case["tank"] else 8.0 * nb[0])], (y0, z0)
    # level 1 a thick ring around the shear layer near the nozzle, level 2 a thinner one inside it, trimmed so that
    # every refined block keeps its neighbours on level 1
    D = case["D"]
    r1, r2 = ((0.25 * D, 0.75 * D), (0.375 * D, 0.75 * D)) if D > 16 else ((4.0, 16.0), (6.0, 12.0))
    f0 = radial(1, r1[0], r1[1], 6.0 * D)
    inside = f0.repeat(2, 0).repeat(2, 1).repeat(2, 2)
    out = np.pad(~inside, ((1, 1), (1, 1), (0, 0)), constant_values=True)
    out = np.pad(out, ((0, 0), (0, 0), (1, 1)))          # a domain face in x is no interface
    near = np.zeros_like(inside)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                near |= out[dz:dz + near.shape[0], dy:dy + near.shape[1], dx:dx + near.shape[2]]
    return [f0, radial(2, r2[0], r2[1], 3.0 * D) & ~near], (y0, z0)


def _jet_fields(case, seed, level, axis):
    """A jet's velocity profile with fluctuations on the whole of a level: u (3, NZ, NY, NX), rho = 1."""
    shape = [8 * case["nbz"], 8 * case["nby"], 8 * case["nbx"]]
    noise = _random_flow(shape, 0.004, seed)
    s = 2 ** level
    if s > 1:
        noise = torch.nn.functional.interpolate(noise[None], scale_factor=s, mode="trilinear")[0]
    z, y = ((torch.arange(n * s, device=noise.device, dtype=torch.float64) + 0.5) / s for n in shape[:2])
    r = ((y[None, :] - axis[0]) ** 2 + (z[:, None] - axis[1]) ** 2).sqrt()
    u = noise * torch.exp(-(r / case["D"]) ** 2)[None, :, :, None]
    u[0] += (0.5 * U_IN * (1.0 - torch.tanh((r - 0.5 * case["D"]) / (0.125 * case["D"]))))[:, :, None]
    return u


def _tank(case, axis):
    if not case["tank"]:
        return {}
    return dict(walls=15, slip=8, outlet=1, nozzle=(axis[0], axis[1], 0.5 * case["D"], case["D"], 3.0 * case["D"]))


def _nu(case):
    return case["nu"] if case["kind"] == "uniform" else 8e-5 * max(1.0, case["D"] / 16) if case["kind"] == "jet" else 0.005


class State:
    """A context with the inputs of its passes; the context goes with it."""

    def __init__(self, case, ctx, **more):
        self.case, self.ctx = case, ctx
        self.__dict__.update(more)

    def __del__(self):
        lbm.lbm_destroy(self.ctx)


def _stations(case):
    return [x * case["D"] for x in (0.5, 1.0, 2.0, 4.0)]


def prepare(case, seed):
    nb = (case["nbx"], case["nby"], case["nbz"])
    omega = 1.0 / (3.0 * _nu(case) + 0.5)
    if case["kind"] == "jet":
        flags, axis = _refine(case)
        ctx = lbm.lbm_create(case["model"], case["storage"], nb, False, flags, omega, case["cs"], **_tank(case, axis))
        lbm.lbm_set_inflow(ctx, axis[0], axis[1], case["D"], U_IN, 0.01, seed)
        if not case["rest"]:
            for l in range(case["levels"]):
                lbm.lbm_init_equilibrium(ctx, l, None, _jet_fields(case, seed, l, axis).cpu().numpy())
        return State(case, ctx, axis=axis)
    rho, u = _initial(case, seed)
    if case["kind"] == "adjoint":
        ctx = lbm.lbm_create("d3q27", case["storage"], nb, True, [], omega, 0.0)
        F = 1e-6 * torch.randn(u.shape, generator=_generator(seed + 1), device=u.device, dtype=torch.float64)
        f0 = Cascaded(u.device).feq(rho.reshape(-1), u.reshape(3, -1)).reshape(27, *rho.shape)
        kind = torch.float64 if case["storage"] == "f64" else torch.float32
        return State(case, ctx, F=F.to(kind).requires_grad_(True), f0=f0.cpu().numpy())
    ctx = lbm.lbm_create(case["model"], case["storage"], nb, True, [], omega, case["cs"], walls=case["walls"], slip=case["slip"])
    rho, u = rho.cpu().numpy(), u.cpu().numpy()
    if not case["restart"]:
        lbm.lbm_init_equilibrium(ctx, 0, rho, u)
    return State(case, ctx, rho=rho, u=u, probes=_probes(case, seed))


def _probes(case, seed):
    n = 512 * case["nbx"] * case["nby"] * case["nbz"]
    return np.sort(np.random.RandomState(seed % (1 << 31)).randint(0, n, 16)).astype(np.int64)


# ------------------------------------------------------------------------------------------------- a pass
def _kept(a, storage, log=False):
    """Fields in the precision of the run's storage; logs of a half-precision run in single precision."""
    a = torch.from_numpy(np.ascontiguousarray(a))
    return a if storage == "f64" else a.half() if storage == "f16" and not log else a.float()


def _objective(f, F):
    """Kinetic energy of the central region, with the half-step velocity."""
    e = torch.tensor(E27, device=f.device, dtype=f.dtype)
    box = tuple(slice(n // 2 - 8 if n > 16 else 0, n // 2 + 8) for n in f.shape[1:])
    g = f[(slice(None),) + box]
    rho = g.sum(0)
    j = torch.einsum("aq,qzyx->azyx", e, g) + 0.5 * F[(slice(None),) + box]
    return 0.5 * ((j * j).sum(0) / rho).sum()


def run(state):
    case, ctx = state.case, state.ctx
    st = case["storage"]
    out = {}
    if case["kind"] == "adjoint":
        state.F.grad = None
        fT = forced_fclb(state.F, ctx, state.f0, case["steps"], case["every"])
        _objective(fT, state.F).backward()
        return {"f": fT.detach(), "gradient": state.F.grad}
    if case["kind"] == "jet":
        if case["sample"]:
            lbm.lbm_stats_reset(ctx)
            for _ in range(case["steps"] // case["sample"]):
                lbm.lbm_step(ctx, case["sample"])
                lbm.lbm_stats_accumulate(ctx)
            mean, var, counts = lbm.lbm_stats_radial(ctx, -1, state.axis[0], state.axis[1], 1.0, 24, _stations(case))
            mean0, var0, _ = lbm.lbm_stats_get(ctx, 0)
            return {"profile": _kept(mean, st, True), "intensity": _kept(var, st, True), "counts": counts,
                    "mean": _kept(mean0, st), "variance": _kept(var0, st, True)}
        lbm.lbm_step(ctx, case["steps"])
        for l in range(case["read"]):
            rho, u = lbm.lbm_macroscopic(ctx, l)
            out.update({"rho%d" % l: _kept(rho, st), "u%d" % l: _kept(u, st)})
        return out
    if case["restart"]:
        lbm.lbm_init_equilibrium(ctx, 0, state.rho, state.u)
    if case["monitor"]:
        log = []
        for _ in range(case["steps"] // case["every"]):
            lbm.lbm_step(ctx, case["every"])
            log.append(lbm.lbm_mass_momentum(ctx) if case["monitor"] == "audit" else lbm.lbm_get_cells(ctx, 0, state.probes))
        out["log"] = _kept(np.stack(log), st, True)
    else:
        lbm.lbm_step(ctx, case["steps"])
    rho, u = lbm.lbm_macroscopic(ctx, 0)
    out.update(rho=_kept(rho, st), u=_kept(u, st))
    return out


def work(case):
    """Each update of an active cell reads and writes its populations (the states of the larger cases are far beyond
    the caches); each sample reads the populations and reads and writes seven sums; fields come back once in float64."""
    Q = 19 if case["model"] == "d3q19" else 27
    size = {"f64": 8, "f32": 4, "f16": 2}[case["storage"]]
    blocks = case["nbx"] * case["nby"] * case["nbz"]
    cells = [512 * blocks]
    if case["kind"] == "jet":
        flags = _refine(case)[0] + [np.zeros(1, bool)]
        region = blocks
        cells = []
        for f in flags:
            cells.append(512 * (region - int(f.sum())))
            region = 8 * int(f.sum())
    updates = case["steps"] * sum(n << l for l, n in enumerate(cells))
    nbytes, flops = 2 * Q * size * updates, (200 if Q == 19 else 300) * updates
    dense = 512 * blocks
    if case["kind"] == "adjoint":
        # forward as above; backward f, lambda in, lambda out, force, gradient; f0, f_T, its adjoint, F and dL/dF
        nbytes += updates * (3 * Q * size + 9 * size) + dense * 8 * (3 * Q + 6)
        flops *= 4
    elif case["kind"] == "jet" and case["sample"]:
        nbytes += case["steps"] // case["sample"] * sum(cells) * (Q * size + 112) + dense * 56
    elif case["kind"] == "jet":
        nbytes += sum(dense * 8 ** l * 32 for l in range(case["read"]))
    else:
        nbytes += dense * 32 * (2 if case["restart"] else 1)
        if case["monitor"] == "audit":
            nbytes += case["steps"] // case["every"] * dense * Q * size
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------------- the same in 64 bits
class Model:
    """A collision in float64; arrays are (Q, cells)."""

    def __init__(self, Q, weights, dev):
        e = [[row[i] for row in E27] for i in range(Q)]
        self.Q, self.ev = Q, e
        self.at = {tuple(v): i for i, v in enumerate(e)}
        self.e = torch.tensor(e, device=dev, dtype=torch.float64)
        self.w = torch.tensor([weights[sum(c * c for c in v)] for v in e], device=dev, dtype=torch.float64)
        x, y, z = self.e.t()
        self.second = torch.stack([x * x, y * y, z * z, x * y, x * z, y * z])


class Mrt(Model):
    """D3Q19, incompressible, Smagorinsky: every rate 1 but that of the five shear moments."""

    def __init__(self, dev):
        super().__init__(19, W19, dev)
        x, y, z = self.e.t()
        xx, yy, zz = x * x, y * y, z * z
        M = torch.stack([torch.ones_like(x), x, y, z, x * y, x * z, y * z, xx - yy, xx - zz, xx + yy + zz,
                         x * yy + x * zz, xx * y + y * zz, xx * z + yy * z, x * yy - x * zz, xx * y - y * zz, xx * z - yy * z,
                         xx * yy - 2 * xx * zz + yy * zz, xx * yy + xx * zz - 2 * yy * zz, xx * yy + xx * zz + yy * zz])
        self.shear = torch.linalg.inv(M)[:, 4:9] @ M[4:9]

    def rest(self):
        return torch.zeros_like(self.w)

    def density(self, f):
        return f.sum(0)

    def velocity(self, f):
        return self.e.t() @ f

    def of_rho(self, rho):
        return rho - 1.0

    def to_rho(self, d):
        return d + 1.0

    def feq(self, d, u):
        eu = self.e @ u
        return self.w[:, None] * (d + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))

    def collide(self, f, tau0, cs, force=None):
        feq = self.feq(self.density(f), self.velocity(f))
        g = f - feq
        P = self.second @ g
        Q = (2.0 * ((P[:3] ** 2).sum(0) + 2.0 * (P[3:] ** 2).sum(0))).sqrt()
        tau = 0.5 * (tau0 + (tau0 * tau0 + 18.0 * cs * cs * Q).sqrt())
        return feq + (1.0 - 1.0 / tau) * (self.shear @ g), 1.5 * Q / tau


class Cascaded(Model):
    """D3Q27, factorized central moments, in product form: above second order every moment is at its equilibrium."""

    def __init__(self, dev):
        super().__init__(27, W27, dev)

    def rest(self):
        return self.w.clone()

    def density(self, f):
        return f.sum(0)

    def velocity(self, f):
        return (self.e.t() @ f) / f.sum(0)

    def of_rho(self, rho):
        return rho

    def to_rho(self, d):
        return d

    @staticmethod
    def line(u, second):
        """Per velocity -1, 0, 1 of one axis: the distribution of the normalised central moments (1, 0, second)."""
        s = u * u + second
        return (0.5 * (s - u), 1.0 - s, 0.5 * (s + u))

    def feq(self, rho, u):
        third = torch.full_like(rho, 1.0 / 3.0)
        p = [self.line(u[a], third) for a in range(3)]
        return torch.stack([rho * p[0][x + 1] * p[1][y + 1] * p[2][z + 1] for x, y, z in self.ev])

    def collide(self, f, tau0, cs, force=None):
        rho, j = f.sum(0), self.e.t() @ f
        u = (j if force is None else j + 0.5 * force) / rho
        M = self.second @ f
        keep = 1.0 - 1.0 / tau0
        pair = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        c = [M[k] - u[a] * j[b] - u[b] * j[a] + u[a] * u[b] * rho for k, (a, b) in enumerate(pair)]
        mean = (c[0] + c[1] + c[2]) / 3.0
        phi = [self.line(u[a], 1.0 / 3.0 + keep * (c[a] - mean) / rho) for a in range(3)]
        psi = [(u[a] - 0.5, -2.0 * u[a], u[a] + 0.5) for a in range(3)]
        kxy, kxz, kyz = (keep * v for v in c[3:])
        out = [None] * 27
        for y in range(3):
            for z in range(3):
                even = rho * phi[1][y] * phi[2][z] + kyz * psi[1][y] * psi[2][z]
                odd = kxy * psi[1][y] * phi[2][z] + kxz * phi[1][y] * psi[2][z]
                if force is not None:
                    chi = [self.line(u[a], torch.zeros_like(rho)) for a in range(3)]
                    first = 0.5 * (force[1] * psi[1][y] * chi[2][z] + force[2] * chi[1][y] * psi[2][z])
                    odd = odd + 0.5 * force[0] * chi[1][y] * chi[2][z]
                for x in range(3):
                    v = phi[0][x] * even + psi[0][x] * odd
                    if force is not None:
                        # the force's own moments have no second order along x
                        v = v + chi[0][x] * first
                    out[self.at[(x - 1, y - 1, z - 1)]] = v
        return torch.stack(out), torch.zeros_like(rho)


def _splitmix(x):
    x = np.asarray(x, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


class Plain:
    """The time-nested solver on a case's grid: dense boxes around each level, gathers by tables."""

    CHUNK = 1 << 22

    def __init__(self, case, seed):
        self.case, self.seed, self.dev = case, seed, _device()
        self.m = Mrt(self.dev) if case["model"] == "d3q19" else Cascaded(self.dev)
        self.cs = case.get("cs", 0.0) if case["model"] == "d3q19" else 0.0
        self.px = case["kind"] != "jet"
        nb = (case["nbz"], case["nby"], case["nbx"])
        flags, self.axis = _refine(case) if case["kind"] == "jet" else ([], None)
        tank = case["kind"] == "jet" and case["tank"]
        self.walls, self.slip = (15, 8) if tank else (case.get("walls", 0), case.get("slip", 0))
        self.outlet = tank
        region = np.ones(nb, bool)
        tau = 3.0 * _nu(case)
        self.lv = []
        for l in range(len(flags) + 1):
            refined = flags[l] if l < len(flags) else np.zeros_like(region)
            self.lv.append(self.level(l, [8 * n << l for n in nb], region, refined, 0.5 + tau * 2 ** l))
            region = refined.repeat(2, 0).repeat(2, 1).repeat(2, 2)
        self.nozzle_level = None
        if tank:
            self.nozzle_level = 1
            self.links(self.lv[1], _tank(case, self.axis)["nozzle"])
        for l, L in enumerate(self.lv):
            self.tables(l, L)
        self.time = 0

    def level(self, l, N, region, refined, tau0):
        """Masks of one level on a box (z, y, x) of cells that starts at `o`."""
        L = type("Level", (), {})()
        L.l, L.N, L.tau0 = l, N, tau0
        if l == 0:
            lo, hi = [0, 0, 0], list(region.shape)
            L.o, pad = [0, 0, 0 if self.px else -1], [(0, 0), (0, 0), (0, 0) if self.px else (1, 1)]
        else:
            at = np.argwhere(region)
            lo, hi = at.min(0), at.max(0) + 1
            L.o, pad = [8 * int(v) - 1 for v in lo], [(1, 1)] * 3
        cut = tuple(slice(a, b) for a, b in zip(lo, hi))

        def cells(b):
            b = torch.from_numpy(np.ascontiguousarray(b[cut])).to(self.dev)
            for d in range(3):
                b = b.repeat_interleave(8, d)
            return torch.nn.functional.pad(b, [v for p in reversed(pad) for v in p])

        def near(mask):
            return torch.nn.functional.max_pool3d(mask[None, None].half(), 3, 1, 1)[0, 0] > 0

        L.region, L.refined = cells(region), cells(refined)
        L.shape = tuple(L.region.shape)
        L.active = L.region & ~L.refined
        one = near(L.active)
        L.hidden = L.refined & near(one)
        L.update = L.active | (L.refined & one)
        x = torch.arange(L.shape[2], device=self.dev) + L.o[2]
        inside = ((x >= 0) & (x < N[2]))[None, None, :]
        L.ghost = near(L.region) & ~L.region & inside if l else torch.zeros_like(L.region)
        L.solid = torch.zeros_like(L.region)
        n = L.region.numel()
        L.f = self.m.rest()[:, None].expand(self.m.Q, n).contiguous()
        L.S = torch.zeros(n, device=self.dev, dtype=torch.float64)
        return L

    def flat(self, L, z, y, x):
        return (z * L.shape[1] + y) * L.shape[2] + x

    def links(self, L, nozzle):
        """Solid cells of the cylinder and the links that meet its surface (first the later of its two entries)."""
        y0, z0, R, x0, x1 = nozzle
        s = 0.5 ** L.l
        zc, yc, xc = ((torch.arange(n, device=self.dev, dtype=torch.float64) + o + 0.5) * s for n, o in zip(L.shape, L.o))
        Z, Y, X = zc[:, None, None], yc[None, :, None], xc[None, None, :]
        L.solid = (X >= x0) & (X <= x1) & ((Y - y0) ** 2 + (Z - z0) ** 2 <= R * R)
        sides = [[] for _ in range(7)]
        for i, (ex, ey, ez) in enumerate(self.m.ev):
            if i == 0:
                continue
            z, y, x = torch.nonzero(torch.roll(L.solid, (-ez, -ey, -ex), (0, 1, 2)) & ~L.solid, as_tuple=True)
            px, py, pz = xc[x], yc[y] - y0, zc[z] - z0
            dx, dy, dz = ex * s, ey * s, ez * s
            ts = torch.where(px > x1, (x1 - px) / dx, torch.where(px < x0, (x0 - px) / dx, torch.zeros_like(px))) if ex else torch.zeros_like(px)
            c, a, b = py * py + pz * pz - R * R, dy * dy + dz * dz, 2.0 * (py * dy + pz * dz)
            tc = torch.where(c > 0, (-b - (b * b - 4.0 * a * c).clamp(min=0).sqrt()) / (2.0 * a), torch.zeros_like(c)) if a else torch.zeros_like(c)
            cap = (px > x1) & (ts >= tc)
            back = self.flat(L, z - ez, y - ey, x - ex)
            for k, v in enumerate((torch.full_like(z, i), torch.full_like(z, self.m.at[(-ex, -ey, -ez)]), self.flat(L, z, y, x),
                                   self.flat(L, z + ez, y + ey, x + ex), back, torch.maximum(ts, tc), cap)):
                sides[k].append(v)
        L.i, L.ib, L.at_f, L.at_b, L.at_s, L.q, L.cap = (torch.cat(v) for v in sides)
        L.second = ~L.solid.reshape(-1)[L.at_s]

    def tables(self, l, L):
        L.active &= ~L.solid
        L.update &= ~L.solid
        L.valid = L.active | (L.hidden & ~L.solid) | L.update
        z, y, x = torch.nonzero(L.update, as_tuple=True)
        L.cells = self.flat(L, z, y, x)
        n, (DZ, DY, DX) = L.region.numel(), L.shape
        L.pull = []
        for q, (ex, ey, ez) in enumerate(self.m.ev):
            sz, sy, sx = z - ez, y - ey, x - ex
            if l == 0:
                sz, sy = sz % DZ, sy % DY
                sx = sx % DX if self.px else sx
            at = q * n + self.flat(L, sz, sy, sx)
            if l == 0 and self.walls:
                W, no = self.walls, torch.zeros_like(z, dtype=torch.bool)
                cy = (y == 0) if ey == 1 and W & 1 else (y == DY - 1) if ey == -1 and W & 2 else no
                cz = (z == 0) if ez == 1 and W & 4 else (z == DZ - 1) if ez == -1 and W & 8 else no
                slip_y, slip_z = bool(self.slip & (1 if ey == 1 else 2)), bool(self.slip & (4 if ez == 1 else 8))
                stop = (cy & (not slip_y)) | (cz & (not slip_z))
                for where, v, cell in ((cy & ~cz, (ex, -ey, ez), (sz, y, sx)), (cz & ~cy, (ex, ey, -ez), (z, sy, sx)),
                                       (cy & cz, (ex, -ey, -ez), (z, y, sx)), (stop, (-ex, -ey, -ez), (z, y, x))):
                    if v in self.m.at:
                        at = torch.where(where, self.m.at[v] * n + self.flat(L, *cell), at)
            L.pull.append(at)
        L.inlet = L.outflow = None
        if not self.px:
            source = L.region | L.ghost
            for name, edge, src, dst in (("inlet", -1, 1, 0), ("outflow", L.N[2], DX - 2, DX - 1)):
                if L.o[2] + dst == edge:
                    z, y = torch.nonzero(source[:, :, src], as_tuple=True)
                    setattr(L, name, (self.flat(L, z, y, torch.full_like(z, src)), self.flat(L, z, y, torch.full_like(z, dst)), z + L.o[0], y + L.o[1]))
        if l == 0:
            return
        C = self.lv[l - 1]
        z, y, x = torch.nonzero(L.ghost, as_tuple=True)
        L.ghosts = self.flat(L, z, y, x)
        axes = []
        for d, v in enumerate((z, y, x)):
            v = v + L.o[d]
            i0 = torch.div(v - 1, 2, rounding_mode="floor")
            t = torch.where(v % 2 == 0, 0.75, 0.25).double()
            i1 = i0 + 1
            if d == 2:
                i0, i1 = i0.clamp(0, C.N[2] - 1), i1.clamp(0, C.N[2] - 1)
            axes.append(((i0 - C.o[d], 1.0 - t), (i1 - C.o[d], t)))
        L.stencil = [(self.flat(C, a[0], b[0], c[0]), a[1] * b[1] * c[1]) for a in axes[0] for b in axes[1] for c in axes[2]]
        z, y, x = torch.nonzero(C.hidden, as_tuple=True)
        C.hides = self.flat(C, z, y, x)
        z, y, x = (2 * (v + C.o[d]) - L.o[d] for d, v in enumerate((z, y, x)))
        C.children = [self.flat(L, z + a, y + b, x + c) for a in (0, 1) for b in (0, 1) for c in (0, 1)]

    def inflow(self, L, sub, z, y):
        p = [self.case["D"], U_IN]
        s = 0.5 ** L.l
        disc = ((y.double() + 0.5) * s - self.axis[0]) ** 2 + ((z.double() + 0.5) * s - self.axis[1]) ** 2 < (0.5 * p[0]) ** 2
        cell = (y + L.N[1] * z).cpu().numpy().astype(np.uint64)
        xi = []
        for c in range(3):
            h = _splitmix(_splitmix(np.uint64(self.seed)) ^ np.uint64(self.time))
            h = _splitmix(h ^ np.uint64((L.l << 32) | sub))
            h = _splitmix(_splitmix(h ^ cell) ^ np.uint64(c))
            xi.append(torch.from_numpy(2.0 * (h >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 - 1.0).to(self.dev))
        u = torch.stack([p[1] * (1.0 + 0.01 * xi[0]), p[1] * 0.01 * xi[1], p[1] * 0.01 * xi[2]])
        return torch.where(disc, u, torch.zeros_like(u))

    def boundaries(self, L, sub):
        m, f = self.m, L.f
        if L.inlet is not None:
            src, dst, z, y = L.inlet
            u = self.inflow(L, sub, z, y)
            f[:, dst] = m.feq(m.density(f[:, src]), torch.zeros_like(u) if self.nozzle_level is not None else u)
        if L.outflow is not None:
            src, dst, z, y = L.outflow
            g = f[:, src]
            if self.outlet:
                d, u = m.density(g), m.velocity(g)
                g = m.feq(torch.full_like(d, float(m.of_rho(1.0))), u) + (g - m.feq(d, u))
            f[:, dst] = g
        if self.nozzle_level == L.l:
            a, b, c, q = f[L.i, L.at_f], f[L.i, L.at_s], f[L.ib, L.at_f], L.q
            low = torch.where(L.second, 2.0 * q * a + (1.0 - 2.0 * q) * b, a)
            v = torch.where(q < 0.5, low, a / (2.0 * q) + (2.0 * q - 1.0) / (2.0 * q) * c)
            at = L.at_b[L.cap]
            z, y = torch.div(at, L.shape[1] * L.shape[2], rounding_mode="floor"), torch.div(at, L.shape[2], rounding_mode="floor") % L.shape[1]
            feq = m.feq(m.density(f[:, at + 1]), self.inflow(L, sub, z + L.o[0], y + L.o[1]))
            v[L.cap] = feq[L.ib[L.cap], torch.arange(len(at), device=self.dev)]
            f[L.ib, L.at_b] = v

    def update(self, L, force=None):
        """Streams and collides the level's updated cells into new arrays."""
        f = L.f.reshape(-1)
        new, newS = L.f.clone(), L.S.clone()
        for a in range(0, len(L.cells), self.CHUNK):
            part = slice(a, a + self.CHUNK)
            g = torch.stack([f[p[part]] for p in L.pull])
            out, S = self.m.collide(g, L.tau0, self.cs, None if force is None else force[:, part])
            new[:, L.cells[part]] = out
            newS[L.cells[part]] = S
        return new, newS

    def advance(self, l, sub):
        L, m = self.lv[l], self.m
        self.boundaries(L, sub)
        old, oldS = L.f, L.S
        new, newS = self.update(L)
        if l + 1 < len(self.lv):
            K = self.lv[l + 1]
            for s in (0, 1):
                F = S = 0.0
                for at, w in K.stencil:
                    F = F + w * (old[:, at] if s == 0 else 0.5 * (old[:, at] + new[:, at]))
                    S = S + w * (oldS[at] if s == 0 else 0.5 * (oldS[at] + newS[at]))
                feq = m.feq(m.density(F), m.velocity(F))
                tc, tf = L.tau0 + 3.0 * self.cs ** 2 * S, K.tau0 + 1.5 * self.cs ** 2 * S
                K.f[:, K.ghosts] = feq + (tf - 1.0) / (2.0 * (tc - 1.0)) * (F - feq)
                K.S[K.ghosts] = 0.5 * S
                self.advance(l + 1, 2 * sub + s)
            L.f, L.S = new, newS
            self.restrict(l)
        L.f, L.S = new, newS

    def restrict(self, l):
        L, K, m = self.lv[l], self.lv[l + 1], self.m
        f = S = 0.0
        for at in L.children:
            g, s = K.f[:, at], K.S[at]
            feq = m.feq(m.density(g), m.velocity(g))
            tf, tc = K.tau0 + 3.0 * self.cs ** 2 * s, L.tau0 + 6.0 * self.cs ** 2 * s
            f = f + (feq + 2.0 * (tc - 1.0) / (tf - 1.0) * (g - feq)) / 8.0
            S = S + 2.0 * s / 8.0
        L.f[:, L.hides] = f
        L.S[L.hides] = S

    def start(self):
        """The states that prepare() sets up (a level at rest otherwise)."""
        m = self.m
        for l, L in enumerate(self.lv):
            if self.px:
                rho, u = _initial(self.case, self.seed)
            elif not self.case["rest"]:
                u = _jet_fields(self.case, self.seed, l, self.axis)
                rho = torch.ones_like(u[0])
            else:
                continue
            z, y, x = (torch.arange(n, device=self.dev) + o for n, o in zip(L.shape, L.o))
            keep = [(v >= 0) & (v < n) for v, n in zip((z, y, x), L.N)]
            box = tuple(slice(int(v[k][0]), int(v[k][-1]) + 1) for v, k in zip((z, y, x), keep))
            own = tuple(slice(b.start - o, b.stop - o) for b, o in zip(box, L.o))
            index = torch.arange(L.region.numel(), device=self.dev).reshape(L.shape)[own].reshape(-1)
            rho, u = rho[box].reshape(-1), u[(slice(None),) + box].reshape(3, -1)
            for a in range(0, len(index), self.CHUNK):
                part = slice(a, a + self.CHUNK)
                L.f[:, index[part]] = m.feq(m.of_rho(rho[part]), u[:, part])
        for l in range(len(self.lv) - 2, -1, -1):
            self.restrict(l)

    def step(self, n):
        for _ in range(n):
            self.advance(0, 0)
            self.time += 1

    def fields(self, l):
        """rho and u on the level's box, of the cells that hold a value (others NaN)."""
        L = self.lv[l]
        d, u = self.m.to_rho(self.m.density(L.f)), self.m.velocity(L.f)
        a = torch.cat([d[None], u])
        return torch.where(L.valid.reshape(-1), a, torch.full_like(a, math.nan)).reshape(4, *L.shape)

    def whole(self, l, a):
        L = self.lv[l]
        out = torch.full((len(a), *L.N), math.nan, device=self.dev, dtype=torch.float64)
        box = [(max(o, 0), min(o + n, N)) for o, n, N in zip(L.o, L.shape, L.N)]
        to = tuple(slice(p, q) for p, q in box)
        out[(slice(None),) + to] = a[(slice(None),) + tuple(slice(p - o, q - o) for (p, q), o in zip(box, L.o))]
        return out

    def rings(self, mean, var, stations, bins):
        sums = torch.zeros(4, len(stations), bins, device=self.dev, dtype=torch.float64)
        for l, L in enumerate(self.lv):
            s = 0.5 ** l
            z, y = ((torch.arange(n, device=self.dev, dtype=torch.float64) + o + 0.5) * s - c
                    for n, o, c in zip(L.shape, L.o, (self.axis[1], self.axis[0])))
            ring = torch.floor((y[None, :] ** 2 + z[:, None] ** 2).sqrt()).long()
            for k, x in enumerate(stations):
                X = int(math.floor(x * 2 ** l)) - L.o[2]
                if not 0 <= X < L.shape[2]:
                    continue
                ok = L.active[:, :, X] & (ring < bins)
                w = 0.25 ** l
                for c, v in enumerate((w * mean[l][1][:, :, X], w * var[l][0][:, :, X], torch.full_like(z, w)[:, None].expand_as(ring),
                                       torch.ones_like(z)[:, None].expand_as(ring))):
                    sums[c, k].index_add_(0, ring[ok], v[ok])
        return sums[0] / sums[2], sums[1] / sums[2]


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    p = Plain(case, seed)
    L = p.lv[0]
    rho, u = _initial(case, seed)
    F = 1e-6 * torch.randn(u.shape, generator=_generator(seed + 1), device=u.device, dtype=torch.float64)
    F = (F if case["storage"] == "f64" else F.float().double()).requires_grad_(True)
    f = p.m.feq(rho.reshape(-1), u.reshape(3, -1))
    n = f.shape[1]

    def one(f, F):
        g = torch.stack([f.reshape(-1)[t] for t in L.pull])
        return p.m.collide(g, L.tau0, 0.0, F.reshape(3, n))[0]

    for _ in range(case["steps"]):
        f = checkpoint(one, f, F, use_reentrant=False)
    f = f.reshape(27, *rho.shape)
    _objective(f, F).backward()
    return {"f": f.detach(), "gradient": F.grad}


def exact(case, seed):
    updates = work(case)["flops"] / (200 if case["model"] == "d3q19" else 300)
    if updates > (8e9 if case["kind"] == "uniform" else 4e9):
        return None   # more than about 20 seconds of plain operations
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    p = Plain(case, seed)
    p.start()
    if case["kind"] == "jet":
        if not case["sample"]:
            p.step(case["steps"])
            out = {}
            for l in range(case["read"]):
                a = p.whole(l, p.fields(l))
                out.update({"rho%d" % l: a[0], "u%d" % l: a[1:]})
            return out
        sums = [0.0] * case["levels"]
        n = case["steps"] // case["sample"]
        for _ in range(n):
            p.step(case["sample"])
            for l in range(case["levels"]):
                a = p.fields(l)
                sums[l] = sums[l] + torch.cat([a, a[1:] ** 2])
        mean = [s[:4] / n for s in sums]
        var = [s[4:] / n - m[1:] ** 2 for s, m in zip(sums, mean)]
        ring, ring_var = p.rings(mean, var, _stations(case), 24)
        return {"profile": ring, "intensity": ring_var, "counts": None, "mean": p.whole(0, mean[0]), "variance": p.whole(0, var[0])}
    out = {}
    if case["monitor"]:
        log, cells = [], torch.from_numpy(_probes(case, seed)).to(p.dev)
        f = p.lv[0]
        for _ in range(case["steps"] // case["every"]):
            p.step(case["every"])
            if case["monitor"] == "probes":
                log.append(f.f[:, cells].t().clone())
            else:
                log.append(torch.cat([(p.m.to_rho(p.m.density(f.f)) - 1.0).sum()[None], (p.m.e.t() @ f.f).sum(1)]))
        out["log"] = torch.stack(log)
    else:
        p.step(case["steps"])
    a = p.fields(0)
    out.update(rho=a[0], u=a[1:])
    return out
