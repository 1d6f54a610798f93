"""The work that the performance of this library is measured on: what users of the solver have it do, through the
public entry points, over the range of sizes, storage types, lattices and kinds that the repository's workloads span.

Every case is one pass of one of five paths:

  march     a stretch of time steps ending in a device copy of the state, as a long run that keeps checkpoints does
  sample    a stretch of time steps ending in the macroscopic fields and the three heat fluxes of a Nusselt study
  report    the fields, totals, wall flux and wall force of a state that is not advanced
  gradient  value and gradient of a heat-flux objective with respect to the heat source and the wall temperatures
  flow      the same through the coupled adjoint, with the gradients by the body force and the inlet velocity too

on one of five geometries: a periodic box, a channel with one heated sphere, a channel with a bed of spheres, a
channel between plates, and a two-dimensional confined cylinder between symmetry planes behind a Zou-He inlet.

Results are returned in the precision of the run's storage (deviations from w rho0 and w T_ref for populations), so
that they are compared at the precision that they were computed in.  `exact` is the same physics written down once more
in 64-bit torch: central moments by explicit transforms, populations in full (not as deviations), gradients by
automatic differentiation of the whole evolution.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2203_01316_gb300 import Solver
from paper_2203_01316_gb300.autograd import flow_objective, thermal_objective

# D3Q27 velocities in the library's documented order; D3Q7 is a subset
E = np.array([
    [0, 1, 0, 0, 1, 1, 0, -1, 0, 0, 1, 1, -1, -1, 0, 0, 1, -1, -1, 0, -1, 1, 1, 1, -1, -1, -1],
    [0, 0, 1, 0, 1, 0, 1, 0, -1, 0, -1, 0, 1, 0, 1, -1, 1, -1, 0, -1, 1, -1, 1, -1, 1, -1, -1],
    [0, 0, 0, 1, 0, 1, 1, 0, 0, -1, 0, -1, 0, 1, -1, 1, 1, 0, -1, -1, 1, 1, -1, -1, -1, 1, -1]]).T
D7 = [0, 1, 2, 3, 7, 8, 9]
DIR = {tuple(e): a for a, e in enumerate(E.tolist())}
OPP = [DIR[tuple(-e)] for e in E]
FLIPY = [DIR[(e[0], -e[1], e[2])] for e in E.tolist()]
FLUID, SOLID, INLET, OUTLET, MIRROR = 0, 1, 2, 3, 4

TYPES = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float16, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "f64": 8, "f16": 2, "bf16": 2}


def _case(name, path, geo, nx, ny, nz, lat=27, kind="trt", storage="f32", steps=10, balls=0, dia=0.0, nu=0.02,
          Pr=100.0, u=0.02, every=0):
    c = dict(path=path, geo=geo, nx=nx, ny=ny, nz=nz, lat=lat, kind=kind, storage=storage, steps=steps, balls=balls,
             dia=dia, nu=nu, Pr=Pr, u=u, every=every)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest grid of the repository: a periodic vortex box, where launches and latency count
        _case("box_32_f32", "march", "box", 32, 32, 32, steps=10, nu=0.02, Pr=100.0, u=0.05),
        # the Gaussian-hill study: two-dimensional, FP64 (the scheme's own error is the result), advected
        _case("hill_256_f64", "march", "box", 256, 256, 1, kind="cum1st", storage="f64", steps=20, nu=1.0 / 6.0,
              Pr=100.0, u=0.1),
        # the confined-cylinder Nusselt study on its coarse mesh: symmetry planes, Zou-He inlet, fluxes now and then
        _case("cylinder_1000x152_f32", "sample", "cylinder", 1000, 152, 1, steps=40, dia=30.0, nu=0.03, Pr=10.0,
              u=0.01),
        # the heated sphere at half scale, an ordinary run that fills the chip a few times
        _case("sphere_192x64x64_f32", "march", "sphere", 192, 64, 64, steps=10, balls=1, dia=16.0, nu=0.016),
        # the headline workload: heated sphere, D3Q27 for both distributions
        _case("sphere_384x128x128_f32", "march", "sphere", 384, 128, 128, steps=10, balls=1, dia=32.0, nu=0.032,
              Pr=1000.0),
        # the same with 16-bit storage and stochastic rounding
        _case("sphere_384x128x128_f16", "march", "sphere", 384, 128, 128, storage="f16", steps=10, balls=1, dia=32.0,
              nu=0.032, Pr=1000.0),
        # a bed on odd sizes, many walls, BF16 storage, the seven-velocity lattice
        _case("bed_251x127x129_bf16_q7", "march", "bed", 251, 127, 129, lat=7, storage="bf16", steps=10, balls=24,
              dia=24.0, nu=0.01, u=0.01),
        # the largest: the porous bed of 33.5 million nodes
        _case("bed_512x256x256_f32_q7", "march", "bed", 512, 256, 256, lat=7, steps=5, balls=200, dia=24.0, nu=0.01,
              Pr=1000.0, u=0.01),
        # gradient by the heat source in the plate channel of the differentiation workload
        _case("plates_128x64x64_gradient", "gradient", "plates", 128, 64, 64, steps=50, every=25, nu=0.02, u=0.02),
        # the same gradient on the headline grid
        _case("sphere_384x128x128_gradient", "gradient", "sphere", 384, 128, 128, steps=20, every=20, balls=1,
              dia=32.0, nu=0.032, Pr=1000.0),
        # design of the flow: the coupled adjoint, force and inlet velocity among the parameters
        # (long enough for the sphere's flux to feel the inlet)
        _case("sphere_192x64x64_flow", "flow", "sphere", 192, 64, 64, steps=60, every=20, balls=1, dia=16.0, nu=0.016),
        # a look at a run: fields, totals, flux and force
        _case("sphere_384x128x128_report", "report", "sphere", 384, 128, 128, balls=1, dia=32.0, nu=0.032, Pr=1000.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["march"] * 6 + ["sample", "report", "gradient", "gradient", "flow"])
    if path == "sample":
        S = math.exp(rng.uniform(math.log(0.3), math.log(2.0)))
        return _case(None, path, "cylinder", int(1000 * S), int(150 * S) + 2, 1, kind=rng.choice(["trt", "srt", "1st"]),
                     steps=rng.choice([20, 40]), dia=30.0 * S, nu=0.03, Pr=rng.choice([10.0, 100.0]), u=0.01 / S)
    geo = "sphere" if path in ("flow", "report") else rng.choice(["plates", "sphere"] if path == "gradient" else
                                                                 ["box", "sphere", "sphere", "bed", "plates"])
    if path == "gradient" or path == "flow":
        nx, ny, nz = size(64, 320), size(32, 112), size(32, 112)
        storage, steps = "f32", rng.choice([10, 20])
    else:
        nx, ny, nz = (size(24, 128),) * 3 if geo == "box" else (size(64, 448), size(32, 160), size(32, 160))
        storage, steps = rng.choice(["f32", "f32", "f16", "bf16"] if path == "march" else ["f32"]), rng.choice([1, 5, 10])
        if geo == "box" and rng.random() < 0.3:
            nz, storage = 1, "f64"
    lat = rng.choice([27, 27, 7])
    kind = rng.choice(["trt", "trt", "trt", "srt", "1st"] + (["cum1st"] if path == "march" and geo == "box" else []))
    balls, dia = 0, 0.0
    if geo == "sphere":
        balls, dia = 1, min(ny, nz, nx) / 4.0
    if geo == "bed":
        dia = min(24.0, min(ny, nz, nx) / 3.0)
        balls = max(2, int(0.5 * nx * ny * nz / (2.2 * dia) ** 3))
    return _case(None, path, geo, nx, ny, nz, lat=lat, kind=kind, storage=storage, steps=steps, balls=balls, dia=dia,
                 nu=0.032, Pr=rng.choice([10.0, 100.0]), u=0.02, every=max(1, steps // rng.choice([1, 2])))


# ---- inputs ------------------------------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _temperatures(c):
    """(T at rest and at the inlet, wall temperatures, T_ref): the shift is the far field's temperature."""
    if c["geo"] == "box":
        return 1.0, [], 1.0
    if c["geo"] == "plates":
        return 0.5, [0.0, 1.0], 0.5
    if c["geo"] == "cylinder":
        return 10.0, [11.0], 10.0
    return 0.0, [1.0], 0.0


def _force(c):
    return (2e-6, 0.0, 0.0) if c["geo"] == "plates" else (0.0, 0.0, 0.0)


def _balls(c, seed):
    """Centres and radii of the spheres: one near a quarter of the length, or a bed without contacts."""
    r = np.random.RandomState(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["geo"] == "cylinder":
        return np.array([[0.2 * nx, 0.5 * (ny - 1), 0.0]]) + np.append(r.uniform(-0.5, 0.5, 2), 0.0), [0.5 * c["dia"]]
    if c["geo"] == "sphere":
        return np.array([[0.25 * nx, 0.5 * ny, 0.5 * nz]]) + r.uniform(0, 1, (1, 3)), np.array([0.5 * c["dia"]])
    got, radii = np.zeros((0, 3)), np.zeros(0)
    for _ in range(40 * c["balls"] if c["geo"] == "bed" else 0):
        R = 0.5 * c["dia"] * r.uniform(0.5, 1.0)
        p = np.array([r.uniform(R + 3, nx - R - 4), r.uniform(0, ny), r.uniform(0, nz)])
        d = got - p
        d[:, 1] -= ny * np.round(d[:, 1] / ny)
        d[:, 2] -= nz * np.round(d[:, 2] / nz)
        if (np.sqrt((d * d).sum(1)) >= radii + R + 2.0).all():
            got, radii = np.vstack([got, p]), np.append(radii, R)
        if len(radii) == c["balls"]:
            break
    return got, radii


def _geometry(c, seed):
    """Flags [nz, ny, nx] and the wall links (node, direction, q, wall) by the rules of lbm.h."""
    nx, ny, nz, geo = c["nx"], c["ny"], c["nz"], c["geo"]
    flags = np.zeros((nz, ny, nx), np.uint8)
    if geo in ("sphere", "bed", "cylinder"):
        flags[:, :, 0], flags[:, :, -1] = INLET, OUTLET
    links = []
    if geo == "plates":
        flags[:, [0, -1], :] = SOLID
        z, x = np.meshgrid(np.arange(nz), np.arange(nx), indexing="ij")
        for a in range(1, 27):
            if E[a][1]:
                y, q, w = (1, 0.3, 0) if E[a][1] < 0 else (ny - 2, 0.7, 1)
                n = (x + nx * (y + ny * z)).reshape(-1)
                links.append((n, np.full(n.size, a), np.full(n.size, q), np.full(n.size, w)))
    elif geo != "box":
        flat = geo == "cylinder"
        found = []
        for p, R in zip(*_balls(c, seed)):
            at = [np.arange(int(math.floor(v - R)) - 2, int(math.ceil(v + R)) + 3) for v in p]
            Z, Y, X = np.meshgrid([0] if flat else at[2], at[1], at[0], indexing="ij")
            d = np.stack([X - p[0], Y - p[1], (Z - p[2]) * (not flat)])
            inside = (d * d).sum(0) <= R * R
            flags[Z[inside] % nz, Y[inside] % ny, X[inside]] = SOLID
            found.append((X, Y, Z, d, inside, R))
        for X, Y, Z, d, inside, R in found:
            for a in range(1, 27):
                e = E[a] * np.array([1, 1, not flat])
                ee = float(e @ e)
                if not ee:
                    continue
                t = d + e[:, None, None, None]
                hit = ~inside & ((t * t).sum(0) <= R * R)
                dh = d[:, hit]
                de, dd = e @ dh, (dh * dh).sum(0)
                q = (-de - np.sqrt(np.maximum(de * de - ee * (dd - R * R), 0.0))) / ee
                n = X[hit] + nx * (Y[hit] % ny + ny * (Z[hit] % nz))
                links.append((n, np.full(n.size, a), np.clip(q, 1e-38, 1.0), np.zeros(n.size)))
    if geo == "cylinder":
        flags[:, [0, -1], :] = MIRROR
    node, dr, q, wall = (np.concatenate([l[k] for l in links]) if links else np.zeros(0) for k in range(4))
    return flags, {"node": node.astype(np.int32), "dir": dr.astype(np.int32), "q": q.astype(np.float32),
                   "wall": wall.astype(np.int32)}


def _fields(c, seed):
    """rho [N], u [3, N], T [N] in 64 bits: a uniform stream with a few smooth modes of seeded phase on it."""
    dev = _device()
    r = np.random.RandomState(seed + 7)

    def wave(n, m, p):
        i = torch.arange(n, dtype=torch.float64, device=dev)
        return torch.sin(2 * math.pi * (m * i / n + p))

    def modes():
        s = 0.0
        for m in (1, 2):
            p = r.uniform(0, 1, 3)
            s = s + (wave(c["nz"], m, p[2])[:, None, None] * wave(c["ny"], m, p[1])[None, :, None] *
                     wave(c["nx"], m, p[0])[None, None, :] / m)
        return s.reshape(-1)

    T0 = _temperatures(c)[0]
    rho = 1.0 + 1e-4 * modes()
    u = torch.stack([c["u"] + 0.2 * c["u"] * modes(), 0.2 * c["u"] * modes(), 0.2 * c["u"] * modes()])
    T = T0 + (0.1 * modes() if c["geo"] in ("box", "cylinder") else 0.05 * (1.0 + 0.5 * modes()))
    return rho, u, T


def _source(c, seed):
    g = torch.Generator().manual_seed(seed + 11)
    n = c["nx"] * c["ny"] * c["nz"]
    th = 1e-5 * torch.rand(n, generator=g, dtype=torch.float32)
    return th.to(_device())


def _objective(c):
    """(kind, index, weight, window): the heat flux of the last wall, mean over the last part of the window."""
    n = max(1, c["steps"] // 4)
    return "surface", 1 if c["geo"] == "plates" else 0, 1.0 / (n + 1), (c["steps"] - n, c["steps"])


def prepare(case, seed):
    c = case
    T0, Tw, T_ref = _temperatures(c)
    s = Solver(c["nx"], c["ny"], c["nz"], nu=c["nu"], Pr=c["Pr"], lat_h=c["lat"], hkind=c["kind"], storage=c["storage"],
               periodic_x=c["geo"] in ("box", "plates"), T_ref=T_ref,
               inlet_bc="zou_he" if c["geo"] == "cylinder" else "equilibrium")
    if c["geo"] in ("sphere", "bed"):
        s.build_spheres(*_balls(c, seed))
    else:
        flags, links = _geometry(c, seed)
        s.set_geometry(flags.reshape(-1), links, n_walls=max(1, len(Tw)))
    for i, T in enumerate(Tw):
        s.set_bc(i, T)
    if c["geo"] in ("sphere", "bed", "cylinder"):
        s.set_inlet((c["u"], 0.0, 0.0), T0)
    s.set_force(_force(c))
    rho, u, T = _fields(c, seed)
    torch.cuda.synchronize()  # the solver runs on a stream of its own
    s.init_fields(rho, u, T)
    s.sync()
    st = {"case": c, "solver": s}
    if c["path"] in ("march", "gradient", "flow"):
        st["copy"] = s.save_state(torch.empty(s.state_size(), dtype=torch.uint8, device="cuda"))
    if c["path"] in ("gradient", "flow"):
        kind, index, weight, st["window"] = _objective(c)
        st["objective"] = s.objective(kind, index, weight)
        st["theta"] = _source(c, seed)
    return st


def run(state):
    c, s = state["case"], state["solver"]
    if c["path"] == "march":
        s.step(c["steps"])
        s.save_state(state["copy"])
        values = 27 + c["lat"], s.N
        pops = state["copy"][-(values[0] * values[1] * SIZE[c["storage"]]):].view(TYPES[c["storage"]]).view(values)
        return pops[:27], pops[27:]
    if c["path"] == "sample":
        s.step(c["steps"])
        q = s.surface_flux(0), s.section_flux(c["nx"] // 20), s.section_flux(c["nx"] - 1 - c["nx"] // 10)
        return [v.float() for v in s.macros(device="cuda")] + [np.float32(v) for v in q]
    if c["path"] == "report":
        fields = [v.float() for v in s.macros(device="cuda")]
        return fields + [np.float32(v) for v in s.balances() + (s.surface_flux(0),)] + [s.wall_force(0).astype("f4")]
    theta = state["theta"].detach().requires_grad_()
    Tw = torch.tensor(_temperatures(c)[1], dtype=torch.float32, requires_grad=True)
    if c["path"] == "gradient":
        J = thermal_objective(theta, Tw, s, state["copy"], c["steps"], state["window"], state["objective"],
                              every=c["every"])
        J.backward()
        return J.detach().float(), theta.grad, Tw.grad
    F = torch.tensor(_force(c), dtype=torch.float32, requires_grad=True)
    u_in = torch.tensor([c["u"], 0.0, 0.0], dtype=torch.float32, requires_grad=True)
    J = flow_objective(theta, Tw, F, u_in, s, state["copy"], c["steps"], state["window"], state["objective"],
                       every=c["every"])
    J.backward()
    return J.detach().float(), theta.grad, Tw.grad, F.grad, u_in.grad


def work(case):
    """Bytes: per step every population of every non-solid node read once and written once (a step cannot start before
    the last one has ended everywhere nearby, so a stretch of n steps is n such passes), then the copy or the fields.
    A gradient adds, per level, the recomputed flow step with what it records, and the adjoint's own read and write.
    Operations: the two transforms and the relaxation of each distribution, per node and step."""
    c = case
    size, Q = SIZE[c["storage"]], 27 + c["lat"]
    nodes = c["nx"] * c["ny"] * c["nz"]
    live = nodes
    if c["balls"]:
        mean = 1.0 if c["geo"] == "sphere" else 15.0 / 32.0  # mean of (d / dia)^3 for d uniform in [dia / 2, dia]
        live -= c["balls"] * math.pi / 6.0 * c["dia"] ** 3 * mean
    if c["geo"] == "cylinder":
        live -= 2 * c["nx"] + math.pi / 4.0 * c["dia"] ** 2
    if c["geo"] == "plates":
        live -= 2 * c["nx"] * c["nz"]
    step, ops = 2 * Q * size, 400 + (400 if c["lat"] == 27 else 60)
    if c["path"] == "march":
        return {"bytes": live * step * c["steps"] + 2 * nodes * Q * size, "flops": live * ops * c["steps"]}
    if c["path"] == "sample":
        return {"bytes": live * (step * c["steps"] + Q * size + 20), "flops": live * ops * c["steps"]}
    if c["path"] == "report":
        return {"bytes": live * (Q * size + 20), "flops": live * (27 * 7 + c["lat"])}
    if c["path"] == "gradient":
        again, back = 54 * size + 12, 2 * c["lat"] * size + 12
    else:
        again, back = step + (10 + c["lat"]) * size, step + (10 + c["lat"]) * size
    return {"bytes": live * (step + again + back) * c["steps"], "flops": live * 2.5 * ops * c["steps"]}


# ---- the same in 64 bits -----------------------------------------------------------------------------------------------
class _Exact:
    """The model of the library's interface with full populations f [27, nz, ny, nx], h [Q, nz, ny, nx] in 64 bits."""

    def __init__(self, c, seed):
        self.c, self.dev = c, _device()
        self.shape = (c["nz"], c["ny"], c["nx"])
        flags, links = _geometry(c, seed)
        self.flags = torch.from_numpy(flags).to(self.dev)
        self.solid = (self.flags == SOLID) | (self.flags == MIRROR)
        self.dirs = list(range(27)) if c["lat"] == 27 else D7
        self.k = c["nu"] / c["Pr"]
        self.sH = 1.0 / (3.0 * self.k + 0.5)
        self.bounded = c["geo"] in ("sphere", "bed", "cylinder")
        self.zou_he = c["geo"] == "cylinder"
        T0, Tw, _ = _temperatures(c)
        self.T_in, self.Tw = T0, torch.tensor(Tw, dtype=torch.float64, device=self.dev)
        self.u_in = torch.tensor([c["u"], 0.0, 0.0], dtype=torch.float64, device=self.dev)
        self.F = torch.tensor(_force(c), dtype=torch.float64, device=self.dev)
        self.Q = torch.zeros((), dtype=torch.float64, device=self.dev)
        w1 = {0: 2 / 3, 1: 1 / 6, -1: 1 / 6}
        w = [w1[x] * w1[y] * w1[z] for x, y, z in E.tolist()]
        self.w = torch.tensor(w, dtype=torch.float64, device=self.dev).view(27, 1, 1, 1)
        self.wh = self.w if c["lat"] == 27 else torch.tensor([0.0] + [1 / 6] * 6, dtype=torch.float64,
                                                            device=self.dev).view(7, 1, 1, 1)
        keys = links["node"].astype(np.int64) * 32 + links["dir"]
        self.links = {}
        for a in range(1, 27):
            at = links["dir"] == a
            if at.any():
                node = links["node"][at].astype(np.int64)
                thin = np.isin(node * 32 + OPP[a], keys)
                put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(self.dev)  # noqa: E731
                self.links[a] = (put(node), put(links["q"][at].astype(np.float64)), put(thin),
                                 put(links["wall"][at].astype(np.int64)))

    # equilibria in product form, w_i(u) = (c_s^2 + u^2 +- u) / 2 and 1 - c_s^2 - u^2 per axis
    def equilibrium(self, psi, u, Q=27):
        one = []
        for d in range(3):
            m, p, z = 0.5 * (1 / 3 + u[d] ** 2 - u[d]), 0.5 * (1 / 3 + u[d] ** 2 + u[d]), 2 / 3 - u[d] ** 2
            one.append({-1: m, 0: z, 1: p})
        if Q == 27:
            return torch.stack([psi * one[0][x] * one[1][y] * one[2][z] for x, y, z in E.tolist()])
        arms = [psi * one[d][s] for s in (1, -1) for d in range(3)]
        return torch.stack([psi - sum(arms)] + arms)

    @staticmethod
    def _axis(C, v, dim, forward):
        a, b, c = C.unbind(dim)
        if forward:
            m0, m1, m2 = a + b + c, c - a, c + a
            return torch.stack([m0, m1 - v * m0, m2 - 2 * v * m1 + v * v * m0], dim)
        m0, m1, m2 = a, b + v * a, c + 2 * v * b + v * v * a
        return torch.stack([0.5 * (m2 - m1), m0 - m2, 0.5 * (m2 + m1)], dim)

    def central(self, g, v):
        """Central moments K[o, n, m] of 27 populations about v."""
        C = torch.stack([g[DIR[(x, y, z)]] for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)])
        C = C.view(3, 3, 3, *g.shape[1:])
        for dim, d in ((2, 0), (1, 1), (0, 2)):
            C = self._axis(C, v[d], dim, True)
        return C

    def populations(self, K, v):
        for dim, d in ((0, 2), (1, 1), (2, 0)):
            K = self._axis(K, v[d], dim, False)
        return torch.stack([K[z + 1, y + 1, x + 1] for x, y, z in E.tolist()])

    @staticmethod
    def moments(f):
        j = [sum(int(e[d]) * f[a] for a, e in enumerate(E) if e[d]) for d in range(3)]
        return f.sum(0), j

    def collide_f(self, f):
        """Cumulants of order two relaxed (shear with omega, the trace to equilibrium), all higher ones zero."""
        rho, j = self.moments(f)
        mu = [v / rho for v in j]
        K = self.central(f, mu)
        om = 1.0 - 1.0 / (3.0 * self.c["nu"] + 0.5)
        xx, yy, zz = K[0, 0, 2], K[0, 2, 0], K[2, 0, 0]
        dxy, dxz = om * (xx - yy), om * (xx - zz)
        xx = rho / 3 + (dxy + dxz) / 3
        yy, zz = xx - dxy, xx - dxz
        xy, xz, yz = om * K[0, 1, 1], om * K[1, 0, 1], om * K[1, 1, 0]
        zero = torch.zeros_like(rho)
        P = {(0, 0, 0): rho, (2, 0, 0): xx, (0, 2, 0): yy, (0, 0, 2): zz, (1, 1, 0): xy, (1, 0, 1): xz, (0, 1, 1): yz,
             (2, 2, 0): (xx * yy + 2 * xy * xy) / rho, (2, 0, 2): (xx * zz + 2 * xz * xz) / rho,
             (0, 2, 2): (yy * zz + 2 * yz * yz) / rho, (2, 1, 1): (xx * yz + 2 * xy * xz) / rho,
             (1, 2, 1): (yy * xz + 2 * xy * yz) / rho, (1, 1, 2): (zz * xy + 2 * xz * yz) / rho,
             (2, 2, 2): (xx * yy * zz + 2 * (xx * yz * yz + yy * xz * xz + zz * xy * xy) + 8 * xy * xz * yz) / rho ** 2}
        K = torch.stack([P.get((m, n, o), zero) for o in range(3) for n in range(3) for m in range(3)])
        v = [mu[d] + self.F[d] / rho for d in range(3)]
        u = [mu[d] + 0.5 * self.F[d] / rho for d in range(3)]
        return self.populations(K.view(3, 3, 3, *rho.shape), v), u

    def collide_h(self, h, u, Q):
        kind, s = self.c["kind"], self.sH
        rate = [{"trt": s if o % 2 else 1.0, "srt": s}.get(kind, s if o == 1 else 1.0) for o in range(7)]
        H = h.sum(0)
        if kind == "cum1st":
            j = [sum(int(E[a][d]) * h[i] for i, a in enumerate(self.dirs) if E[a][d]) for d in range(3)]
            return self.equilibrium(H + Q, [u[d] + (1.0 - s) * (j[d] / H - u[d]) for d in range(3)], self.c["lat"])
        relax = lambda Y, eq, o: (1 - rate[o]) * Y + rate[o] * (H + 0.5 * Q) * eq + (1 - 0.5 * rate[o]) * Q * eq  # noqa: E731
        if self.c["lat"] == 27:
            K = self.central(h, u)
            eq = {0: 1.0, 1: 0.0, 2: 1 / 3}
            K = torch.stack([relax(K[o, n, m], eq[m] * eq[n] * eq[o], m + n + o)
                             for o in range(3) for n in range(3) for m in range(3)])
            return self.populations(K.view(3, 3, 3, *H.shape), u)
        y0 = relax(H, 1.0, 0)
        plus, minus = [], []
        for d in range(3):
            m1, m2 = h[1 + d] - h[4 + d], h[1 + d] + h[4 + d]
            y1, y2 = relax(m1 - u[d] * H, 0.0, 1), relax(m2 - 2 * u[d] * m1 + u[d] ** 2 * H, 1 / 3, 2)
            m1, m2 = y1 + u[d] * y0, y2 + 2 * u[d] * y1 + u[d] ** 2 * y0
            plus.append(0.5 * (m2 + m1))
            minus.append(0.5 * (m2 - m1))
        return torch.stack([y0 - sum(plus) - sum(minus)] + plus + minus)

    def start(self, rho, u, T):
        """Equilibrium, one collision, and the planes' and solid nodes' values."""
        rho, T, u = rho.view(self.shape), T.view(self.shape), [v.view(self.shape) for v in u]
        f, u2 = self.collide_f(self.equilibrium(rho, u))
        h = self.collide_h(self.equilibrium(rho * T, u, self.c["lat"]), u2, self.Q)
        return self.planes(f, h, True)

    def inlet(self):
        u = [self.u_in[d].view(1, 1) for d in range(3)]
        one = torch.ones(1, 1, dtype=torch.float64, device=self.dev)
        return self.equilibrium(one, u), self.equilibrium(self.T_in * one, u, self.c["lat"])

    def planes(self, f, h, start=False):
        if self.bounded and (start or not self.zou_he):
            fi, hi = self.inlet()
            at = (self.flags == INLET)
            f = torch.where(at, fi[..., None], f)
            h = torch.where(at, hi[..., None], h)
        return torch.where(self.solid, self.w, f), torch.where(self.solid, self.wh * _temperatures(self.c)[2], h)

    def mirror(self, g, dirs):
        flip = [dirs.index(FLIPY[a]) for a in dirs]
        g = g.clone()
        g[:, :, 0], g[:, :, -1] = g[flip][:, :, 1], g[flip][:, :, -2]
        return g

    def pull(self, g, dirs):
        out = []
        for i, a in enumerate(dirs):
            x, y, z = E[a].tolist()
            r = torch.roll(g[i], (z, y, x), (0, 1, 2))
            if self.bounded and x == -1:  # zero gradient at the outlet
                last = torch.roll(g[i][:, :, -1], (z, y), (0, 1))
                r = torch.cat([r[:, :, :-1], last[:, :, None]], 2)
            out.append(r)
        return torch.stack(out)

    def walls(self, g, post, dirs, sign):
        """Interpolated bounce-back (sign 1) or anti-bounce-back (sign -1, the wall's temperature) of every link."""
        n = g[0].numel()
        flat, old = g.reshape(-1), post.reshape(-1)
        at, new = [], []
        for i, a in enumerate(dirs):
            if a not in self.links:
                continue
            node, q, thin, wall = self.links[a]
            b = dirs.index(OPP[a])
            own, back, far = old[i * n + node], old[b * n + node], flat[i * n + node]
            add = 0.0 if sign > 0 else 2.0 * float(self.wh.view(-1)[i]) * self.Tw[wall]
            qq = torch.clamp(q, min=0.5)
            near = sign * (2 * q * own + (1 - 2 * q) * far) + add
            other = (sign * own + (2 * qq - 1) * back + add) / (2 * qq)
            at.append(b * n + node)
            new.append(torch.where((q <= 0.5) & ~thin, near, other))
        if not at:
            return g
        return flat.index_put((torch.cat(at),), torch.cat(new)).view(g.shape)

    def fill_inlet(self, f, h):
        """Zou-He: the unknown arrivals (e_x = 1) of the inlet plane."""
        u = [self.u_in[d] for d in range(3)]
        p = f[:, :, :, 0]
        rho = (sum(p[a] for a in range(27) if E[a][0] == 0) + 2 * sum(p[a] for a in range(27) if E[a][0] == -1)) / (1 - u[0])
        fe = self.equilibrium(rho, u)
        N = [sum(int(E[a][d]) * (p[a] - fe[a]) for a in range(27) if E[a][0] == 0 and E[a][d]) / 6 for d in range(3)]
        p = [p[OPP[a]] + fe[a] - fe[OPP[a]] - int(E[a][1]) * N[1] - int(E[a][2]) * N[2] if E[a][0] == 1 else p[a]
             for a in range(27)]
        known = sum(h[i, :, :, 0] for i, a in enumerate(self.dirs) if E[a][0] != 1)
        amount = (rho * self.T_in - known) / (0.5 * (1 / 3 + u[0] ** 2 + u[0]))
        he = self.equilibrium(amount, u, self.c["lat"])
        r = [he[i] if E[a][0] == 1 else h[i, :, :, 0] for i, a in enumerate(self.dirs)]
        f, h = f.clone(), h.clone()
        f[:, :, :, 0], h[:, :, :, 0] = torch.stack(p), torch.stack(r)
        return f, h

    def arrive(self, f, h):
        if self.c["geo"] == "cylinder":
            f, h = self.mirror(f, list(range(27))), self.mirror(h, self.dirs)
        gf, gh = self.pull(f, list(range(27))), self.pull(h, self.dirs)
        gf, gh = self.walls(gf, f, list(range(27)), 1), self.walls(gh, h, self.dirs, -1)
        return self.fill_inlet(gf, gh) if self.zou_he else (gf, gh)

    def step(self, f, h):
        gf, gh = self.arrive(f, h)
        f, u = self.collide_f(gf)
        return self.planes(f, self.collide_h(gh, u, self.Q))

    # what is read off a state
    def fields(self, f, h):
        rho, j = self.moments(f)
        u = torch.stack([(j[d] - 0.5 * self.F[d]) / rho for d in range(3)])
        T = (h.sum(0) - 0.5 * self.Q) / rho
        if self.bounded:
            at = self.flags == INLET
            rho, T = torch.where(at, 1.0, rho), torch.where(at, self.T_in, T)
            u = torch.where(at, self.u_in.view(3, 1, 1, 1), u)
        return [torch.where(self.solid, 0.0, v).reshape(*v.shape[:-3], -1) for v in (rho, u, T)]

    def surface_flux(self, h, wall):
        g = self.walls(self.pull(h, self.dirs), h, self.dirs, -1)
        n, total = h[0].numel(), 0.0
        for i, a in enumerate(self.dirs):
            if a in self.links:
                node, _, _, w = self.links[a]
                node = node[w == wall]
                total = total + (g.reshape(-1)[self.dirs.index(OPP[a]) * n + node] - h.reshape(-1)[i * n + node]).sum()
        return total

    def wall_force(self, f):
        dirs = list(range(27))
        g = self.walls(self.pull(f, dirs), f, dirs, 1)
        n, F = f[0].numel(), np.zeros(3)
        for a, (node, _, _, _) in self.links.items():
            F += E[a] * float((f.reshape(-1)[a * n + node] + g.reshape(-1)[OPP[a] * n + node]).sum())
        return F

    def section_flux(self, h, x):
        live = ~self.solid[:, :, x]
        return float(sum(int(E[a][0]) * h[i, :, :, x][live].sum() for i, a in enumerate(self.dirs) if E[a][0]))


def exact(case, seed):
    c = case
    m = _Exact(c, seed)
    with torch.no_grad():
        f, h = m.start(*_fields(c, seed))
        if c["path"] == "march":
            for _ in range(c["steps"]):
                f, h = m.step(f, h)
            T_ref = _temperatures(c)[2]
            return (f - m.w).view(27, -1), (h - m.wh * T_ref).view(c["lat"], -1)
        if c["path"] == "sample":
            for _ in range(c["steps"]):
                f, h = m.step(f, h)
            q = m.surface_flux(h, 0).item(), m.section_flux(h, c["nx"] // 20), m.section_flux(h, c["nx"] - 1 - c["nx"] // 10)
            return m.fields(f, h) + list(q)
        if c["path"] == "report":
            live = ~m.solid
            totals = [float(f.sum(0)[live].sum()), float(h.sum(0)[live].sum())]
            return m.fields(f, h) + totals + [m.surface_flux(h, 0).item(), m.wall_force(f)]
    theta = _source(c, seed).double().requires_grad_()
    m.Q = theta.view(m.shape)
    m.Tw.requires_grad_()
    kind, wall, weight, (lo, hi) = _objective(c)
    leaves = [theta, m.Tw]
    if c["path"] == "flow":
        # the library takes these as 32-bit values from the caller
        m.F, m.u_in = (v.float().double().requires_grad_() for v in (m.F, m.u_in))
        leaves += [m.F, m.u_in]
    J = 0.0
    for k in range(c["steps"] + 1):
        if lo <= k <= hi:
            J = J + weight * checkpoint(m.surface_flux, h, wall, use_reentrant=False)
        if k < c["steps"]:
            if c["path"] == "flow":
                f, h = checkpoint(m.step, f, h, use_reentrant=False)
            else:  # the flow does not depend on the heat source
                with torch.no_grad():
                    gf = m.walls(m.pull(f, list(range(27))), f, list(range(27)), 1)
                    f, u = m.collide_f(gf)

                def warm(h, u=u):
                    gh = m.walls(m.pull(h, m.dirs), h, m.dirs, -1)
                    return m.collide_h(gh, u, m.Q)

                f, h = m.planes(f, checkpoint(warm, h, use_reentrant=False))
    grads = torch.autograd.grad(J, leaves)
    return [J.detach()] + list(grads)
