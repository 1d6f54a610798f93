"""The FP64 totals and wall sums of the library against exactly rounded sums
(math.fsum) of the populations that it stores, at sizes around the edges of
their kernels: a few nodes, more nodes than one sweep of the grid, ragged ones.

Tolerance of the totals: a node's values are added as an FP32 pair (error 2^-48
of the node's sum of magnitudes per addition, 53 additions), nodes in FP64
(2^-53 of the running total per addition): 2^-42 of the sum of all magnitudes
bounds both."""
import math

import numpy as np
import pytest

from paper_2203_01316_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _box(dims, storage, qh):
    from paper_2203_01316_gb300 import Solver
    nx, ny, nz = dims
    N = nx * ny * nz
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, lat_h=qh, storage=storage, periodic_x=True, T_ref=0.3)
    s.set_geometry(np.zeros(N, np.uint8))
    s.init_fields(1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0))
    return s, N


def _stored(s, N, qh, storage):
    """The stored deviations as float64 [27 + qh, N]."""
    import torch
    buf = s.save_state(torch.empty(s.state_size(), dtype=torch.uint8, device="cuda"))
    dt = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
    size = torch.empty(0, dtype=dt).element_size()
    return buf, buf[-(27 + qh) * N * size:].view(dt).view(27 + qh, N)


@pytest.mark.parametrize("qh", [27, 7])
@pytest.mark.parametrize("storage", ["f32", "f64", "f16", "bf16"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (33, 7, 5), (101, 67, 53)])
def test_totals_equal_the_exact_sums(dims, storage, qh):
    s, N = _box(dims, storage, qh)
    v = _stored(s, N, qh, storage)[1].double().cpu().numpy()
    mass, energy = s.balances()
    for got, x, shift in ((mass, v[:27], 1.0 * N), (energy, v[27:], 0.3 * N)):
        assert abs(got - (math.fsum(x.reshape(-1)) + shift)) <= 2.0 ** -42 * (np.abs(x).sum() + shift)


@pytest.mark.parametrize("qh", [27, 7])
def test_totals_of_values_beyond_the_float_range(qh):
    """Finite values whose sum is no float: the FP64 total is finite, the state is not diverged."""
    s, N = _box((9, 5, 3), "f32", qh)
    buf, v = _stored(s, N, qh, "f32")
    v[3, 17] = v[5, 17] = 3e38
    s.load_state(buf)
    mass, energy = s.balances()
    x = v.double().cpu().numpy()
    assert mass == pytest.approx(math.fsum(x[:27].reshape(-1)) + N, rel=1e-12)
    assert energy == pytest.approx(math.fsum(x[27:].reshape(-1)) + 0.3 * N, rel=1e-12)


@pytest.mark.parametrize("qh", [27, 7])
@pytest.mark.parametrize("wall_bc", ["iabb", "eq"])
@pytest.mark.parametrize("dims", [(6, 5, 3), (70, 9, 41), (300, 5, 131)])
def test_wall_sums_of_one_and_of_many_sweeps(dims, wall_bc, qh):
    """Surface flux and force of two walls between which the links alternate, against the oracle; the last grid
    has more wall nodes (78,600) than one sweep of the reduction's lane groups (9,728 or 38,912)."""
    from oracle import oracle as O
    from paper_2203_01316_gb300 import Solver
    nx, ny, nz = dims
    N = nx * ny * nz
    flags = I.channel_flags(nx, ny, nz, periodic_x=True)
    links = I.plate_walls(flags, 0.3, 0.8)
    links["wall"] = (np.arange(len(links["node"])) % 2).astype(np.int32)
    rho, u, T = 1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0)
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, lat_h=qh, storage="f64", periodic_x=True, T_ref=0.3, wall_bc=wall_bc)
    o = O.Oracle(O.make_params(nx=nx, ny=ny, nz=nz, qh=qh, periodic_x=True, nu=0.02, k=1e-3, wall_bc=wall_bc))
    s.set_geometry(flags.reshape(-1), links, n_walls=2)
    o.set_geometry(flags, links, nwalls=2)
    for w, Tw in enumerate((0.25, 1.5)):
        s.set_bc(w, Tw)
        o.set_wall_temperature(w, Tw)
    s.init_fields(rho, u, T)
    o.init_fields(rho, u, T)
    tol = 1e-13 * len(links["node"])  # FP64 link values of O(1), each within a few hundred ulp of the oracle's
    for w in range(2):
        assert abs(s.surface_flux(w) - o.surface_flux(w)) <= tol
        assert np.abs(s.wall_force(w) - o.wall_force(w)).max() <= tol


@pytest.mark.parametrize("n_walls", [1, 3, 64, 65])
def test_wall_temperature_gradient_of_few_and_many_walls(n_walls):
    """dJ/dT_w summed over the links of each wall, on the device up to 64 walls and on the host beyond, against the
    oracle's adjoint (1e-9 of the largest entry, the tolerance of the FP64 adjoint); a second gradient from reset
    accumulators is the same."""
    import torch
    from oracle import oracle as O
    from paper_2203_01316_gb300 import Solver
    from paper_2203_01316_gb300.autograd import thermal_objective
    nx, ny, nz = 19, 9, 11
    N = nx * ny * nz
    flags = I.channel_flags(nx, ny, nz, periodic_x=True)
    links = I.plate_walls(flags, 0.3, 0.8)
    links["wall"] = (np.arange(len(links["node"])) * 7 % n_walls).astype(np.int32)
    Tw = list(I.uniform(4, n_walls, 0.0, 1.0).astype(np.float32).astype(np.float64))
    fields = 1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0)
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, storage="f64", periodic_x=True)
    o = O.Oracle(O.make_params(nx=nx, ny=ny, nz=nz, periodic_x=True, nu=0.02, k=1e-3))
    s.set_geometry(flags.reshape(-1), links, n_walls=n_walls)
    o.set_geometry(flags, links, nwalls=n_walls)
    for w, T in enumerate(Tw):
        s.set_bc(w, T)
        o.set_wall_temperature(w, T)
    s.init_fields(*fields)
    state0 = s.save_state(torch.empty(s.state_size(), dtype=torch.uint8, device="cuda"))
    f0, h0 = s.populations()
    ref = o.adjoint(f0, h0, 5, (3, 5), ("surface", 0, 0.5), nwalls=n_walls)[2]
    for _ in range(2):
        theta = torch.zeros(N, dtype=torch.float64, device="cuda", requires_grad=True)
        T = torch.tensor(Tw, dtype=torch.float64, requires_grad=True)
        thermal_objective(theta, T, s, state0, 5, (3, 5), s.objective("surface", 0, 0.5), every=3).backward()
        assert np.abs(T.grad.numpy() - ref).max() <= 1e-9 * np.abs(ref).max()
