"""Symmetry rows, the Zou-He inlet and the two-launch wall split in 16-bit
storage with either h lattice, where (f, h) are words (D3Q27) or arrays (D3Q7):
replayed graphs against single launches and one step against the oracle.

Tolerance against the oracle: a stored deviation v is stochastically rounded to
one of its two neighbours, at most one spacing away (2^-10 |v| in FP16, 2^-7 |v|
in BF16, 2^-24 for FP16's smallest), behind the FP32 step (2e-6)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01316_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LATTICES = [27, 7]


def _solver(storage, qh, kernel="auto", inlet="zou_he", seed=4, kind="trt"):
    from paper_2203_01316_gb300 import Solver
    w = I.confined_cylinder(0.2, seed=seed)
    nx, ny, nz = w["dims"]
    s = Solver(nx, ny, nz, nu=0.03, k=3e-3, lat_h=qh, hkind=kind, storage=storage, periodic_x=False, T_ref=w["T_in"],
               inlet_bc=inlet, step_kernel=kernel)
    s.set_geometry(w["flags"], w["links"], n_walls=1)
    s.set_bc(0, w["T_cyl"])
    s.set_inlet(w["u_in"], w["T_in"])
    s.init_fields(w["rho"], w["u"].reshape(-1), w["T"])
    assert len(np.unique(w["links"]["node"])) * 400 >= s.N  # the wall nodes have a launch of their own
    return s, w


@pytest.mark.parametrize("inlet", ["zou_he", "equilibrium"])
@pytest.mark.parametrize("qh", LATTICES)
@pytest.mark.parametrize("storage", ["f32", "f64", "f16", "bf16"])
def test_graph_steps_equal_single_launches(storage, qh, inlet):
    a, b = (_solver(storage, qh, k, inlet)[0] for k in ("auto", "classic"))
    for n in (37, 4, 1, 6):
        a.step(n)
        b.step(n)
        assert a.save_state() == b.save_state()


@pytest.mark.parametrize("inlet", ["zou_he", "equilibrium"])
@pytest.mark.parametrize("qh", LATTICES)
@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_one_step_matches_oracle(storage, qh, inlet):
    s, w = _solver(storage, qh, inlet=inlet)
    nx, ny, nz = w["dims"]
    o = O.Oracle(O.make_params(nx=nx, ny=ny, nz=nz, qh=qh, periodic_x=False, nu=0.03, k=3e-3, u_in=w["u_in"],
                               T_in=w["T_in"], inlet_bc=inlet))
    o.set_geometry(w["flags"], w["links"], nwalls=1)
    o.set_wall_temperature(0, w["T_cyl"])
    o.init_fields(w["rho"], w["u"].reshape(-1), w["T"])
    s.step(6)
    o.set_post(*s.populations())
    assert o.stream() == 0
    s.step(1)
    live = (w["flags"] != I.SOLID) & (w["flags"] != I.MIRROR)
    eps = 2.0 ** -10 if storage == "f16" else 2.0 ** -7
    for got, ref, q, shift in zip(s.populations(), o.post(), (27, qh), (1.0, w["T_in"])):
        stored = ref - O.lattice(q)[1][:, None] * shift
        assert (np.abs(got - ref) <= eps * np.abs(stored) + 2.0 ** -24 + 2e-6)[:, live].all()
