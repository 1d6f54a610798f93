"""Surface flux and wall force of FP32 and 16-bit states against exactly rounded
sums (math.fsum) of the stored populations.

With half-way walls (wall_bc "abb") at T_w = T_ref a link returns what it took,
h_ibar = -h_i and f_abar = f_a, exactly, so a link's flux is -2 h_i and its force
2 e (f_a + w rho0) in terms of the stored deviations.  The library adds them in
FP64: at most 2^-53 of the running sum per addition, some hundred additions
between a lane and the total; 1e-13 of the sum of magnitudes is allowed."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01316_gb300 import inputs as I

from test_gpu_reductions import _stored

pytestmark = pytest.mark.gpu


def _plates(dims, storage, qh):
    from paper_2203_01316_gb300 import Solver
    nx, ny, nz = dims
    N = nx * ny * nz
    flags = I.channel_flags(nx, ny, nz, periodic_x=True)
    links = I.plate_walls(flags, 0.3, 0.8)
    links["wall"] = (np.arange(len(links["node"])) % 2).astype(np.int32)
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, lat_h=qh, storage=storage, periodic_x=True, T_ref=0.25, wall_bc="abb")
    s.set_geometry(flags.reshape(-1), links, n_walls=2)
    for w in range(2):
        s.set_bc(w, 0.25)
    s.init_fields(1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0))
    return s, N, links


def _check(s, N, links, v, qh):
    e, w27 = O.lattice(27)[:2]
    e = e.astype(float)
    d7 = [0, 1, 2, 3, 7, 8, 9]
    h_of = {a: a for a in range(27)} if qh == 27 else {a: i for i, a in enumerate(d7)}
    for wall in range(2):
        on = links["wall"] == wall
        node, a = links["node"][on], links["dir"][on]
        k = np.array([x in h_of for x in a])
        q = -2.0 * v[27 + np.array([h_of[x] for x in a[k]]), node[k]]
        assert abs(s.surface_flux(wall) - math.fsum(q)) <= 1e-13 * np.abs(q).sum()
        F = e[a] * (2.0 * v[a, node] + 2.0 * w27[a])[:, None]
        got = s.wall_force(wall)
        for d in range(3):
            assert abs(got[d] - math.fsum(F[:, d])) <= 1e-13 * np.abs(F[:, d]).sum()


@pytest.mark.parametrize("qh", [27, 7])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("dims", [(6, 5, 3), (70, 9, 41), (300, 5, 131)])
def test_wall_sums_are_the_exact_sums(dims, storage, qh):
    s, N, links = _plates(dims, storage, qh)
    s.step(2)
    _check(s, N, links, _stored(s, N, qh, storage)[1].double().cpu().numpy(), qh)


@pytest.mark.parametrize("qh", [27, 7])
def test_finite_wall_sums_beyond_the_float_range(qh):
    dims = (6, 5, 3)
    s, N, links = _plates(dims, "f32", qh)
    buf, v = _stored(s, N, qh, "f32")
    v[:27, links["node"][0]] = 3e38
    v[27:, links["node"][0]] = 3e38
    s.load_state(buf)
    _check(s, N, links, v.double().cpu().numpy(), qh)
