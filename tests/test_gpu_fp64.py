"""FP64 steps keep the precision of the stored deviations: the totals of a
small-amplitude periodic box over 2000 steps and a state at rest.

Totals: the stored deviations added exactly (math.fsum) hold to 1e-14 per node;
a step rounds 27 + 27 stores of at most 2e-3, 2 x 27 x 2^-53 x 2e-3 = 1.2e-17
per node, and 2000 steps of equal sign would give 2.4e-14, rounding of either
sign about 45 steps' worth.  A state at rest has deviations of exactly zero and
keeps them."""
import math

import numpy as np
import pytest

from paper_2203_01316_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _solver(kind, qh, T_ref, u, rho_dev, T_dev, N, dims):
    from paper_2203_01316_gb300 import Solver
    s = Solver(*dims, nu=0.02, k=1e-3, lat_h=qh, hkind=kind, storage="f64", periodic_x=True, T_ref=T_ref)
    s.set_geometry(np.zeros(N, np.uint8))
    s.init_fields(1.0 + rho_dev, u, (T_ref + T_dev) / (1.0 + rho_dev))
    return s


def _stored(s, N, qh):
    v = np.frombuffer(s.save_state()[-(27 + qh) * N * 8:], dtype=np.float64).reshape(27 + qh, N)
    return v[:27], v[27:]


@pytest.mark.parametrize("kind,qh", [("trt", 27), ("cum1st", 27), ("cum1st", 7)])
def test_totals_hold_over_2000_steps(kind, qh):
    dims = (17, 9, 5)
    N = 17 * 9 * 5
    s = _solver(kind, qh, 1.0, I.uniform(2, 3 * N, -1e-3, 1e-3), I.uniform(1, N, -1e-3, 1e-3),
                I.uniform(3, N, -1e-3, 1e-3), N, dims)
    before = [math.fsum(x.reshape(-1)) for x in _stored(s, N, qh)]
    s.step(2000)
    for x, total in zip(_stored(s, N, qh), before):
        assert abs(math.fsum(x.reshape(-1)) - total) <= 1e-14 * N


@pytest.mark.parametrize("kind", ["trt", "cum1st"])
@pytest.mark.parametrize("T_ref", [1.0, 300.0])
def test_state_at_rest_stays(kind, T_ref):
    dims, N = (7, 6, 5), 210
    z = np.zeros(N)
    s = _solver(kind, 27, T_ref, np.zeros(3 * N), z, z, N, dims)
    s.step(100)
    f, h = _stored(s, N, 27)
    assert not f.any() and not h.any()
