"""The accumulators of dJ/dF over a sweep of many levels and at the end of the
float range (FP32 adjoint).

A level on given records adds the same terms each time it is run, so n of them
have to give n times one.  Tolerance: on 32 nodes a component has one FP64
accumulator, whose n additions round by at most 2^-53 of the running sum each:
n 2^-53 relative, 2.3e-12 for 20,000 levels.

Range: dJ/dF is linear in mu_f.  With mu_f 2^122 times as large the terms of a
node are finite floats and 32 of them are beyond the float range; the sums are
those of mu_f times 2^122 to the accuracy of the 32-term sums (32^2 2^-49 of the
sum of magnitudes, which is the sum here: all terms are of one sign)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01316_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _level(dims, storage="f32"):
    import torch
    from paper_2203_01316_gb300 import Solver
    nx, ny, nz = dims
    N = nx * ny * nz
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, storage=storage, periodic_x=True, T_ref=0.3)
    s.set_geometry(np.zeros(N, np.uint8))
    s.init_fields(1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0))
    dt = torch.float32 if storage == "f32" else torch.float64
    F, H = s.flow_record_size()
    f, h = torch.empty(F, dtype=dt, device="cuda"), torch.empty(H, dtype=dt, device="cuda")
    s.step_record_pre(1, f, h)
    e = O.lattice(27)[0].astype(float)
    mu = np.empty((27, N))  # about e . (1, 2, 3): dJ/dF of a node is about (1, 2, 3)
    mu[:] = (e @ np.array([1.0, 2.0, 3.0]))[:, None] * (1.0 + I.uniform(5, N, -0.1, 0.1))
    muf = torch.tensor(mu.reshape(-1), dtype=dt, device="cuda")
    zero = torch.zeros(27 * N, dtype=dt, device="cuda")
    out = torch.empty_like(muf), torch.empty_like(zero)
    torch.cuda.synchronize()

    def run(n, scale=1.0):
        m = muf * scale
        torch.cuda.synchronize()
        for _ in range(n):
            s.adjoint_flow_step(f, h, m, zero, *out)
        return s.adjoint_flow_gradient(reset=True)[0]
    return run


@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_many_levels_add_up_in_fp64(storage):
    run = _level((4, 4, 2), storage)
    one = run(1)
    n = 20000
    assert (np.abs(one) > 1.0).all()
    assert np.abs(run(n) - n * one).max() <= n * 2.0 ** -53 * n * np.abs(one).max()


@pytest.mark.parametrize("dims", [(4, 4, 2), (13, 7, 5)])
def test_sums_beyond_the_float_range_are_finite(dims):
    run = _level(dims)
    one, big = run(1), run(1, 2.0 ** 122)
    assert np.isfinite(big).all() and np.abs(big).max() > 3.5e38
    assert np.abs(big * 2.0 ** -122 - one).max() <= 32 ** 2 * 2.0 ** -49 * np.abs(one).max()
