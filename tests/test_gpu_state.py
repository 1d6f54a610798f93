"""The saved state's bytes against the populations that the library reports,
through every way a state is copied: host memory, device memory, device memory
at an odd address, on either side of the size (32 MiB) up to which one launch
copies it; and the f-only step, which must leave h as it is.

The copies are exact.  A population is reported as stored + w (FP64): equal to
1e-15 (one rounding of an O(0.3) sum)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01316_gb300 import inputs as I

pytestmark = pytest.mark.gpu
HEADER = 56


def _solver(dims, storage, qh, w=None):
    from paper_2203_01316_gb300 import Solver
    nx, ny, nz = dims
    N = nx * ny * nz
    s = Solver(nx, ny, nz, nu=0.02, k=1e-3, lat_h=qh, storage=storage, periodic_x=w is None, T_ref=0.3)
    if w is None:
        s.set_geometry(np.zeros(N, np.uint8))
    else:
        s.set_geometry(w["flags"], w["links"], n_walls=1)
        s.set_bc(0, 1.0)
        s.set_inlet(w["u_in"], w["T_in"])
    s.init_fields(1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0))
    return s, N


def _decode(raw, N, qh, storage):
    import torch
    dt = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
    v = torch.frombuffer(bytearray(raw[HEADER:]), dtype=dt).double().numpy().reshape(27 + qh, N)
    return v[:27], v[27:]


CASES = [((33, 7, 5), st, qh) for st in ("f16", "bf16", "f32", "f64") for qh in (27, 7)] + [
    ((5, 3, 1), "f16", 27), ((101, 61, 25), "f32", 27), ((101, 61, 26), "f32", 27)]


@pytest.mark.parametrize("dims,storage,qh", CASES)
def test_every_copy_of_a_state_holds_the_populations(dims, storage, qh):
    import torch
    s, N = _solver(dims, storage, qh)
    s.step(2)
    f, h = s.populations()
    _, w27, _, _ = O.lattice(27)
    _, wh, _, _ = O.lattice(qh)
    raw = s.save_state()
    fs, hs = _decode(raw, N, qh, storage)
    assert np.abs(fs + w27[:, None] - f).max() <= 1e-15 and np.abs(hs + 0.3 * wh[:, None] - h).max() <= 1e-15
    n = s.state_size()
    even = s.save_state(torch.empty(n, dtype=torch.uint8, device="cuda"))
    odd = s.save_state(torch.empty(n + 1, dtype=torch.uint8, device="cuda")[1:])
    assert bytes(even.cpu().numpy()) == raw and bytes(odd.cpu().numpy()) == raw
    s.step(3)
    after = s.save_state()
    for again in (raw, even, odd):  # the same state from each copy, and the same steps from it
        s.load_state(again)
        assert s.save_state() == raw
        s.step(3)
        assert s.save_state() == after


@pytest.mark.parametrize("storage", ["f16", "bf16", "f32"])
@pytest.mark.parametrize("qh", [27, 7])
def test_f_only_steps_leave_h(storage, qh):
    import torch
    w = I.heated_sphere(41, 19, 13, D=7.0, cx=14.0, seed=9, u_in=0.03, T_in=0.1)
    s, N = _solver(w["dims"], storage, qh, w)
    s.step(2)
    raw = s.save_state()
    f0, h0 = s.populations()
    u = torch.empty(3 * 3 * N, dtype=torch.float32, device="cuda")
    s.step_record(3, u, advance_h=False)
    f1, h1 = s.populations()
    s.load_state(raw)
    s.step_record(3, u, advance_h=True)
    f2, h2 = s.populations()
    # f of the two kernels: two spacings of the storage at the largest deviation (below 2^-4)
    tol = {"f16": 2.0 ** -13, "bf16": 2.0 ** -10, "f32": 2.0 ** -26}[storage]
    assert np.array_equal(h1, h0) and np.abs(f1 - f2).max() <= tol and not np.array_equal(h2, h0)
