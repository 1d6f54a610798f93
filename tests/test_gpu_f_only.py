"""Steps of f alone in 16-bit storage, n in one call (with D3Q27 h: f leaves the
(f, h) words for arrays of its own and returns with the last step) against n
calls of one (which move h along), behind symmetry rows, walls and either inlet:
the same recorded velocities, the same state, byte for byte, and h as it was."""
import numpy as np
import pytest

from paper_2203_01316_gb300 import inputs as I

from test_gpu_16bit_boundaries import LATTICES, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inlet", ["zou_he", "equilibrium"])
@pytest.mark.parametrize("qh", LATTICES)
@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7])
def test_f_only_steps_in_one_call_and_one_by_one(n, storage, qh, inlet):
    import torch
    a, w = _solver(storage, qh, inlet=inlet)
    b = _solver(storage, qh, inlet=inlet)[0]
    N = a.N
    live = torch.tensor((w["flags"] != I.SOLID) & (w["flags"] != I.MIRROR), device="cuda")
    ua, ub = (torch.zeros(n * 3 * N, dtype=torch.float32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    for s in (a, b):
        s.step(5)
    h0 = a.populations()[1]
    a.step_record(n, ua, advance_h=False)
    for i in range(n):
        b.step_record(1, ub[i * 3 * N:], advance_h=False)
    for s in (a, b):
        s.sync()
    assert torch.equal(ua.view(n, 3, N)[:, :, live], ub.view(n, 3, N)[:, :, live])
    assert np.array_equal(a.populations()[1], h0) and np.array_equal(b.populations()[1], h0)
    assert a.save_state() == b.save_state()
    for s in (a, b):  # and h goes on with f
        s.step(5)
    assert a.save_state() == b.save_state()
    assert not np.array_equal(a.populations()[1], h0)
