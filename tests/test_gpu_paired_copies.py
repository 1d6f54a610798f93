"""Copies of states kept as (f, h) words, at every alignment of the buffer and
through the other level's memory, which must show in no later state."""
import numpy as np
import pytest

from paper_2203_01316_gb300 import inputs as I

from test_gpu_16bit_boundaries import LATTICES, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [(3, 1, 2), (3, 2, 1)])
@pytest.mark.parametrize("qh", LATTICES)
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_saving_a_state_does_not_change_later_ones(storage, qh, steps):
    a, b = (_solver(storage, qh)[0] for _ in range(2))
    for n in steps:
        a.step(n)
        a.save_state()
        b.step(n)
    assert a.save_state() == b.save_state()


@pytest.mark.parametrize("offset", [0, 2, 4, 6, 8, 1])
@pytest.mark.parametrize("dims", [(1, 1, 1), (25, 7, 13), (76, 1, 1), (64, 32, 5)])
def test_paired_copies_at_every_alignment(dims, offset):
    """27 N words: below and beyond a tile of 2048, whole ones (76 and 10,240 nodes leave 4 and 0 over), odd counts."""
    import torch
    from paper_2203_01316_gb300 import Solver
    N = int(np.prod(dims))
    s = Solver(*dims, nu=0.02, k=1e-3, storage="f16", periodic_x=True, T_ref=0.3)
    s.set_geometry(np.zeros(N, np.uint8))
    s.init_fields(1.0 + I.uniform(1, N, -1e-2, 1e-2), I.uniform(2, 3 * N, -0.05, 0.05), I.uniform(3, N, 0.0, 1.0))
    raw = s.save_state()
    n = s.state_size()
    room = torch.full((n + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    s.save_state(room[16 + offset:])
    host = bytes(room.cpu().numpy())
    assert host[16 + offset:16 + offset + n] == raw
    assert set(host[:16 + offset]) == {0xA5} and set(host[16 + offset + n:]) <= {0xA5}
    s.step(2)
    s.load_state(room[16 + offset:16 + offset + n])
    assert s.save_state() == raw
