"""The adjoint on a device with little memory left: it falls back to checkpoints where the whole trajectory
does not fit, with the same bits, and gives its workspaces back with the simulation."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
STEPS = 150


def _gradient(sim, sy, every):
    sim.set_state(sy.pos, sy.vel)
    T.titan_set_step(sim.handle, 0)
    s = torch.zeros(sy.n_masses, 3, device="cuda")
    s[:, 0] = 1.0 / sy.n_masses
    ga = torch.empty(sy.n_springs, device="cuda")
    gp = torch.empty_like(ga)
    torch.cuda.synchronize()
    T.titan_adjoint(sim.handle, STEPS, every, s, None, ga, gp)
    sim.sync()
    x, v, t = sim.snapshot()
    return ga.cpu().numpy(), gp.cpu().numpy(), x.copy(), v.copy(), t


def test_checkpoints_where_the_trajectory_does_not_fit():
    sy = inputs.actuated_box(50, 50, 50, np.random.default_rng(5))
    whole = sy.n_masses * 32 * STEPS                  # at least: the layout adds unused slots
    assert 500 << 20 < whole and whole * 1.5 < 1 << 30
    with T.Sim(sy) as sim:
        want = _gradient(sim, sy, 20)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with T.Sim(sy) as sim:
        fill = torch.empty(torch.cuda.mem_get_info()[0] - (450 << 20), dtype=torch.uint8, device="cuda")
        try:
            got = _gradient(sim, sy, 20)
        finally:
            del fill
            torch.cuda.empty_cache()
    assert np.abs(want[0]).max() > 0 and np.abs(want[1]).max() > 0
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - (64 << 20)
