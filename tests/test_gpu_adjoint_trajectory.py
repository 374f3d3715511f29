"""The adjoint of a rollout too long for its whole trajectory to be kept (1 GiB of states):
checkpoints and recomputed segments give the bits of one kept segment, and the simulation ends
where plain steps leave it."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu


def test_recomputed_segments_equal_kept_ones():
    import torch
    rng = np.random.default_rng(8)
    sy = inputs.actuated_box(50, 50, 50, rng)
    steps, seed = 301, np.zeros((sy.n_masses, 3), np.float32)
    assert sy.n_masses * 32 * steps > 1 << 30
    seed[:, 0] = 1.0 / sy.n_masses
    out = []
    for every in (301, 70):
        with T.Sim(sy) as sim:
            sim.step(3)
            s = torch.as_tensor(seed, device="cuda")
            ga = torch.empty(sy.n_springs, dtype=torch.float32, device="cuda")
            gp = torch.empty_like(ga)
            T.titan_adjoint(sim.handle, steps, every, s, None, ga, gp)
            sim.step(4)
            x, v, t = sim.snapshot()
            out.append((ga.cpu().numpy(), gp.cpu().numpy(), x.copy(), v.copy(), t))
    with T.Sim(sy) as sim:
        sim.step(3 + steps + 4)
        x, v, t = sim.snapshot()
    assert np.abs(out[0][0]).max() > 0 and np.abs(out[0][1]).max() > 0
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
    assert np.array_equal(out[0][2], x) and np.array_equal(out[0][3], v) and out[0][4] == t
