"""A fixed mass passes no force adjoint on: a seed of NaN or infinity there leaves every gradient as a seed of
0 gives it."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", ["pos", "vel"])
def test_seed_on_a_fixed_mass(value, which):
    sy = inputs.actuated_box(4, 3, 3, np.random.default_rng(6))
    sy.fixed[:5] = 1
    out = []
    for at in (0.0, value):
        seeds = [torch.full((sy.n_masses, 3), 1.0 / sy.n_masses, device="cuda") for _ in range(2)]
        for s in seeds:
            s[:5] = 0.0
        seeds[which == "vel"][:5] = at
        with T.Sim(sy) as sim:
            ga = torch.empty(sy.n_springs, device="cuda")
            gp = torch.empty_like(ga)
            torch.cuda.synchronize()
            T.titan_adjoint(sim.handle, 60, 0, seeds[0], seeds[1], ga, gp)
            sim.sync()
        out.append((ga.cpu().numpy(), gp.cpu().numpy()))
    assert np.abs(out[0][0]).max() > 0
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
