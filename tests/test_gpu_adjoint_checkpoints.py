"""Checkpointed gradients of small robots (the limit on kept states set so that the whole trajectory is not
kept): the bits of the whole trajectory's, whatever the interval, and the simulation left where it leaves it;
and, on the robots that test_gpu_adjoint holds the whole trajectory to, the FP64 oracle's gradients."""
import numpy as np
import pytest

import oracle
from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T
from test_gpu_adjoint import _close, _robot

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
STEPS = 120


def _run(sy, every, limit, seed=None, steps=STEPS):
    with T.Sim(sy) as sim:
        if limit is not None:
            T.titan_adjoint_limit(sim.handle, limit)
        seed = oracle.centroid_x_seed(sy.n_masses) if seed is None else seed
        s = torch.as_tensor(seed, dtype=torch.float32, device="cuda")
        ga = torch.full((sy.n_springs,), float("nan"), device="cuda")
        gp = torch.full_like(ga, float("nan"))
        torch.cuda.synchronize()
        T.titan_adjoint(sim.handle, steps, every, s, None, ga, gp)
        sim.step(3)
        x, v, t = sim.snapshot()
    return ga.cpu().numpy(), gp.cpu().numpy(), x.copy(), v.copy(), t


@pytest.mark.parametrize("every", [1, 7, 40, 50, 119, 120, 300])
def test_checkpoints_give_the_bits_of_the_whole_trajectory(every):
    sy = inputs.actuated_box(4, 4, 3, np.random.default_rng(3))
    whole = _run(sy, every, None)
    for limit in (0, 32 * 256 * STEPS // 2):          # none kept; a limit below the trajectory
        got = _run(sy, every, limit)
        for a, b in zip(whole, got):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("every", [7, 50])
@pytest.mark.parametrize("ground", [False, True], ids=["floating", "on-ground"])
def test_checkpointed_gradient_matches_the_oracle(ground, every):
    sy, steps = _robot(ground=ground, all_actuated=not ground), 200
    rng = np.random.default_rng(0)
    seed = oracle.centroid_x_seed(sy.n_masses) if ground else rng.standard_normal((sy.n_masses, 3))
    ga, gp = _run(sy, every, 0, seed, steps)[:2]
    ra, rp, _, _ = oracle.adjoint(sy, steps, seed)
    _close(ga.astype(np.float64), ra)
    _close(gp.astype(np.float64), rp)


def test_a_limit_below_the_trajectory_bounds_the_memory():
    sy = inputs.actuated_box(40, 40, 40, np.random.default_rng(4))
    taken = []
    for limit in (0, None):
        with T.Sim(sy) as sim:
            if limit is not None:
                T.titan_adjoint_limit(sim.handle, limit)
            s = torch.zeros(sy.n_masses, 3, device="cuda")
            ga = torch.empty(sy.n_springs, device="cuda")
            gp = torch.empty_like(ga)
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            T.titan_adjoint(sim.handle, 200, 15, s, None, ga, gp)
            sim.sync()
            taken.append(before - torch.cuda.mem_get_info()[0])
            del s, ga, gp
    states = 32 * sy.n_masses
    # 16 + 13 states and, per half-edge of up to 26 a slot, 28 bytes; slots are up to 1.5 a mass
    assert taken[0] <= 1.5 * (30 * states + 26 * 28 * sy.n_masses) + (64 << 20)
    assert taken[1] >= 200 * states


def test_limit_refuses_a_null_handle():
    with pytest.raises(T.TitanError):
        T.titan_adjoint_limit(None, 0)
