"""The actuated forms of the halo and box step kernels on grids of more than two CTAs per SM (the
two-column form) and of fewer (the deep form), sinusoid and worm, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu
STEPS, OMEGA, PERIOD = 12, 20.0, 1.0


@pytest.mark.parametrize("n", [20, 46])
@pytest.mark.parametrize("worm", [False, True])
@pytest.mark.parametrize("kernel", [6, 4])
def test_actuated_step_matches_oracle(kernel, worm, n):
    rng = np.random.default_rng(100 * kernel + 10 * worm + n)
    sy = inputs.actuated_box(n, n, n, rng)
    sy.vel = rng.normal(0, 0.05, sy.pos.shape)
    if kernel == 4:                                   # off the grid: the halo kernel
        sy.pos = sy.pos + rng.uniform(-0.01, 0.01, sy.pos.shape)
    if worm:                                          # offsets half a step off, as the edits test has them
        sy.act_phase = (np.floor(rng.uniform(0, PERIOD, sy.n_springs) / sy.dt) + 0.5) * sy.dt
    with T.Sim(sy, exec_mode=T.EXEC_LAUNCH) as sim:
        assert sim.csr_kernel == kernel
        if worm:
            T.titan_set_worm_actuation(sim.handle, np.arange(sy.n_springs), sy.act_amp, sy.act_phase, OMEGA, PERIOD)
        sim.step(STEPS)
        x, _, _ = sim.snapshot()
    xo, _ = oracle.run(sy, STEPS, act_mode=2, worm=(OMEGA, PERIOD)) if worm else oracle.run(sy, STEPS)
    assert np.abs(x - xo).max() <= 1e-4 * sy.spacing
