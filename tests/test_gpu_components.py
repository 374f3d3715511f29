"""Bodies that overlap in space: one system of many robots steps with the halo kernel and to the
states each robot has on its own."""
import numpy as np
import pytest

import oracle
from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("actuated", [True, False])
def test_overlapping_robots_step_as_each_alone(actuated):
    rng = np.random.default_rng(5)
    robots = []
    for a, b, c in rng.integers(2, 10, (64, 3)).tolist() + [[1, 1, 2], [12, 12, 12]]:
        sy = inputs.actuated_box(a, b, c, rng)
        if not actuated:
            sy.act_amp = sy.act_phase = None
        robots.append(sy)
    u, mo, _ = T.union_system(robots)
    if not actuated:
        u.act_amp = u.act_phase = None
    with T.Sim(u, exec_mode=T.EXEC_LAUNCH) as sim:
        assert sim.csr_kernel == 4
        sim.step(60)
        x, _, _ = sim.snapshot()
    for r in (0, 17, 40, 63, 64, 65):
        xo, _ = oracle.run(robots[r], 60)
        assert np.abs(x[mo[r]:mo[r + 1]] - xo).max() <= 1e-4 * u.spacing
