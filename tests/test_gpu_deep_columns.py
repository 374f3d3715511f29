"""Both forms of the halo and box step kernels - two columns in flight, and the
deep form of grids of at most two CTAs per SM - on systems just below and just
above that line, with every option the kernels are compiled for: equal bits to
the direct-load kernel, which has no such forms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _system(shape, ground, act, per_spring):
    from paper_1911_10274_gb300 import inputs
    rng = np.random.default_rng(7)
    if isinstance(shape, tuple):
        sy = inputs.actuated_box(*shape, rng)
    else:
        sy = inputs.random_mesh(n_points=shape, knn=5, seed=3, k=50.0)
        sy.act_amp, sy.act_phase, sy.act_freq = rng.uniform(0, 0.2, sy.n_springs), rng.uniform(0, 6, sy.n_springs), 2.0
    sy.vel[:] = rng.normal(0.0, 0.1, sy.vel.shape)
    sy.pos[:, 2] -= 1e-4
    sy.ground = ground
    if not act:
        sy.act_amp = None
    if per_spring:
        sy.damping = rng.uniform(0.5, 1.5, sy.n_springs)
    return sy


# 8 x 8 x 4 cells a CTA: 304 and 305 CTAs, ragged; 256 points a CTA
@pytest.mark.parametrize("shape", [(8 * 76, 8, 16), (8 * 61, 8, 20), (30, 29, 31), 304 * 256, 304 * 256 + 1, 777],
                         ids=str)
@pytest.mark.parametrize("ground,act,per_spring", [(False, False, False), (True, True, False), (True, False, True),
                                                    (False, True, True)])
def test_halo_and_box_forms_equal_direct_loads(shape, ground, act, per_spring):
    from paper_1911_10274_gb300 import titan as T
    sy = _system(shape, ground, act, per_spring)
    out = []
    for variant in (1, 4, 6) if isinstance(shape, tuple) else (1, 4):
        with T.Sim(sy, exec_mode=T.EXEC_LAUNCH, kernel_variant=variant) as sim:
            sim.step(7)
            out.append(sim.snapshot())
    for o in out[1:]:
        assert np.array_equal(out[0][0], o[0]) and np.array_equal(out[0][1], o[1])
