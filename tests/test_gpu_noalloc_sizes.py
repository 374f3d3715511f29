"""The allocation-free step on both sides of its one-launch form's limits (8,192 masses, 32,768
springs) against the regular atomic step, and skipped springs reported from each form."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu


def _args(sy, torch):
    f = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    p = T.titan_default_params()
    p.dt, p.ground, p.ground_k, p.mu = sy.dt, int(sy.ground), sy.ground_k, sy.mu
    return (sy.n_masses, f(sy.pos), f(sy.vel), f(1.0 / sy.mass), sy.n_springs,
            torch.tensor(sy.ends.astype(np.int32), device="cuda"), f(sy.k), f(sy.rest), 1.0, p,
            torch.empty(sy.n_masses, 3, device="cuda"), torch.empty(sy.n_masses, 3, device="cuda"))


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 1), (3, 3, 3), (14, 14, 14), (15, 15, 15), (1, 64, 128), (1, 64, 129)])
@pytest.mark.parametrize("ground", [False, True])
def test_step_matches_the_regular_atomic_step(dims, ground):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(sum(dims))
    pos, ends = inputs.lattice_points(*dims, 0.1), inputs.lattice_springs(*dims)
    s = len(ends)
    e = ends.astype(np.int64).reshape(-1, 2)
    length = np.linalg.norm(pos[e[:, 1]] - pos[e[:, 0]], axis=1)
    sy = inputs.System(pos=pos - [0, 0, 1e-3], vel=rng.normal(0, 0.1, pos.shape), mass=np.full(len(pos), 0.1),
                       fixed=np.zeros(len(pos), np.uint8), ends=ends, k=np.full(s, 1e4),
                       rest=length * rng.uniform(0.97, 1.03, s), damping=np.full(s, 1.0), dt=1e-4, ground=ground,
                       spacing=0.1)
    a = _args(sy, torch)
    T.titan_step_atomic_noalloc(*a)
    torch.cuda.synchronize()
    with T.Sim(sy, accumulate=T.ACCUM_ATOMIC, order=T.ORDER_INPUT) as sim:
        sim.step(1)
        x, v, _ = sim.snapshot()
    assert np.abs(a[-2].cpu().numpy() - x).max() <= 1e-4 * sy.spacing
    assert np.abs(a[-1].cpu().numpy() - v).max() <= 1e-1 * sy.spacing
    if s:                                             # a bad spring is reported by the next call, once
        good = a[5].clone()
        a[5][s - 1, 1] = a[5][s - 1, 0]
        T.titan_step_atomic_noalloc(*a)
        a[5].copy_(good)
        with pytest.raises(T.TitanError, match="skipped 1 spring"):
            T.titan_step_atomic_noalloc(*a)
        T.titan_step_atomic_noalloc(*a)
        torch.cuda.synchronize()
        assert np.abs(a[-2].cpu().numpy() - x).max() <= 1e-4 * sy.spacing
