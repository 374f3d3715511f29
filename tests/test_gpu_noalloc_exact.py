"""The allocation-free step to the accuracy of its sums, on both sides of its one-launch form's limits: no
spring can be missing from it, a refused call writes nothing, and the call after that steps whole.

The regular atomic step evaluates the same springs in FP32 and adds them in another order.  Of a mass with d
springs the sum of forces then differs by at most 2 (d - 1) u sum|f| (u = 2^-24, d <= 26), its velocity by
that times dt / m and a few roundings of v itself, its position by dt times that and a few roundings of x."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300 import titan as T
from test_gpu_noalloc_sizes import _args

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _system(dims, springs, ground):
    rng = np.random.default_rng(sum(dims))
    pos, ends = inputs.lattice_points(*dims, 0.1), inputs.lattice_springs(*dims)[:springs]
    s, e = len(ends), ends.astype(np.int64)
    length = np.linalg.norm(pos[e[:, 1]] - pos[e[:, 0]], axis=1)
    rest = length * rng.uniform(0.97, 1.03, s)
    rest[-1] = 0.9 * length[-1]                       # the last spring pulls with 100 N or more
    sy = inputs.System(pos=pos - [0, 0, 1e-3], vel=rng.normal(0, 0.1, pos.shape), mass=np.full(len(pos), 0.1),
                       fixed=np.zeros(len(pos), np.uint8), ends=ends, k=np.full(s, 1e4), rest=rest,
                       damping=np.full(s, 1.0), dt=1e-4, ground=ground, spacing=0.1)
    d = sy.pos[e[:, 1]] - sy.pos[e[:, 0]]
    f = np.abs(1e4 * (length - rest)) + np.abs(((sy.vel[e[:, 1]] - sy.vel[e[:, 0]]) * d).sum(1) / length)
    total = np.bincount(e.ravel(), np.repeat(f, 2), len(pos)).max()
    dv = 2 * 25 * U * total * sy.dt / 0.1 + 8 * U * (np.abs(sy.vel).max() + total * sy.dt / 0.1)
    return sy, dv, sy.dt * dv + 4 * U * (np.abs(sy.pos).max() + 1e-3)


@pytest.mark.parametrize("dims,springs", [((2, 1, 1), 1), ((3, 3, 3), None), ((14, 14, 14), None), ((15, 15, 15), 32768),
                                          ((15, 15, 15), 32769), ((1, 64, 128), None), ((1, 64, 129), None)])
@pytest.mark.parametrize("ground", [False, True])
def test_every_spring_counts(dims, springs, ground):
    torch = pytest.importorskip("torch")
    sy, dv, dx = _system(dims, springs, ground)
    assert 100.0 * sy.dt / 0.1 > 1000 * dv            # a missing spring is far outside the tolerance
    with T.Sim(sy, accumulate=T.ACCUM_ATOMIC, order=T.ORDER_INPUT) as sim:
        sim.step(1)
        x, v, _ = sim.snapshot()
    a = _args(sy, torch)
    out = a[-2:]

    def whole():
        for o in out:
            o.fill_(float("nan"))
        T.titan_step_atomic_noalloc(*a)
        torch.cuda.synchronize()
        assert np.abs(out[0].cpu().numpy().astype(np.float64) - x).max() <= dx
        assert np.abs(out[1].cpu().numpy().astype(np.float64) - v).max() <= dv

    whole()
    good, last = a[5].clone(), sy.ends[-1].astype(np.int64)
    a[5][-1, 1] = a[5][-1, 0]
    T.titan_step_atomic_noalloc(*a)
    torch.cuda.synchronize()
    off = np.abs(out[1].cpu().numpy().astype(np.float64) - v).max(axis=1)
    assert off[last].min() > 100 * dv and np.delete(off, last).max(initial=0.0) <= dv       # that spring only
    a[5].copy_(good)
    for o in out:
        o.fill_(float("nan"))
    with pytest.raises(T.TitanError, match="skipped 1 spring"):
        T.titan_step_atomic_noalloc(*a)
    torch.cuda.synchronize()
    assert all(torch.isnan(o).all().item() for o in out)
    whole()
