"""The row-register form of the persistent kernel against one launch per step with
direct loads (equal bits) where it can go wrong: a CTA's last thread and one mass
more, every cluster size, masses copied to several CTAs, fixed masses without
springs that start with a velocity, rows that just fit and just do not, every
actuation, and launches that follow one another."""
import numpy as np
import pytest

from test_gpu_batch_rows import _box, _tangle

pytestmark = pytest.mark.gpu


def _with_strays(sy):
    """Three fixed masses and one free one that no spring touches."""
    sy.pos = np.concatenate([sy.pos, [[9.0, 9.0, 1.0 + k] for k in range(4)]])
    sy.vel = np.concatenate([sy.vel, np.ones((4, 3))])
    sy.mass = np.concatenate([sy.mass, np.full(4, 0.1)])
    sy.fixed = np.concatenate([sy.fixed, [1, 1, 1, 0]]).astype(np.uint8)
    return sy


def _star(n, seed):
    """One mass joined to n others: the widest row is n (rounded up to even)."""
    sy = _tangle(64, seed)
    keep = (sy.ends[:, 0] != 0) & (sy.ends[:, 1] != 0)
    ends = np.concatenate([sy.ends[keep][:150], np.stack([np.zeros(n), 1 + np.arange(n)], 1)]).astype(np.uint32)
    s = len(ends)
    sy.ends, sy.k, sy.rest, sy.damping = ends, np.full(s, 10.0), np.full(s, 0.4), np.full(s, 1.0)
    sy.act_amp, sy.act_phase = np.full(s, 0.1), np.linspace(0, 6, s)
    return sy


SYSTEMS = {"one_cta": lambda: _box(8, 8, 8, 1), "cube": lambda: _box(10, 10, 10, 2),
           "tangle_512": lambda: _tangle(512, 3), "tangle_513": lambda: _tangle(513, 4),
           "tangle_2000": lambda: _tangle(2000, 5), "strays": lambda: _with_strays(_box(7, 5, 4, 6)),
           "row_26": lambda: _star(26, 7), "row_28": lambda: _star(28, 8)}


@pytest.mark.parametrize("act", ["none", "sine", "worm"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_persistent_rows_equal_launches(name, act):
    from paper_1911_10274_gb300 import titan as T
    sy = SYSTEMS[name]()
    amp = sy.act_amp
    if act != "sine":
        sy.act_amp = None
    out = []
    for kw in (dict(exec_mode=T.EXEC_PERSISTENT), dict(exec_mode=T.EXEC_LAUNCH, kernel_variant=1)):
        with T.Sim(sy, **kw) as sim:
            if act == "worm":
                off = np.linspace(0.0, 0.9, sy.n_springs)
                T.titan_set_worm_actuation(sim.handle, np.arange(sy.n_springs), amp, off, 20.0, 0.01)
            sim.step(1).step(50).step(77)
            out.append(sim.snapshot())
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
