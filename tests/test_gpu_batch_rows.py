"""The row-register form of the batch kernel against the looped form with one
thread per mass (the same rows summed in the same order: equal bits) at the
sizes where its planning can go wrong: one warp, a CTA's last slot, one mass
more, every cluster size, masses copied to several CTAs' halos, short and
empty rows, fixed masses, unactuated systems; and against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _box(a, b, c, seed, act=True):
    from paper_1911_10274_gb300 import inputs
    rng = np.random.default_rng(seed)
    sy = inputs.actuated_box(a, b, c, rng)
    sy.vel[:] = rng.normal(0.0, 0.1, sy.vel.shape)
    sy.fixed[:2] = 1
    if not act:
        sy.act_amp = None
    return sy


def _tangle(n, seed, act=True):
    """Masses joined at random (at most 26 springs each): their neighbours lie in every CTA."""
    from paper_1911_10274_gb300 import inputs
    rng = np.random.default_rng(seed)
    deg, seen = np.zeros(n, int), set()
    for i, j in rng.integers(0, n, (12 * n, 2)):
        key = (min(i, j), max(i, j))
        if i != j and key not in seen and deg[i] < 26 and deg[j] < 26:
            seen.add(key)
            deg[i] += 1
            deg[j] += 1
    ends = np.array(sorted(seen), np.uint32)
    s = len(ends)
    pos = rng.uniform(0.0, 1.0, (n, 3))
    sy = inputs.System(pos=pos, vel=rng.normal(0.0, 0.1, (n, 3)), mass=np.full(n, 0.1), fixed=np.zeros(n, np.uint8),
                       ends=ends, k=rng.uniform(5.0, 20.0, s), rest=rng.uniform(0.1, 0.9, s), damping=np.full(s, 1.0),
                       dt=1e-4, ground=True)
    if act:
        sy.act_amp, sy.act_phase, sy.act_freq = rng.uniform(0, 0.2, s), rng.uniform(0, 6.0, s), 2.0
    return sy


CASES = {"one_warp": lambda act: [_box(4, 4, 2, 1, act), _box(3, 3, 3, 2, act)],
         "last_slot_and_one_more": lambda act: [_box(8, 8, 6, 3, act), _box(11, 7, 5, 4, act)],
         "clusters_2_3_4": lambda act: [_box(12, 8, 4, 5, act), _box(12, 8, 8, 6, act), _box(11, 11, 11, 7, act)],
         "clusters_5_6_8": lambda act: [_box(12, 12, 12, 8, act), _box(14, 13, 12, 9, act), _box(14, 14, 13, 10, act)],
         "many_copies": lambda act: [_tangle(1100, 11, act), _tangle(700, 12, act)]}


@pytest.mark.parametrize("act", [True, False], ids=["actuated", "plain"])
@pytest.mark.parametrize("name", list(CASES))
def test_rows_form_equals_looped_form(name, act):
    import oracle
    from paper_1911_10274_gb300 import titan as T
    robots = CASES[name](act)
    with T.Batch(robots) as rows, T.Batch(robots) as loop:
        for g in range(len(loop.groups())):
            loop.configure(g, 512, 1)
        for b in (rows, loop):
            b.rollout(37).rollout(64)
        for r, sy in enumerate(robots):
            x, v = rows.read(r)
            y, w = loop.read(r)
            assert np.array_equal(x, y) and np.array_equal(v, w), (name, r)
            xo, _ = oracle.run(sy, 101)
            assert np.abs(x.astype(np.float64) - xo).max() <= 1e-4 * 0.1, (name, r)
