"""Rollouts launched directly, captured on a count's second use and replayed, in every order: the bits of one
rollout of all their steps."""
import numpy as np
import pytest

from paper_1911_10274_gb300 import titan as T
from test_gpu_batch_rows import _box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act", [True, False], ids=["actuated", "plain"])
def test_every_sequence_of_rollouts(act):
    robots = [_box(4, 4, 2, 1, act), _box(8, 8, 6, 3, act), _box(11, 7, 5, 4, act), _box(12, 12, 12, 5, act)]
    with T.Batch(robots) as b, T.Batch(robots) as one:
        for seq in ([5, 5, 5, 5, 5], [3, 5, 3, 5, 3, 5], [7], [7], [7], [7, 7], [5] * 9, [1, 1, 1, 2, 2, 2, 2]):
            b.reset()
            for k in seq:
                b.rollout(k)
            one.reset()
            one.rollout(sum(seq))
            for r in range(len(robots)):
                x, y = b.read(r), one.read(r)
                assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1]), (seq, r)
        b.configure(0, 256, 1)                        # a new shape drops what was captured
        for _ in range(4):
            b.reset()
            b.rollout(7)
        one.reset()
        one.rollout(7)
        for r in range(len(robots)):
            assert np.array_equal(b.read(r)[0], one.read(r)[0])
