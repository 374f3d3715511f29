"""Group centroids where the number of threads per group changes (groups of fewer than 32, fewer than 128 and
more masses on average), with empty groups, groups of one, and one large group among many small ones: against
numpy in FP64 on the same FP32 positions, in both engines."""
import numpy as np
import pytest

from test_gpu_group_mean import _line

pytestmark = pytest.mark.gpu

SIZES = {"eights": [8] * 300, "ragged_small": [k % 7 for k in range(257)], "one_large": [3] * 200 + [1500] + [3] * 70,
         "two_large": [700, 1, 129] + [2] * 130 + [128], "warps": [40 + k % 60 for k in range(37)],
         "warps_one_large": [33] * 30 + [2000] + [0, 129, 128, 1], "just_32": [32] * 9, "just_31": [31] * 129 + [32],
         "just_128": [128] * 5, "just_127": [127, 128, 126, 127, 0], "blocks": [500, 0, 1, 129]}


@pytest.mark.parametrize("name", list(SIZES))
def test_sizes(name):
    import torch
    from paper_1911_10274_gb300 import titan as T
    sizes = SIZES[name]
    sy = _line(sum(sizes), len(sizes))
    first = np.cumsum([0] + sizes)
    origin = np.random.default_rng(1).uniform(-0.5, 0.5, (len(sizes), 3)).astype(np.float32)
    with T.Sim(sy) as sim:
        f = torch.tensor(first.astype(np.int32), device="cuda")
        o = torch.tensor(origin, device="cuda")
        out = torch.full((len(sizes), 3), float("nan"), device="cuda")
        T.titan_group_centroids(sim.handle, f, o, out)
        sim.sync()
        p, _, _ = sim.snapshot()
    p = p.astype(np.float64)
    want = np.stack([p[a:b].mean(0) - q if b > a else np.zeros(3) for a, b, q in zip(first[:-1], first[1:], origin)])
    # one FP32 rounding of an FP64 result: half an ulp of values up to 2, the order immaterial
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=1.22e-7)
    robots = [_line(max(2, k), k) for k in sizes[:140]]
    with T.Batch(robots) as b:
        c = b.centroids()
        want = np.stack([b.read(r)[0].astype(np.float64).mean(0) for r in range(b.n)])
    np.testing.assert_allclose(c, want, rtol=0, atol=6.1e-8)
