"""Group centroids of the single-system and batch engines at the sizes where
the block-wide FP64 sum can go wrong (fewer masses than threads, a remainder,
an exact multiple), against numpy in FP64 on the same FP32 positions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _line(n, seed):
    from paper_1911_10274_gb300 import inputs
    rng = np.random.default_rng(seed)
    pos = rng.uniform(-1.0, 1.0, (n, 3))
    ends = np.stack([np.arange(n - 1), np.arange(1, n)], 1).astype(np.uint32)
    s = n - 1
    return inputs.System(pos=pos, vel=rng.normal(0.0, 0.1, (n, 3)), mass=np.full(n, 0.1), fixed=np.zeros(n, np.uint8),
                         ends=ends, k=np.full(s, 10.0), rest=np.full(s, 0.5), damping=np.full(s, 0.1), dt=1e-4)


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 640, 1500])
def test_centroid_of_every_block_remainder(n):
    import torch
    from paper_1911_10274_gb300 import titan as T
    sizes = [n, 3, 0, n + 1]
    sy = _line(sum(sizes), n)
    first = np.cumsum([0] + sizes)
    with T.Sim(sy) as sim:
        f = torch.tensor(first.astype(np.int32), device="cuda")
        out = torch.empty(len(sizes), 3, device="cuda")
        T.titan_group_centroids(sim.handle, f, None, out)
        sim.sync()
        p, _, _ = sim.snapshot()
    p = p.astype(np.float64)
    want = np.stack([p[a:b].mean(0) if b > a else np.zeros(3) for a, b in zip(first[:-1], first[1:])])
    # one FP32 rounding of an FP64 sum: half an ulp of values up to 1, the order immaterial
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=6.1e-8)
    robots = [_line(max(2, k), k) for k in sizes]
    with T.Batch(robots) as b:
        c = b.centroids()
        want = np.stack([b.read(r)[0].astype(np.float64).mean(0) for r in range(b.n)])
    np.testing.assert_allclose(c, want, rtol=0, atol=6.1e-8)
