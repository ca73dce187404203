"""Epipolar verification: the group offsets (an atomic cursor over CTAs of 1024
counts) at the sizes where the tiling changes, against the medians of the
distances that the call itself returns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dags():
    from paper_2602_21644_gb300 import build
    build.build()
    from paper_2602_21644_gb300 import dags as d
    d.load()
    return d


@pytest.mark.parametrize("n,m", [(1, 1), (1, 300), (5, 257), (1024, 4000), (1025, 3), (70_001, 50_000)])
def test_medians_follow_from_the_distances(dags, n, m):
    rng = np.random.default_rng(n + m)
    gid = rng.integers(0, n, m).astype(np.int32)
    pose = np.eye(4)[:3]
    pose_j = pose.copy()
    pose_j[:, 3] = (0.1, -0.05, 0.02)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    p1 = rng.uniform(0, 60, (m, 2)).astype(np.float32)
    p2 = (p1 + rng.normal(0, 1, (m, 2))).astype(np.float32)
    gauss = torch.zeros((n, 16), dtype=torch.float32, device="cuda")
    gauss[:, 11] = 0.9
    labels = torch.ones(n, dtype=torch.uint8, device="cuda")
    ctx = dags.Context(n, 64, 64, 1)
    cam = dags.Camera(60.0, 60.0, 32.0, 32.0, 64, 64)
    d, dbar = ctx.epipolar_verify(cam, t(pose.reshape(12)), t(pose_j.reshape(12)), t(p1), t(p2), t(gid), gauss, labels)
    torch.cuda.synchronize()
    ctx.check()
    d, dbar = d.cpu().numpy(), dbar.cpu().numpy()
    order = np.lexsort((d, gid))
    start = np.searchsorted(gid[order], np.arange(n))
    count = np.bincount(gid, minlength=n)
    want = np.full(n, np.nan, np.float32)
    has = count > 0
    want[has] = d[order][start[has] + (count[has] - 1) // 2]     # the lower median, an element of the group
    np.testing.assert_array_equal(dbar, want)
