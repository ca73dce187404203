"""MP update: the compact list of observed Gaussians, the radix select with its
grid barriers, and both forms of the association's gather, at the sizes where
their tiling changes."""
import numpy as np
import pytest

from test_gpu_mp import check, mp_scene, run_both

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dags():
    from paper_2602_21644_gb300 import build
    build.build()
    from paper_2602_21644_gb300 import dags as d
    d.load()
    return d


@pytest.mark.parametrize("n", [1, 2, 255, 257, 1024, 1025, 155_649, 1_400_001])
def test_medians_and_labels_are_exact(dags, n):
    # every Gaussian in view and none occluded (no occlusion test), so the list
    # holds all of them: the medians and labels follow from the written records.
    # 1.4M entries are more than the threads' registers hold
    W, H = 64, 48
    rng = np.random.default_rng(n % 1000)
    z = rng.uniform(1.0, 3.0, n)
    u, v = rng.uniform(0, W - 1, n), rng.uniform(0, H - 1, n)
    rec = np.zeros((n, 16), np.float32)
    rec[:, 0], rec[:, 1], rec[:, 2] = (u - W / 2) * z / 60.0, (v - H / 2) * z / 60.0, z
    mp0 = rng.uniform(0, 1, n).astype(np.float32)
    mp0[rng.random(n) < 0.3] = 0.5                         # many equal values
    rec[:, 11] = mp0
    gauss = torch.from_numpy(rec).cuda()
    P = W * H
    image = torch.from_numpy(rng.uniform(0, 1, (8, P)).astype(np.float32)).cuda()
    tg = torch.from_numpy(rng.uniform(0.5, 1, (P, 4)).astype(np.float32)).cuda()
    inst = torch.from_numpy((rng.random(P) < 0.3).astype(np.uint8)).cuda()
    table = torch.tensor([[0.1, 0.05], [0.9, 0.8]], dtype=torch.float32, device="cuda")
    labels = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    pose = torch.eye(4, dtype=torch.float64, device="cuda")[:3].reshape(12).contiguous()
    ctx = dags.Context(n, W, H, 1)
    cam = dags.Camera(60.0, 60.0, W / 2, H / 2, W, H)
    stats = ctx.mp_update(gauss, cam, pose, tg, image, inst, table, labels,
                          dags.default_mp_cfg(vis_tol=0.0, tau_floor=0.25), True)
    torch.cuda.synchronize()
    ctx.check()
    st, M = stats.cpu().numpy(), gauss[:, 11].cpu().numpy()
    assert st[5] == n
    med = np.sort(M)[(n - 1) // 2]
    assert st[2] == med and st[0] == max(float(med), 0.25)
    np.testing.assert_array_equal(labels.cpu().numpy(), (M.astype(np.float64) > st[0]).astype(np.uint8))


@pytest.mark.parametrize("r_s,scales", [(0.5, 1), (1.5, 2), (2.5, 1), (3.0, 3)])
def test_association_radii(dags, r_s, scales):
    # up to 2 the gather's rows are unrolled, above they are loops
    d = mp_scene(30_000, 31, 253, 189, seed=8)
    gpu, ref = run_both(dags, d, {"r_s": r_s, "scales": scales})
    check(gpu, ref, d["table"].shape[0])
