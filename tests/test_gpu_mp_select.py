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


def test_update_replays_from_a_graph(dags):
    # the cooperative launch is captured like the others: a replay gives the
    # medians and labels of a plain call on the same records
    d = mp_scene(20_000, 31, 160, 120, seed=9)
    cam = dags.Camera(*d["cam"].as_tuple())
    P = cam.width * cam.height
    image = torch.zeros((8, P), dtype=torch.float32)
    image[0:3] = torch.from_numpy(d["rend"][:, 0:3].T.copy())
    image[3] = torch.from_numpy(d["rend"][:, 3].copy())
    image = image.cuda()
    rec = torch.from_numpy(d["rec"].copy()).cuda()
    tg, inst, table, lab0 = (torch.from_numpy(d[k].copy()).cuda() for k in ("obs", "inst", "table", "labels0"))
    pose = torch.from_numpy(np.ascontiguousarray(d["pose"])).cuda()
    ctx = dags.Context(rec.shape[0], cam.width, cam.height, 1)
    cfg = dags.default_mp_cfg()
    gauss, labels = rec.clone(), lab0.clone()
    stats = ctx.mp_update(gauss, cam, pose, tg, image, inst, table, labels, cfg, True)
    torch.cuda.synchronize()
    want = gauss[:, 11].clone(), labels.clone(), stats.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.mp_update(gauss, cam, pose, tg, image, inst, table, labels, cfg, True, stats=stats)
    for _ in range(2):
        gauss.copy_(rec)
        labels.copy_(lab0)
        stats.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ctx.check()
        # the region sums' float atomics may round differently between runs
        assert (gauss[:, 11] - want[0]).abs().max().item() <= 1e-6
        assert (labels != want[1]).sum().item() <= 2
        assert stats[5].item() == want[2][5].item()
