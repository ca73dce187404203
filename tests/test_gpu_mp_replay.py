"""Everything that an MP update writes, from a replay of a captured graph: the
statistics follow from the records that this replay wrote, and the rest agrees
with a plain call."""
import numpy as np
import pytest

from test_gpu_mp_select import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [4_097, 300_001])
def test_replay_writes_statistics_and_labels(dags, n):  # noqa: F811
    # every Gaussian in view and none occluded (no occlusion test): all observed
    W, H, head = 96, 64, dags.MP_STATS_HEAD
    rng = np.random.default_rng(n)
    z = rng.uniform(1.0, 3.0, n)
    rec = np.zeros((n, 16), np.float32)
    rec[:, 0] = (rng.uniform(0, W - 1, n) - W / 2) * z / 60.0
    rec[:, 1] = (rng.uniform(0, H - 1, n) - H / 2) * z / 60.0
    rec[:, 2] = z
    rec[:, 11] = rng.uniform(0, 1, n)
    first = torch.from_numpy(rec).cuda()
    P = W * H
    image = torch.from_numpy(rng.uniform(0, 1, (8, P)).astype(np.float32)).cuda()
    tg = torch.from_numpy(rng.uniform(0.5, 1, (P, 4)).astype(np.float32)).cuda()
    inst = torch.from_numpy((rng.random(P) < 0.3).astype(np.uint8)).cuda()
    table = torch.tensor([[0.1, 0.05], [0.9, 0.8]], dtype=torch.float32, device="cuda")
    pose = torch.eye(4, dtype=torch.float64, device="cuda")[:3].reshape(12).contiguous()
    ctx = dags.Context(n, W, H, 1)
    cam = dags.Camera(60.0, 60.0, W / 2, H / 2, W, H)
    cfg = dags.default_mp_cfg(vis_tol=0.0, tau_floor=0.25)
    gauss, labels = first.clone(), torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    stats = ctx.mp_update(gauss, cam, pose, tg, image, inst, table, labels, cfg, True)
    torch.cuda.synchronize()
    want = stats.cpu().numpy().copy()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.mp_update(gauss, cam, pose, tg, image, inst, table, labels, cfg, True, stats=stats)
    for _ in range(2):
        gauss.copy_(first)
        labels.fill_(7)
        stats.fill_(-5.0)
        graph.replay()
        torch.cuda.synchronize()
        ctx.check()
        st, M = stats.cpu().numpy(), gauss[:, 11].cpu().numpy()
        assert st[5] == n
        assert st[2] == np.sort(M)[(n - 1) // 2] and st[0] == max(st[2], 0.25)
        np.testing.assert_array_equal(labels.cpu().numpy(), (M.astype(np.float64) > st[0]).astype(np.uint8))
        # the rest against the plain call. The region sums' float atomics may
        # round differently: a CTA's 256 residuals, each a few 2^-24 of the sum,
        # move means, and with them M_p, by under 1e-6; U_tilde divides by the
        # range of U, above a half here
        assert want[4] - want[3] > 0.5
        np.testing.assert_allclose(st[:head], want[:head], rtol=0, atol=4e-6)
        np.testing.assert_array_equal(st[head::4], want[head::4])          # the regions' counts
        np.testing.assert_allclose(st[head:], want[head:], rtol=4e-6, atol=0)
