"""The MP update beside its failure path: the grid barrier that gives up (the
self-test waits for an arrival that nothing makes) leaves the context usable."""
import numpy as np
import pytest

from test_gpu_mp import mp_scene
from test_gpu_mp_select import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("spins", [0, 1000])
def test_update_after_a_barrier_gave_up(dags, spins):  # noqa: F811
    d = mp_scene(3_000, 31, 64, 48, seed=11)
    cam = dags.Camera(*d["cam"].as_tuple())
    image = torch.zeros((8, cam.width * cam.height), dtype=torch.float32)
    image[0:3] = torch.from_numpy(d["rend"][:, 0:3].T.copy())
    image[3] = torch.from_numpy(d["rend"][:, 3].copy())
    rec, tg, inst, table, lab0 = (torch.from_numpy(d[k].copy()).cuda()
                                  for k in ("rec", "obs", "inst", "table", "labels0"))
    pose = torch.from_numpy(np.ascontiguousarray(d["pose"])).cuda()
    out = []
    for give_up in (False, True):
        ctx = dags.Context(rec.shape[0], cam.width, cam.height, 1)
        if give_up:
            ctx.selftest_timeout(spins)
            with pytest.raises(dags.DagsError) as e:
                ctx.check()
            assert e.value.code == -4             # DAGS_E_TIMEOUT
        gauss, labels = rec.clone(), lab0.clone()
        stats = ctx.mp_update(gauss, cam, pose, tg, image.cuda(), inst, table, labels, dags.default_mp_cfg(), True)
        torch.cuda.synchronize()
        ctx.check()
        out.append((gauss[:, 11], labels, stats))
    # (the region sums' float atomics may round differently between runs)
    assert (out[0][0] - out[1][0]).abs().max().item() <= 1e-6
    assert (out[0][1] != out[1][1]).sum().item() <= 2
    assert out[0][2][5].item() == out[1][2][5].item() > 0
