"""A Gaussian whose colour has overflowed to infinity reaches only the pixels
that take it: the Jacobian render leaves the other pixels of their 8x4 blocks as
they are."""
import numpy as np
import pytest

from paper_2602_21644_gb300 import synth

from gpu_common import to_dev
from test_gpu_splat import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_infinite_colour_stays_in_its_pixels(dags):  # noqa: F811
    sc = synth.tiny_scene(0, n=300)
    cam = dags.Camera(*sc.camera.as_tuple())
    gauss, poses, targets = to_dev(sc, torch)
    ctx = dags.Context(gauss.shape[0], cam.width, cam.height, 1)
    order = np.argsort(sc.records[:, 8:11].max(1))
    out = []
    for value in (0.0, 1.0, np.inf):
        rgb = synth.record_rgb(sc.records)
        rgb[order[20]] = value                    # one of the smallest splats
        rec = synth.pack_records(sc.records[:, :3], sc.records[:, 3], sc.records[:, 4:8], sc.records[:, 8:11],
                                 sc.records[:, 11], rgb)
        image = torch.empty((1, 8, cam.height, cam.width), device="cuda")
        _, jac = ctx.normal_equations(torch.from_numpy(rec).cuda(), cam, poses.reshape(-1), targets, jac=True,
                                      image=image)
        torch.cuda.synchronize()
        out.append((image[0].cpu().numpy().reshape(8, -1), jac.cpu().numpy()))
    ctx.check()
    takes = (out[0][0][:3] != out[1][0][:3]).any(0)
    assert 0 < takes.sum() < 200
    # the pixels that take it are not confined to whole blocks
    blocks = takes.reshape(cam.height // 4, 4, cam.width // 8, 8).any((1, 3))
    assert takes.sum() < 32 * blocks.sum()
    assert np.isinf(out[2][0][:3, takes]).any()
    np.testing.assert_array_equal(out[2][0][:, ~takes], out[0][0][:, ~takes])
    np.testing.assert_array_equal(out[2][1][~takes], out[0][1][~takes])
