"""A pixel's transmittance is its own: entries that other pixels of its 8x4 block
take, hundreds of them in front of and behind it, leave the gradient of the one
Gaussian that it takes alone, bit for bit."""
import numpy as np
import pytest

from paper_2602_21644_gb300 import synth

from test_gpu_splat import dags, run  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("flags", ["GRAD_GAUSS", "BOTH"])
def test_entries_of_other_pixels_leave_a_gradient_alone(dags, flags):  # noqa: F811
    rng = np.random.default_rng(3)
    n, f, width, height = 801, 40.0, 16, 16
    # Gaussian 0 around pixel (1, 1), the others around (6, 1): at most 0.56 px
    # wide, so that none reaches alpha = 1 / 255 within 2 px of the other's
    z = np.concatenate([[2.0], rng.uniform(1.0, 3.0, n - 1)])
    px = np.concatenate([[1.0], np.full(n - 1, 6.0)])
    means = np.stack([(px - 8) * z / f, (1 - 8.0) * z / f, z], 1)
    logit = np.concatenate([[1.0], np.full(n - 1, -4.5)])
    rec = synth.pack_records(means, logit, np.tile([1.0, 0, 0, 0], (n, 1)), np.full((n, 3), -8.0), np.full(n, 0.1),
                             rng.uniform(0.2, 0.8, (n, 3)))
    tg = np.zeros((1, width * height, 4), np.float32)
    tg[0, :, :3] = rng.uniform(0, 1, (width * height, 3))
    tg[0, :, 3] = rng.uniform(1, 4, width * height)
    cam = synth.Camera(f, f, 8.0, 8.0, width, height)
    bits = dags.GRAD_GAUSS | (dags.GRAD_POSE if flags == "BOTH" else 0)
    grads, taken = [], []
    for records in (rec[:1], rec):
        res = run(dags, synth.Scene(records, cam, synth.identity_pose()[None], tg, np.zeros(len(records), bool)), bits)
        grads.append(res["gg"][0])
        taken.append(res["last"][0].cpu().numpy())
    assert taken[0][1, 1] > 0 and taken[0][:, 3:].max() == 0 and taken[1][1, 6] > 700
    assert np.abs(grads[0]).max() > 0
    np.testing.assert_array_equal(grads[0], grads[1])
