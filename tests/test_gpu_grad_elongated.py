"""Gradients of splats that are long and thin off the image axes (discs seen
edge-on) against the FP64 oracle, where the adjoint accumulates moments (one kind
of gradient asked for): the gradient of such a splat's centre is what is left of
two terms that nearly cancel."""
import numpy as np
import pytest

from paper_2602_21644_gb300 import synth

from gpu_common import mask_flagged_targets, oracle_views
from test_gpu_splat import dags, run  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def edge_on_scene(seed, sigma, n=24, width=320, height=240):
    """n discs seen edge-on with a standard deviation of `sigma` pixels, turned by
    17 to 70 degrees either way in the image plane; smooth targets, so that the
    sums over a splat's pixels add up."""
    rng = np.random.default_rng(seed)
    f = 240.0
    z = rng.uniform(1.5, 2.5, n)
    means = np.stack([rng.uniform(-0.33, 0.33, n) * z * width / f, rng.uniform(-0.33, 0.33, n) * z * height / f, z], 1)
    length, thin = np.log(sigma * z / f), np.full(n, -9.0)
    half = rng.uniform(0.15, 0.6, n) * rng.choice([-1, 1], n)
    c, s, r = np.cos(half), np.sin(half), np.sqrt(0.5)
    # the normal (local z) turned into the image plane, then both turned in it
    quats, scales = np.stack([c * r, c * r, s * r, s * r], 1), np.stack([length, length, thin], 1)
    rec = synth.pack_records(means, rng.normal(1, 0.5, n), quats, scales, np.full(n, 0.1), rng.uniform(0.2, 0.8, (n, 3)))
    tg = np.zeros((1, width * height, 4), np.float32)
    yy, xx = np.mgrid[0:height, 0:width]
    for k in range(3):
        tg[0, :, k] = (0.5 + 0.5 * np.sin(xx / 37 + yy / 23 + k)).ravel()
    tg[0, :, 3] = (2 + np.sin(xx / 51 - yy / 33)).ravel()
    cam = synth.Camera(f, f, width / 2 + 0.3, height / 2 - 0.2, width, height)
    return synth.Scene(rec, cam, synth.identity_pose()[None], tg, np.zeros(n, bool))


# The standard deviation across a splat is sqrt(0.3) px (the dilation) and its
# aspect sigma / 0.55. Where the two terms cancel within a pixel, each is rounded
# to 2^-24 of up to `aspect` times what is left, in the offset, in the conic
# entries that the forward evaluates and in the terms themselves: 4 2^-24 aspect
# for their sum over the splats, which the sums' own rounding (a few 2^-24) does
# not reach. Terms that are first summed over a splat's pixels, hundreds of
# blocks, are off by the rounding of every one of these sums instead.
@pytest.mark.parametrize("sigma", [30.0, 60.0])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_edge_on_discs(dags, seed, sigma):  # noqa: F811
    sc, _ = mask_flagged_targets(edge_on_scene(seed, sigma))
    _, _, (ref,) = oracle_views(sc)
    bound = 4 * 2.0 ** -24 * sigma / np.sqrt(0.3)
    pose = run(dags, sc, flags=dags.GRAD_POSE)["gp"][0]
    assert np.linalg.norm(pose - ref["pose_grad"]) <= bound * np.linalg.norm(ref["pose_grad"])
    mean, want = run(dags, sc, flags=dags.GRAD_GAUSS)["gg"][:, :3], ref["grad"][:, :3]
    assert np.linalg.norm(mean - want) <= bound * np.linalg.norm(want)
