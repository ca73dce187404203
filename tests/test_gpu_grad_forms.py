"""The forms in which the adjoint accumulates 2D gradients (moments, or
gradients formed per pixel when both the Gaussians' and the twists' are asked
for) against the FP64 oracle and against each other, over image sizes that
divide into tiles and into warps' pixel blocks in every way, lists shorter and
longer than the 1,024 entries whose forward masks are recorded, and one or
several views."""
import numpy as np
import pytest

from paper_2602_21644_gb300 import synth

from gpu_common import GRAD_NORM, POSE_REL, compare_grads, mask_flagged_targets, oracle_views
from test_gpu_splat import dags, run  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,width,height,views", [
    (1, 16, 16, 1), (300, 33, 17, 1), (2000, 160, 120, 1), (1500, 8, 4, 1), (6000, 31, 19, 1), (900, 47, 65, 3)])
def test_forms_agree_with_oracle(dags, n, width, height, views):  # noqa: F811
    sc = synth.tiny_scene(5, n=n, width=width, height=height, f=0.75 * max(width, height))
    if views > 1:
        poses = np.stack([sc.poses[0]] * views)
        poses[:, 0, 3] += 0.05 * np.arange(views)
        sc = synth.Scene(sc.records, sc.camera, poses, np.concatenate([sc.targets] * views), sc.dynamic)
    sc, _ = mask_flagged_targets(sc)
    _, _, outs = oracle_views(sc)
    ref, mag = sum(o["grad"] for o in outs), sum(o["grad_mag"] for o in outs)
    both = run(dags, sc, flags=dags.GRAD_GAUSS | dags.GRAD_POSE)
    gauss = run(dags, sc, flags=dags.GRAD_GAUSS)
    pose = run(dags, sc, flags=dags.GRAD_POSE)
    for res in (both, gauss):
        for name, err in compare_grads(res["gg"], ref, mag=mag).items():
            assert err <= GRAD_NORM, (name, err)
    for res in (both, pose):
        for v, o in enumerate(outs):
            assert np.linalg.norm(res["gp"][v] - o["pose_grad"]) <= POSE_REL * np.linalg.norm(o["pose_grad"]) + 1e-12
    # the two forms differ by roundings of the same FP32 terms: per word a few
    # hundred additions of 2^-24 of the magnitudes, which cancel to at worst
    # a hundredth
    scale = np.linalg.norm(gauss["gg"])
    assert np.linalg.norm(both["gg"] - gauss["gg"]) <= 1e-5 * scale + 1e-30


def test_other_threshold_in_the_adjoint(dags):  # noqa: F811
    """An adjoint asked for another alpha_min than its forward's cannot rely on
    what the forward recorded: it tests every listed entry again."""
    sc = synth.tiny_scene(0)
    cam = dags.Camera(*sc.camera.as_tuple())
    gauss, poses, targets = (torch.from_numpy(np.ascontiguousarray(a)).cuda()
                             for a in (sc.records, sc.poses, sc.targets))
    ctx = dags.Context(gauss.shape[0], cam.width, cam.height)
    ctx.eval_counting(True)
    seen, grads = [], []
    for factor in (1.0, 1.0 + 1e-6, 0.25):
        rcfg = dags.default_raster_cfg()
        rcfg.alpha_min *= factor
        image, last, _ = ctx.forward(gauss, cam, poses, targets)
        gg, _ = ctx.backward(gauss, cam, poses, targets, image, last, dags.GRAD_GAUSS, rcfg=rcfg)
        torch.cuda.synchronize()
        seen.append(ctx.eval_read())
        grads.append(gg.double())
    ctx.check()
    # nearly the same threshold: the same contributions, found among more entries
    assert seen[1]["bwd_eval"] > seen[0]["bwd_eval"]
    assert seen[1]["bwd_contrib"] <= seen[0]["bwd_contrib"]
    assert (grads[1] - grads[0]).norm() <= 1e-4 * grads[0].norm()
    # a lower one takes contributions that no pixel of a warp took in the forward
    assert seen[2]["bwd_contrib"] > seen[0]["bwd_contrib"]
