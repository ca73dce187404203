"""The normal equations against the FP64 oracle where the Jacobian render's
shapes can go wrong: one pixel block and less, image edges inside a block, more
tiles than one group of the FP64 sums and a remainder, lists shorter than a
staged chunk and longer than the sorted ones kept in shared memory; and the LM
loop, whose buckets and counters must be left as it found them, against itself."""
import numpy as np
import pytest

import oracle
from paper_2602_21644_gb300 import synth

from gpu_common import mask_flagged_targets
from test_gpu_splat import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def scene(n, width, height):
    sc, _ = mask_flagged_targets(synth.tiny_scene(3, n=n, width=width, height=height, f=0.75 * max(width, height)))
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.records, sc.poses.reshape(-1, 12)[0],
                                                                      sc.targets[0])]
    return sc, dags_camera(sc), *dev


def dags_camera(sc):
    from paper_2602_21644_gb300 import dags as d
    return d.Camera(*sc.camera.as_tuple())


@pytest.mark.parametrize("n,width,height", [(1, 16, 16), (40, 5, 3), (700, 33, 17), (2500, 112, 80), (3000, 129, 87),
                                            (5000, 24, 20)])
def test_normal_equations(dags, n, width, height):  # noqa: F811
    sc, cam, gauss, pose, target = scene(n, width, height)
    ctx = dags.Context(n, width, height)
    normal, jac = ctx.normal_equations(gauss, cam, pose, target, jac=True)
    torch.cuda.synchronize()
    ctx.check()
    ref = oracle.render_jac(oracle.params_from_records(sc.records), oracle.camera_vec(*sc.camera.as_tuple()),
                            sc.poses[0], sc.targets[0])
    H, g = oracle.unpack_normal(normal.cpu().numpy())
    # FP32 tangents and per-tile sums against FP64: the bounds of the LM parity
    # tests (terms relative to 2^-24 times the depth of the composited chain)
    assert abs(normal[0].item() - ref["L"]) <= 1e-5 * abs(ref["L"]) + 1e-12
    assert np.linalg.norm(H - ref["H"]) <= 1e-3 * np.linalg.norm(ref["H"]) + 1e-12
    assert np.linalg.norm(g - ref["g"]) <= 1e-3 * np.linalg.norm(ref["g"]) + 1e-12
    # a second call on the same workspace gives the same bits: every counter and
    # bucket is back at its start
    again, _ = ctx.normal_equations(gauss, cam, pose, target)
    assert torch.equal(again, normal)
    assert torch.isfinite(jac).all()


@pytest.mark.parametrize("n,width,height", [(700, 33, 17), (3000, 129, 87), (5000, 24, 20)])
def test_loop_repeats_and_matches_its_steps(dags, n, width, height):  # noqa: F811
    _, cam, gauss, pose, target = scene(n, width, height)
    ctx = dags.Context(n, width, height)
    states = []
    for use_graph in (True, False, True):
        p = pose.clone()
        states.append(ctx.track_lm(gauss, cam, p, target, iters=4, use_graph=use_graph).clone())
    # the loop's iterations are the general layout's linearisations and steps
    state = torch.empty(dags.LM_STATE, dtype=torch.float64, device="cuda")
    tried, best = torch.empty(12, dtype=torch.float64, device="cuda"), torch.empty(12, dtype=torch.float64, device="cuda")
    ctx.lm_init(pose, state, tried)
    for _ in range(4):
        normal, _ = ctx.normal_equations(gauss, cam, tried, target)
        ctx.lm_step(normal, state, tried, best)
    torch.cuda.synchronize()
    ctx.check()
    for s in states[1:] + [state]:
        assert torch.equal(s, states[0])
