"""A tracking loop overwrites the workspace of the last forward, also when it
replays a graph that an earlier call captured: no backward and no reading of
that forward's lists may follow."""
import pytest

from paper_2602_21644_gb300 import synth

from gpu_common import to_dev
from test_gpu_splat import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("loop", ["first_order", "second_order"])
@pytest.mark.parametrize("iters", [1, 12])
def test_no_backward_after_a_replay(dags, loop, iters):  # noqa: F811
    sc = synth.tiny_scene(0)
    cam = dags.Camera(*sc.camera.as_tuple())
    gauss, poses, targets = to_dev(sc, torch)
    ctx = dags.Context(gauss.shape[0], cam.width, cam.height, 1)
    pose = poses.reshape(-1).clone()
    image = torch.empty((1, 8, cam.height, cam.width), device="cuda")
    last = torch.empty((1, cam.height, cam.width), dtype=torch.int32, device="cuda")
    loss, twist, adam = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (1, 6, 13))
    state = torch.empty(dags.LM_STATE, dtype=torch.float64, device="cuda")

    def track(k):
        if loop == "first_order":
            ctx.track(gauss, cam, pose, targets, k, adam, image, last, loss, twist)
        else:
            ctx.track_lm(gauss, cam, pose, targets, k, state=state)

    track(iters)                                  # captures
    im, la, _ = ctx.forward(gauss, cam, poses, targets)
    track(0)                                      # replays nothing: the forward still stands
    ctx.backward(gauss, cam, poses, targets, im, la, dags.GRAD_POSE)
    im, la, _ = ctx.forward(gauss, cam, poses, targets)
    track(iters)                                  # replays
    with pytest.raises(dags.DagsError) as e:
        ctx.backward(gauss, cam, poses, targets, im, la, dags.GRAD_POSE)
    assert e.value.code == -6                     # DAGS_E_ORDER
    with pytest.raises(dags.DagsError):
        ctx.backward_upstream(gauss, cam, poses, im, la, torch.zeros((1, 6, cam.height, cam.width), device="cuda"))
    with pytest.raises(dags.DagsError):
        ctx.copy_bins(1, cam)
    im, la, _ = ctx.forward(gauss, cam, poses, targets)
    ctx.backward(gauss, cam, poses, targets, im, la, dags.GRAD_POSE)
    torch.cuda.synchronize()
    ctx.check()
