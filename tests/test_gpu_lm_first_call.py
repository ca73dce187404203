"""The first second-order call on a context allocates its buffers. It neither
waits for the caller's other streams nor disturbs a stream capture that another
thread has under way."""
import threading

import pytest

from paper_2602_21644_gb300 import synth

from gpu_common import to_dev
from test_gpu_splat import dags  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_first_call_beside_a_capture(dags):  # noqa: F811
    sc = synth.tiny_scene(0)
    cam = dags.Camera(*sc.camera.as_tuple())
    gauss, poses, targets = to_dev(sc, torch)
    pose = poses.reshape(-1)
    ctx, ref = (dags.Context(gauss.shape[0], cam.width, cam.height, 1) for _ in range(2))
    want, _ = ref.normal_equations(gauss, cam, pose, targets)
    normal = torch.empty_like(want)
    x = torch.ones(1024, device="cuda")
    torch.cuda.synchronize()
    graph, begun, done, failed = torch.cuda.CUDAGraph(), threading.Event(), threading.Event(), []

    def capture():
        try:
            with torch.cuda.graph(graph, capture_error_mode="thread_local"):
                x.add_(1.0)
                begun.set()
                done.wait(60)
                x.mul_(2.0)
        except Exception as e:   # noqa: BLE001  (the thread's error is the test's)
            failed.append(e)
        finally:
            begun.set()

    t = threading.Thread(target=capture)
    t.start()
    begun.wait(60)
    stream = torch.cuda.Stream()
    try:
        with torch.cuda.stream(stream):
            ctx.normal_equations(gauss, cam, pose, targets, normal=normal)
    finally:
        done.set()
        t.join()
    assert not failed, failed
    stream.synchronize()
    torch.testing.assert_close(normal, want, rtol=0, atol=0)
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 4.0).all()
    ctx.check()
