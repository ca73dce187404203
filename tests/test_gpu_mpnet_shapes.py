"""Training gradients of the MP network at the edges of its kernels' tiling:
strips of 128 pixels, one contiguous range of rows per
warpgroup (fewer rows than CTAs, ranges that cross strips and images), and one
context whose scratch serves frames that shrink and grow."""
import numpy as np
import pytest

from oracle import mpnet as N
from test_gpu_mpnet import group_errors, random_params, random_targets, to_vec, train_setup

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Each of dz3, dz2 and dz1 is rounded to BF16 (2^-9 relative), so a group's
# gradient is at most 3 x 2^-9 = 5.9e-3 off, whatever the number of pixels.
GRAD_REL = 1e-2


@pytest.fixture(scope="module")
def ctx():
    from paper_2602_21644_gb300 import build
    build.build()
    from paper_2602_21644_gb300 import dags
    return dags.Context(16, 16, 16, 1)


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (1, 1, 129), (1, 2, 127), (2, 33, 257), (1, 3, 128), (3, 5, 126),
                                   (5, 61, 131), (1, 240, 2), (2, 7, 384)])
def test_train_gradients_at_tile_edges(ctx, B, H, W):
    rng = np.random.default_rng(1000 * B + 10 * H + W)
    p = random_params(15)
    x = N.bf16_round(rng.uniform(0, 1, (B, H, W, 8)))
    target = random_targets(rng, (B, H, W))
    target[0, 0, 0] = 0.25                               # at least one pixel counts
    wt, master, m, v, feats, tg = train_setup(p, x, target)
    grad = torch.empty(10881, dtype=torch.float32, device="cuda")
    loss = ctx.mpnet_train_step(wt, master, m, v, 1, feats, tg, 0.0, grad=grad)
    torch.cuda.synchronize()
    ctx.check()
    L, g, _ = N.loss_and_grads(x, target, p)
    assert loss.item() == pytest.approx(L, rel=1e-4)
    errs = group_errors(grad.cpu().numpy().astype(np.float64), to_vec(g))
    assert max(errs.values()) <= GRAD_REL, errs
