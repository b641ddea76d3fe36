"""The SiLU backward over every shape of its pixels: one list of rows, large images, many tiny ones."""
import pytest
import torch

from paper_2409_01076_gb300 import nn as K

pytestmark = pytest.mark.gpu


def tensors(n, h, w, c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n, h, w, c, generator=g, device="cuda") for _ in range(2)]


def dz64(da, z):
    s = torch.sigmoid(z.double())
    return da.double() * s * (1 + z.double() * (1 - s))


def blocked(x):
    n, h, w, c = x.shape
    return x.view(n, h, w, c // 8, 8).permute(0, 3, 1, 2, 4).reshape(-1)


# images smaller than the grid's stride in pixels, equal to it (760 blocks x 256 threads / G) and larger
@pytest.mark.parametrize("n,h,w,c", [(70000, 1, 1, 8), (9000, 2, 6, 16), (3000, 8, 8, 32), (3, 128, 190, 64),
                                     (2, 152, 320, 64), (1, 300, 402, 8), (5, 40, 34, 24)])
@pytest.mark.parametrize("pooled", [False, True])
def test_blocked_backward_places_every_pixel(n, h, w, c, pooled):
    da, z = tensors(n, h, w, c, n + c)
    db = torch.zeros(c, device="cuda")
    dz, dzb = torch.empty_like(da), torch.empty(da.numel(), dtype=torch.float16, device="cuda")
    if pooled:
        if h % 2 or w % 2:
            pytest.skip("pooling needs even sides")
        dp = torch.randn(n, h // 2, w // 2, c, device="cuda")
        K.smrt_nn_bias_act_bwd_addpool_blocked(da, dp, z, 1, dz, db, dzb)
        da = da + 0.25 * dp.repeat_interleave(2, 1).repeat_interleave(2, 2)
    else:
        K.smrt_nn_bias_act_bwd_blocked(da, z, 1, dz, db, dzb)
    want = dz64(da, z)
    assert (dz.double() - want).abs().max() <= 4e-6 * want.abs().max()     # some float32 roundings of |dz| <= 6
    assert torch.equal(dzb, blocked(dz.half()))
    assert (db.double() - want.sum((0, 1, 2))).abs().max() <= 1e-5 * want.abs().sum((0, 1, 2)).max()


def fastest(f, reps=5):
    f()
    best = 1e30
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("n,h,w,c", [(16, 256, 256, 32), (16, 256, 256, 20), (400000, 2, 2, 16), (100000, 8, 8, 8)])
def test_backward_takes_no_more_than_a_few_forward_passes(n, h, w, c):
    """Both move three arrays of one size (the blocked backward 2.5): 400 times the forward's time was once lost
    to a loop over the grid's stride."""
    da, z = tensors(n, h, w, c, 1)
    out, out2 = torch.empty_like(da), torch.empty_like(da)
    bias, db = torch.zeros(c, device="cuda"), torch.zeros(c, device="cuda")
    fwd = fastest(lambda: K.smrt_nn_bias_act(da, bias, 1, out, out2))
    assert fastest(lambda: K.smrt_nn_bias_act_bwd(da, z, 1, out, db)) <= 5 * fwd
    if c % 8 == 0:
        half = torch.empty(da.numel(), dtype=torch.float16, device="cuda")
        assert fastest(lambda: K.smrt_nn_bias_act_bwd_blocked(da, z, 1, None, db, half)) <= 5 * fwd
