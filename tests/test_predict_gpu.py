"""UNet.predict: a shape that repeats is recorded and replayed; the replayed outputs equal the eager ones."""
import pytest
import torch

from paper_2409_01076_gb300 import unet as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", [(1, 64, 64), (3, 40, 72)])
def test_repeated_predictions_equal_the_forward_pass(n, h, w):
    net = U.UNet(base=32, seed=3)
    g = torch.Generator(device="cuda").manual_seed(5)
    for k in range(5):                      # eager, recorded, replayed; other inputs each time
        x = torch.rand(n, h, w, 3, generator=g, device="cuda")
        want = net.forward(x, None)
        got = net.predict(x)
        assert torch.equal(got, want)
        if k == 3:                          # a replay reads the current parameters
            net.load_numpy({"enc1a.w": 0.5 * net.to_numpy()["enc1a.w"]})
    kept = got.clone()
    net.predict(torch.zeros_like(x))        # a later call leaves an earlier result alone
    assert torch.equal(got, kept)


def test_shapes_take_turns():
    net = U.UNet(base=32, seed=4)
    xs = [torch.rand(1, 32, 32, 3, device="cuda"), torch.rand(2, 48, 64, 3, device="cuda")]
    for x in [xs[0], xs[0], xs[0], xs[1], xs[1], xs[0], xs[1], xs[0], xs[0]]:
        assert torch.equal(net.predict(x), net.forward(x, None))
