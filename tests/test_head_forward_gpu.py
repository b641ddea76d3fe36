"""The head's forward pass over every channel count: by pixel, or staged for whole groups of 32 channels."""
import pytest
import torch

from paper_2409_01076_gb300 import nn as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [4, 12, 20, 28, 32, 36, 60, 64])
@pytest.mark.parametrize("P,cout", [(1, 3), (255, 1), (257, 2), (70001, 3)])
def test_sums_in_channel_order(P, C, cout):
    g = torch.Generator(device="cuda").manual_seed(P + C)
    x, w = torch.randn(P, C, generator=g, device="cuda"), torch.randn(cout, C, generator=g, device="cuda")
    b = torch.randn(cout, generator=g, device="cuda")
    for bias in (b, None):
        y = torch.empty(P, cout, device="cuda")
        K.smrt_nn_conv1x1_small(x, w, bias, y)
        want = torch.zeros(P, cout, dtype=torch.float64, device="cuda") if bias is None else bias.double().expand(P, cout)
        for c in range(C):          # each step one fused multiply-add: exact in 64 bits, then one rounding to 32
            want = (want + x[:, c:c + 1].double() * w[:, c].double()).float().double()
        assert (y.double() - want).abs().max() <= 1e-6 * want.abs().max()


def fastest(f, reps=10):
    best = 1e30
    f()
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("C", [12, 20, 24, 28])
def test_near_the_copy_rate(C):
    """4 M pixels, three outputs, against a copy that moves as many bytes: 1.1 times its time by pixel, 1.5 to 2 staged."""
    P, cout = 1 << 22, 3
    x, w, y = torch.randn(P, C, device="cuda"), torch.randn(cout, C, device="cuda"), torch.empty(P, cout, device="cuda")
    half = torch.empty(P * (C + cout) // 2, device="cuda")
    copy = fastest(lambda: half.copy_(x.view(-1)[:half.numel()] if half.numel() <= x.numel() else half))
    assert fastest(lambda: K.smrt_nn_conv1x1_small(x, w, None, y)) <= 1.4 * copy
