"""3x3 convolutions over every tile shape and pipeline depth that the launch rule chooses on 152 SMs, and over outputs
of every alignment: direct products in 64 bits, and the fused epilogues against the separate kernels bit for bit."""
import pytest
import torch

from paper_2409_01076_gb300 import nn as K

pytestmark = pytest.mark.gpu

SHAPES = [
    (4, 64, 64, 64, 128),       # 128 single tiles of 128 channels (77 to 152: one per SM, four stages)
    (3, 100, 56, 80, 256),      # 294 tiles of 128 channels
    (16, 64, 40, 96, 128),      # 320: stacked pairs
    (8, 40, 40, 64, 64),        # 120 tiles of 64 channels (four stages over 4 chunks)
    (16, 40, 40, 64, 64),       # 240 (two stages)
    (16, 100, 60, 96, 64),      # 896 (one stage)
    (16, 100, 60, 48, 40),      # the same, part of the channels
    (8, 64, 64, 96, 32),        # 256 tiles of 32 channels (two stages over 6 chunks)
    (1, 40, 24, 64, 256),       # few tiles: 32-wide ones of the 128-wide packing
    (1, 33, 17, 48, 64),        # ... of the 64-wide packing, ragged
    (1, 20, 12, 32, 200),       # ... the last of them without channels
]


def blocked(x):
    n, h, w, c = x.shape
    return x.view(n, h, w, c // 8, 8).permute(0, 3, 1, 2, 4).contiguous().view(-1)


def operands(n, h, w, C, cout):
    g = torch.Generator(device="cuda").manual_seed(h * w + C + cout)
    x = torch.randn(n, h, w, C, generator=g, device="cuda").half()
    wt = torch.randn(cout, 9 * C, generator=g, device="cuda").half()
    wp = torch.empty(K.smrt_nn_pack3_halves(cout, C), dtype=torch.float16, device="cuda")
    K.smrt_nn_pack3(wt, C, wp)
    return g, x, blocked(x), wt, wp, torch.zeros(1, dtype=torch.int32, device="cuda")


def product(x, wt):
    n, h, w, C = x.shape
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    out = 0
    for t in range(9):
        out = out + xp[:, t // 3:t // 3 + h, t % 3:t % 3 + w].reshape(-1, C) @ wt[:, t * C:(t + 1) * C].double().T
    return out


def at_offset(rows, cols, floats, seed=None):
    """A contiguous (rows, cols) float32 tensor that starts `floats` floats behind a 256-byte boundary."""
    buf = torch.full((rows * cols + floats,), float("nan"), device="cuda")
    return buf[floats:].view(rows, cols)


@pytest.mark.parametrize("n,h,w,C,cout", SHAPES)
def test_forward_matches_64_bits_at_every_alignment(n, h, w, C, cout):
    _, x, xb, wt, wp, err = operands(n, h, w, C, cout)
    want = product(x, wt)
    ys = []
    for floats in (0, 4, 1):                    # 32-, 16- and 4-byte stores
        y = at_offset(n * h * w, cout, floats)
        K.smrt_nn_conv3_tma(xb, (n, h, w, C), wp, y, cout, 1.0, 0.0, err)
        ys.append(y)
    assert int(err.item()) == 0
    assert (ys[0] - want).abs().max() <= 1e-5 * want.abs().max()
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])
    # onto y itself, in rows wider than the channels
    y0 = torch.randn(n * h * w, cout + 3, device="cuda")
    y = y0.clone()
    K.smrt_nn_conv3_tma(xb, (n, h, w, C), wp, y, cout, 0.5, 2.0, err)
    assert torch.equal(y[:, cout:], y0[:, cout:])
    assert (y[:, :cout] - (0.5 * want + 2.0 * y0[:, :cout].double())).abs().max() <= 1e-5 * want.abs().max()


@pytest.mark.parametrize("n,h,w,C,cout", SHAPES)
@pytest.mark.parametrize("floats", [0, 4])
def test_bias_and_silu_in_the_epilogue(n, h, w, C, cout, floats):
    g, x, xb, wt, wp, err = operands(n, h, w, C, cout)
    rows = n * h * w
    bias = torch.randn(cout, generator=g, device="cuda")
    y, z1, a1 = (torch.empty(n, h, w, cout, device="cuda") for _ in range(3))
    half1, half2 = (torch.empty(rows * cout, dtype=torch.float16, device="cuda") for _ in range(2))
    K.smrt_nn_conv3_tma(xb, (n, h, w, C), wp, y, cout, 1.0, 0.0, err)
    K.smrt_nn_bias_act_blocked(y, bias, 1, z1, a1, half1)
    z2, a2 = at_offset(rows, cout, floats), at_offset(rows, cout, floats)
    K.smrt_nn_conv3_tma_bias_act(xb, (n, h, w, C), wp, cout, bias, 1, z2, a2, half2, err)
    assert int(err.item()) == 0
    assert torch.equal(z1.view_as(z2), z2) and torch.equal(a1.view_as(a2), a2) and torch.equal(half1, half2)


@pytest.mark.parametrize("n,h,w,C,cout", SHAPES)
@pytest.mark.parametrize("floats", [0, 4])
def test_silu_backward_in_the_epilogue(n, h, w, C, cout, floats):
    g, x, xb, wt, wp, err = operands(n, h, w, C, cout)
    rows = n * h * w
    z = at_offset(rows, cout, floats)
    z.copy_(torch.randn(rows, cout, generator=g, device="cuda"))
    d, dz1 = (torch.empty(n, h, w, cout, device="cuda") for _ in range(2))
    half1, half2 = (torch.empty(rows * cout, dtype=torch.float16, device="cuda") for _ in range(2))
    db1, db2 = torch.zeros(cout, device="cuda"), torch.zeros(cout, device="cuda")
    K.smrt_nn_conv3_tma(xb, (n, h, w, C), wp, d, cout, 1.0, 0.0, err)
    K.smrt_nn_bias_act_bwd_blocked(d, z.clone().view_as(d), 1, dz1, db1, half1)
    dz2 = at_offset(rows, cout, floats)
    K.smrt_nn_conv3_tma_act_bwd(xb, (n, h, w, C), wp, cout, z, 1, dz2, db2, half2, err)
    assert int(err.item()) == 0
    assert torch.equal(dz1.view_as(dz2), dz2) and torch.equal(half1, half2)
    assert (db1 - db2).abs().max() <= 1e-5 * dz1.abs().sum((0, 1, 2)).max()
