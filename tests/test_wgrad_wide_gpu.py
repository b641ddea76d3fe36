"""The 3x3 weight gradient where cout is a multiple of 64 (64-wide CTAs of two kinds that share out the taps)."""
import numpy as np
import pytest
import torch

from paper_2409_01076_gb300 import nn as K

pytestmark = pytest.mark.gpu


def blocked(x):
    n, h, w, c = x.shape
    return x.view(n, h, w, c // 8, 8).permute(0, 3, 1, 2, 4).contiguous().view(-1)


def exact(x, dz):
    """(cout, 9, C) in 64 bits: sum over pixels of dz(p)[o] x(p + tap)[c]."""
    n, h, w, c = x.shape
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    d = dz.double().reshape(-1, dz.shape[3]).T
    return torch.stack([d @ xp[:, ky:ky + h, kx:kx + w].reshape(-1, c) for ky in range(3) for kx in range(3)], 1)


def gradient(n, h, w, C, cout, seed, extra=0, alpha=1.0):
    """(computed, exact, start) as (cout, 9, C); rows of the result `extra` floats apart from each other."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.nn.functional.silu(torch.randn(n, h, w, C, generator=g, device="cuda")).half()
    dz = (0.1 * torch.randn(n, h, w, cout, generator=g, device="cuda")).half()
    buf = torch.randn(cout, 9 * C + extra, generator=g, device="cuda")
    start = buf.clone()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    K.smrt_nn_conv3_wgrad_tma(blocked(x), (n, h, w, C), blocked(dz), cout, buf, alpha, err)
    assert int(err.item()) == 0
    assert torch.equal(buf[:, 9 * C:], start[:, 9 * C:])
    at = lambda t: t[:, :9 * C].double().view(cout, 9, C)  # noqa: E731
    return at(buf), at(start) + alpha * exact(x, dz), at(start)


@pytest.mark.parametrize("n,h,w,C,cout", [
    (1, 5, 3, 64, 64),            # one tile: the second kind of CTA has no share of the middle tap
    (2, 16, 8, 96, 128),          # two tiles, one CTA pair each
    (1, 33, 9, 136, 64),          # two input-channel blocks (the second of one plane), ragged tiles
    (2, 37, 21, 48, 192),         # three output blocks
    (3, 100, 77, 64, 64),         # 210 tiles over 76 pairs of CTAs: 2 or 3 each, the last CTA of a kind short
    (4, 64, 64, 384, 128),        # 128 tiles, 12 pairs: 11 each, every pipeline stage reused
    (8, 128, 96, 64, 64),         # 768 tiles: 11 each
    (1, 40, 40, 264, 1600),       # more channel blocks than half the SMs: one pair of CTAs takes every tile
])
def test_matches_64_bits(n, h, w, C, cout):
    got, want, start = gradient(n, h, w, C, cout, seed=n * h + C, extra=cout % 5, alpha=0.5)
    assert (got - want).abs().max() <= 1e-5 * want.abs().max()
    assert ((got - start) - (want - start)).norm() <= 2e-5 * (want - start).norm()


@pytest.mark.parametrize("n,h,w,C,cout", [(16, 128, 128, 64, 64), (16, 64, 64, 128, 128)])
def test_every_tap_sums_chains_of_one_length(n, h, w, C, cout):
    """A column's error grows with the tiles that its CTA adds one after another, so equal chains show equal errors
    (4,096 entries a tap: 2 % of spread; chains of 25 and 31 tiles differ by 24 %), and the middle tap, whose chains
    are half as long, a smaller one."""
    got, want, start = gradient(n, h, w, C, cout, seed=3)
    off = ((got - want).norm(dim=(0, 2)) / (want - start).norm(dim=(0, 2))).tolist()
    others = off[:4] + off[5:]
    assert max(others) <= 1.1 * min(others), off
    assert off[4] <= max(others), off
