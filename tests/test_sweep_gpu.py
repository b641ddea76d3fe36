"""Several updates in one pass over memory: smrt_step(h, n) against n calls of smrt_step(h, 1).

A call with n >= 2 on the two-buffer layout runs, in a float format, the sweep kernel (strips of 120
columns, segments of rows, 2 or 3 updates per pass), and on a small lattice in any format the tile kernel
(2 to 8 updates per launch); a call with n == 1 runs the one-update kernel.  All do the same operations on
the same values, so the fields are equal bit for bit.
"""
import numpy as np
import pytest

import paper_2409_01076_gb300 as S
from gpu_util import get_f, make
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# sweeps: the narrowest, one strip that a row fills, several, ragged ones, short and long segments
WIDE = [(9, 41001), (30, 12100), (128, 3000), (600, 601), (599, 640), (721, 720), (1201, 500), (2047, 331)]
# tiles: smallest, ragged, every plan of the rule
SMALL = [(8, 8), (9, 11), (64, 64), (65, 31), (123, 130), (241, 9), (361, 70), (300, 301), (470, 430)]
FLOWS = {"cavity": W.CAVITY, "periodic": W.ALL_PERIODIC, "couette": W.COUETTE,
         "walls_x": W.bc_flags(W.MOVING, W.WALL, W.PERIODIC, W.PERIODIC),
         "all_moving": W.bc_flags(W.MOVING, W.MOVING, W.MOVING, W.MOVING)}


def fields(nx, ny, bc, prec, kind, rounding, calls):
    h = make(nx, ny, 0.6, 0.1, bc, prec, "ab", kind, 0.9)
    S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, rounding)
    f0 = W.random_node_populations(nx * ny, 7 * nx + ny)
    S.smrt_set_f(h, np.ascontiguousarray(f0.T).reshape(9, ny, nx))
    for n in calls:
        S.smrt_step(h, n)
    f = get_f(h)
    t = S.smrt_time(h)
    S.smrt_destroy(h)
    return f, t


@pytest.mark.parametrize("size", WIDE + SMALL)
@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("prec,kind,rounding", [
    ("f64", "smrt", S.SMRT_ROUND_NEAREST), ("f64", "two_tau", S.SMRT_ROUND_NEAREST),
    ("f32", "smrt", S.SMRT_ROUND_NEAREST), ("f32", "srt", S.SMRT_ROUND_NEAREST),
    ("f32", "two_tau", S.SMRT_ROUND_NEAREST), ("f16", "smrt", S.SMRT_ROUND_NEAREST),
    ("f16", "two_tau", S.SMRT_ROUND_STOCHASTIC), ("bf16", "srt", S.SMRT_ROUND_NEAREST),
    ("bf16", "smrt", S.SMRT_ROUND_STOCHASTIC)])
def test_one_call_equals_single_updates(size, flow, prec, kind, rounding):
    one, _ = fields(*size, FLOWS[flow], prec, kind, rounding, [1] * 13)
    for calls in ([13], [2, 11], [4, 9]):       # passes of 3 and 2 updates in every order; whole and cut tiles
        got, t = fields(*size, FLOWS[flow], prec, kind, rounding, calls)
        assert t == 13
        assert np.array_equal(one, got), (calls, np.abs(one - got).max())


@pytest.mark.parametrize("size", [(4096, 4096), (4099, 4097), (4095, 4096)])    # the last one is below the rule
@pytest.mark.parametrize("flow", ["cavity", "periodic"])
def test_stochastic_rounding_at_the_size_that_takes_passes(size, flow):
    import torch
    nx, ny = size
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    rho = 1.0 + 0.01 * torch.sin(0.37 * x) * torch.cos(0.11 * y)
    u = torch.stack([0.05 * torch.sin(0.05 * x) * torch.cos(0.3 * y), 0.05 * torch.cos(0.2 * x + 0.07 * y)])
    out = []
    for calls in ([1] * 5, [5], [2, 3]):
        h = make(nx, ny, 0.6, 0.1, FLOWS[flow], "bf16", "ab", "smrt")
        S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, S.SMRT_ROUND_STOCHASTIC)
        S.smrt_init_macros(h, rho, u)
        for n in calls:
            S.smrt_step(h, n)
        r, v = torch.empty_like(rho), torch.empty_like(u)
        S.smrt_macros(h, r, v)
        S.smrt_sync(h)
        S.smrt_destroy(h)
        out.append((r, v))
    for r, v in out[1:]:
        assert torch.equal(r, out[0][0]) and torch.equal(v, out[0][1])


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("size", [(131, 70), (731, 710)])
@pytest.mark.parametrize("node", [(0, 0), (119, 5), (120, 31), (-1, -1)])
def test_divergence_is_reported(prec, size, node):
    """One node with rho < 0, in a corner, on either side of a strip boundary, in the last row."""
    nx, ny = size
    f = np.repeat(np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4), nx * ny).reshape(9, ny, nx).copy()
    f[:, node[1], node[0]] = -0.2
    h = make(nx, ny, 0.6, 0.1, W.CAVITY, prec)
    S.smrt_set_f(h, f)
    with pytest.raises(S.SmrtError) as e:
        S.smrt_step(h, 3)
    assert e.value.status == S.SMRT_ERR_DIVERGED
    S.smrt_destroy(h)


# many lattices of one narrow width take one update per launch, few or wider ones passes
@pytest.mark.parametrize("count,nx,ny", [(300, 8, 8), (300, 32, 19), (300, 64, 33), (300, 72, 33), (3, 64, 33), (1, 8, 8)])
@pytest.mark.parametrize("kind", ["smrt", "srt"])
def test_batch_of_one_width_equals_single_lattices(count, nx, ny, kind):
    tau = [0.6 + 0.3 * k / count for k in range(count)]
    b = S.smrt_batch_create([nx] * count, [ny] * count, tau, [0.08] * count, W.CAVITY, S.SMRT_PREC_F32, S.SMRT_LAYOUT_AB,
                            {"smrt": S.SMRT_COLLISION_SMRT, "srt": S.SMRT_COLLISION_SRT}[kind])
    for n in (1, 5, 8):
        S.smrt_batch_step(b, n)
    for k in {0, count // 2, count - 1}:
        h = make(nx, ny, tau[k], 0.08, W.CAVITY, "f32", "ab", kind)
        for _ in range(14):
            S.smrt_step(h, 1)
        f = np.empty((9, ny, nx))
        S.smrt_batch_get_f(b, k, f)
        assert np.array_equal(get_f(h), f), k
        S.smrt_destroy(h)
    S.smrt_batch_destroy(b)
