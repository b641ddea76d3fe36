"""Several updates in one pass over memory: smrt_step(h, n) against n calls of smrt_step(h, 1).

A call with n >= 2 on the two-buffer layout in a float format runs the sweep kernel (strips of 120
columns, segments of rows, 2 or 3 updates per pass); a call with n == 1 runs the one-update kernel.
Both do the same operations on the same values, so the fields are equal bit for bit.
"""
import numpy as np
import pytest

import paper_2409_01076_gb300 as S
from gpu_util import get_f, make
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# smallest; around one strip and its shared columns; ragged; several strips; short and long segments
SIZES = [(8, 8), (9, 11), (31, 9), (119, 8), (120, 66), (121, 33), (123, 130), (124, 17), (125, 65), (128, 128),
         (239, 40), (241, 9), (244, 100), (361, 70)]
FLOWS = {"cavity": W.CAVITY, "periodic": W.ALL_PERIODIC, "couette": W.COUETTE,
         "walls_x": W.bc_flags(W.MOVING, W.WALL, W.PERIODIC, W.PERIODIC),
         "all_moving": W.bc_flags(W.MOVING, W.MOVING, W.MOVING, W.MOVING)}


def fields(nx, ny, bc, prec, kind, rounding, calls):
    h = make(nx, ny, 0.6, 0.1, bc, prec, "ab", kind, 0.9)
    S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, rounding)
    S.smrt_set_f(h, W.random_populations(nx, ny, 7 * nx + ny))
    for n in calls:
        S.smrt_step(h, n)
    f = get_f(h)
    t = S.smrt_time(h)
    S.smrt_destroy(h)
    return f, t


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("prec,kind,rounding", [
    ("f32", "smrt", S.SMRT_ROUND_NEAREST), ("f32", "srt", S.SMRT_ROUND_NEAREST),
    ("f32", "two_tau", S.SMRT_ROUND_NEAREST), ("f16", "smrt", S.SMRT_ROUND_NEAREST),
    ("f16", "two_tau", S.SMRT_ROUND_STOCHASTIC), ("bf16", "srt", S.SMRT_ROUND_NEAREST),
    ("bf16", "smrt", S.SMRT_ROUND_STOCHASTIC)])
def test_one_call_equals_single_updates(size, flow, prec, kind, rounding):
    one, _ = fields(*size, FLOWS[flow], prec, kind, rounding, [1] * 7)
    for calls in ([7], [2, 5], [4, 3]):         # passes of 3 and 2 updates in every order
        got, t = fields(*size, FLOWS[flow], prec, kind, rounding, calls)
        assert t == 7
        assert np.array_equal(one, got), (calls, np.abs(one - got).max())


@pytest.mark.parametrize("node", [(0, 0), (119, 5), (120, 31), (130, 69)])
def test_divergence_is_reported(node):
    """One node with rho < 0, in a corner, on either side of a strip boundary, in the last row."""
    f = np.repeat(np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4), 131 * 70).reshape(9, 70, 131).copy()
    f[:, node[1], node[0]] = -0.2
    h = make(131, 70, 0.6, 0.1, W.CAVITY, "f32")
    S.smrt_set_f(h, f)
    with pytest.raises(S.SmrtError) as e:
        S.smrt_step(h, 3)
    assert e.value.status == S.SMRT_ERR_DIVERGED
    S.smrt_destroy(h)
