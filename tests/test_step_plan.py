"""smrt_step_plan: what smrt_step launches, without a device; and, on one, the launches that a capture records."""
import ctypes
import os
import sys

import pytest

import paper_2409_01076_gb300 as S
from gpu_util import make
from paper_2409_01076_gb300 import workloads as W

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

STEP, SWEEP, TILE = S.SMRT_KERNEL_STEP, S.SMRT_KERNEL_SWEEP, S.SMRT_KERNEL_TILE


def plan(nx, ny, prec, n, layout="ab", rounding=S.SMRT_ROUND_NEAREST):
    h = make(nx, ny, 0.7, 0.1, W.CAVITY, prec, layout)
    S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, rounding)
    return S.smrt_step_plan(h, n)


@pytest.mark.parametrize("n,passes", [(0, 0), (1, 1), (2, 1), (3, 1), (4, 2), (5, 2), (6, 2), (7, 3), (20, 7),
                                      (10 ** 12, (10 ** 12 + 2) // 3)])
def test_sweeps_go_by_threes_and_twos(n, passes):
    for prec in ("f32", "f16", "bf16"):
        assert plan(8192, 8192, prec, n) == (passes, SWEEP if n >= 2 else STEP)


def test_everything_else_by_single_updates():
    assert plan(4096, 4096, "f64", 20) == (20, STEP)
    assert plan(4096, 4096, "f32", 20, "aa") == (20, STEP)
    assert plan(64, 64, "f64", 20, "aa") == (20, STEP)
    assert plan(7, 4096, "f32", 20) == (20, STEP) and plan(4096, 7, "f32", 20) == (20, STEP)
    assert plan(8192, 8192, "f16", 20, rounding=S.SMRT_ROUND_STOCHASTIC) == (20, STEP)


def test_small_lattices_in_tiles():
    launches, kernel = plan(64, 64, "f64", 2000)
    assert kernel == TILE and 2000 / 8 <= launches <= 2000 / 2
    per = round(2000 / launches)
    assert [plan(64, 64, "f64", n)[0] for n in (2, per, per + 1, 2 * per - 1)] == [1, 1, 2, 2]
    assert plan(64, 64, "f64", per + 1)[1] == TILE
    assert plan(256, 256, "f64", 50) == (50, STEP)      # the double pipe is full: one by one


def test_arguments():
    h = make(64, 64, 0.7, 0.1, W.CAVITY, "f32")
    with pytest.raises(S.SmrtError) as e:
        S.smrt_step_plan(h, -1)
    assert e.value.status == S.SMRT_ERR_ARG


def test_the_benchmark_asks_the_library():
    """No rule of its own, and every update kernel's source in its hash."""
    with open(bench.__file__) as fh:
        text = fh.read()
    assert "smrt_step_plan" in text and not hasattr(bench, "update_launches")
    assert all('"%s"' % name in text for name in ("d2q9.cuh", "kernels.cuh", "sweep.cuh", "tile.cuh"))


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,prec,layout,rounding", [
    (64, 64, "f64", "ab", 0), (130, 100, "f64", "ab", 0), (300, 300, "f64", "ab", 0), (64, 64, "f32", "aa", 0),
    (64, 64, "f32", "ab", 0), (384, 384, "f16", "ab", 0), (512, 512, "f32", "ab", 0), (1024, 1030, "bf16", "ab", 0),
    (1024, 1030, "f16", "ab", 1), (7, 300, "f32", "ab", 0)])
def test_a_capture_records_as_many_launches(nx, ny, prec, layout, rounding):
    import torch
    torch.cuda.init()
    with open("/proc/self/maps") as fh:
        rt = ctypes.CDLL(next(line.split()[-1] for line in fh if "libcudart.so" in line))
    h = make(nx, ny, 0.7, 0.1, W.CAVITY, prec, layout)
    S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, rounding)
    S.smrt_set_option(h, S.SMRT_OPT_CHECK_DIVERGENCE, 0)
    for n in (1, 23):                           # whatever a first call loads
        S.smrt_step(h, n)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    S.smrt_set_stream(h, side)
    st, graph, nodes = ctypes.c_void_p(side.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    for n in (1, 2, 5, 8, 23):
        assert rt.cudaStreamBeginCapture(st, 1) == 0
        S.smrt_step(h, n)
        assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) == 0
        assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(nodes)) == 0
        assert nodes.value == S.smrt_step_plan(h, n)[0], n
        assert rt.cudaGraphDestroy(graph) == 0
    S.smrt_set_stream(h, None)
    S.smrt_destroy(h)


@pytest.mark.parametrize("nx,ny,kernel", [
    (16, 16, TILE), (64, 64, TILE), (96, 96, TILE), (112, 112, TILE), (128, 64, TILE), (16, 1000, TILE),
    (144, 144, STEP), (192, 192, STEP), (256, 256, STEP), (500, 40, STEP), (40, 500, STEP), (300, 100, STEP)])
def test_double_tiles_where_they_were_measured_faster(nx, ny, kernel):
    """Tiles against one update per launch on 152 SMs, both measured: 64^2 3.3 / 4.7 us per update, 112^2 4.3 / 4.9,
    16 x 1000 4.2 / 8.1; 144^2 6.0 / 5.3, 500 x 40 6.0 / 5.7."""
    assert plan(nx, ny, "f64", 240)[1] == kernel


def test_bf16_stochastic_rounding_takes_passes_from_2048_squared():
    """One per launch / passes: 15.9 / 20.2 us at 1536^2, 30.8 / 28.2 at 2048^2."""
    sr = S.SMRT_ROUND_STOCHASTIC
    assert plan(2048, 2048, "bf16", 60, rounding=sr) == (20, SWEEP)
    assert plan(2048, 2047, "bf16", 60, rounding=sr) == (60, STEP)
    assert plan(2048, 2047, "bf16", 60) == (20, SWEEP)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(2048, 2048), (2049, 2051)])
@pytest.mark.parametrize("flow", [W.CAVITY, W.ALL_PERIODIC], ids=["cavity", "periodic"])
def test_bf16_stochastic_rounding_by_passes_is_the_same(nx, ny, flow):
    import numpy as np
    fields = []
    for calls in ([1] * 5, [5], [2, 3]):
        h = make(nx, ny, 0.6, 0.1, flow, "bf16")
        S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, S.SMRT_ROUND_STOCHASTIC)
        S.smrt_init_macros(h, *W.random_macros(nx, ny, seed=5, u_amp=0.03))
        for n in calls:
            S.smrt_step(h, n)
        rho, u = np.empty((ny, nx)), np.empty((2, ny, nx))
        S.smrt_macros(h, rho, u)
        S.smrt_destroy(h)
        fields.append((rho, u))
    for rho, u in fields[1:]:
        assert np.array_equal(rho, fields[0][0]) and np.array_equal(u, fields[0][1])
