"""A launch that fails is reported by its own call and by no later one."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2409_01076_gb300 as S
from gpu_util import make
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu

THREAD_LOCAL = 1


def runtime():
    """The CUDA runtime that torch has loaded."""
    torch.cuda.init()
    with open("/proc/self/maps") as fh:
        path = next(line.split()[-1] for line in fh if "libcudart.so" in line)
    return ctypes.CDLL(path)


@pytest.mark.parametrize("nx,ny,prec,layout,n", [(64, 64, "f64", "ab", 4), (731, 710, "f32", "ab", 3), (64, 64, "f32", "aa", 2)])
def test_a_failed_update_leaves_the_next_call_alone(nx, ny, prec, layout, n):
    """The launch fails on the host: the stream's capture was spoilt by waiting for it."""
    rt = runtime()
    h = make(nx, ny, 0.7, 0.1, W.CAVITY, prec, layout)
    S.smrt_set_option(h, S.SMRT_OPT_CHECK_DIVERGENCE, 0)
    S.smrt_step(h, n)
    rho, u = np.empty((ny, nx)), np.empty((2, ny, nx))
    S.smrt_macros(h, rho, u)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    S.smrt_set_stream(h, side.cuda_stream)
    st = ctypes.c_void_p(side.cuda_stream)
    assert rt.cudaStreamBeginCapture(st, THREAD_LOCAL) == 0
    assert rt.cudaStreamSynchronize(st) != 0                # not permitted: the capture is invalid from here on
    with pytest.raises(S.SmrtError) as e:
        S.smrt_step(h, n)
    assert e.value.status == S.SMRT_ERR_CUDA
    graph = ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) != 0
    rt.cudaGetLastError()                                   # torch's runtime; the library links its own
    S.smrt_set_stream(h, 0)
    rho2, u2 = np.empty_like(rho), np.empty_like(u)
    S.smrt_macros(h, rho2, u2)                              # launches, and asks for the last error
    assert np.array_equal(rho, rho2) and np.array_equal(u, u2)
    assert S.smrt_time(h) == n
    S.smrt_destroy(h)
