"""Device scratch of a batch's host-array calls: given back where it is large."""
import numpy as np
import pytest
import torch

import paper_2409_01076_gb300 as S
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_host_arrays_leave_little_scratch_behind():
    n = 2000                                    # 288 MB of populations, 96 MB of fields
    b = S.smrt_batch_create([n, 64], [n, 64], [0.6, 0.7], [0.05, 0.05], W.CAVITY, S.SMRT_PREC_F32)
    rho, u = np.ones((n, n)), np.zeros((2, n, n))
    small = np.ones((64, 64)), np.zeros((2, 64, 64))
    S.smrt_batch_init_macros(b, 1, *small)      # whatever a first call loads
    S.smrt_batch_macros(b, 1, *small)
    f = np.empty((9, 64, 64))
    S.smrt_batch_get_f(b, 1, f)
    before = free()
    f = np.empty((9, n, n))
    u[0] = 0.01
    S.smrt_batch_init_macros(b, 0, rho, u)
    assert before - free() <= 72 << 20          # 64 MiB may be kept, in pages of 2
    S.smrt_batch_get_f(b, 0, f)
    assert before - free() <= 72 << 20
    r, v = np.empty_like(rho), np.empty_like(u)
    S.smrt_batch_macros(b, 0, r, v)
    assert before - free() <= 72 << 20
    assert np.abs(r - 1.0).max() <= 1e-6 and np.abs(v - u).max() <= 1e-6
    assert np.abs(f.sum(0) - 1.0).max() <= 1e-6
    S.smrt_batch_macros(b, 1, *small)           # and the small lattice's calls go on
    S.smrt_batch_destroy(b)
