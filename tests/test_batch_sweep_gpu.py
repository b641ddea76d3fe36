"""FP32 two-buffer batches, which take two or three updates per launch, against lattices of their own, bit for bit:
uneven widths and heights, every pairing of sides, and lattices that retire under a recorded run."""
import numpy as np
import pytest

import paper_2409_01076_gb300 as S
from gpu_util import get_f, make
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FLOWS = {"cavity": W.CAVITY, "periodic": W.ALL_PERIODIC, "couette": W.COUETTE, "channel": W.CHANNEL,
         "walls_x": W.bc_flags(W.MOVING, W.WALL, W.PERIODIC, W.PERIODIC)}
KINDS = {"smrt": S.SMRT_COLLISION_SMRT, "srt": S.SMRT_COLLISION_SRT}

# wide enough for passes to pay; widths that are multiples of 4 and 120, and that are not (one of them gives every
# lattice of a periodic batch the seam's loads); heights that are no multiple of any segment
UNEVEN = [(250, 301), (363, 97), (131, 260), (512, 333), (64, 64), (240, 129), (8, 8), (9, 250), (1001, 57), (128, 40),
          (1023, 640), (1601, 421)]
ALIGNED = [(n, m) for n, m in UNEVEN if n % 4 == 0] + [(1024, 640), (1600, 421)]


def create(sizes, tau, u, bc, kind="smrt"):
    return S.smrt_batch_create([s[0] for s in sizes], [s[1] for s in sizes], tau, u, bc, S.SMRT_PREC_F32,
                               S.SMRT_LAYOUT_AB, KINDS[kind])


def start_fields(nx, ny, seed):
    return W.random_macros(nx, ny, seed=seed, u_amp=0.03)


def batch_f(b, k, nx, ny):
    f = np.empty((9, ny, nx))
    S.smrt_batch_get_f(b, k, f)
    return f


@pytest.mark.parametrize("sizes", [UNEVEN, ALIGNED], ids=["uneven", "aligned"])
@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_steps_equal_single_lattices(sizes, flow, kind):
    n = len(sizes)
    tau, u = [0.55 + 0.04 * k for k in range(n)], [0.1 - 0.005 * k for k in range(n)]
    b = create(sizes, tau, u, FLOWS[flow], kind)
    for k, (nx, ny) in enumerate(sizes):
        S.smrt_batch_init_macros(b, k, *start_fields(nx, ny, k))
    for calls in (1, 2, 3, 4, 7):               # every order of passes, either buffer at the end
        S.smrt_batch_step(b, calls)
    for k, (nx, ny) in enumerate(sizes):
        h = make(nx, ny, tau[k], u[k], FLOWS[flow], "f32", "ab", kind)
        S.smrt_init_macros(h, *start_fields(nx, ny, k))
        for _ in range(17):
            S.smrt_step(h, 1)
        assert np.array_equal(get_f(h), batch_f(b, k, nx, ny)), (nx, ny)
        S.smrt_destroy(h)
    S.smrt_batch_destroy(b)


@pytest.mark.parametrize("check_every", [2, 10, 14, 200])
@pytest.mark.parametrize("residual", [S.SMRT_BATCH_RESIDUAL_STEP, S.SMRT_BATCH_RESIDUAL_STRIDE], ids=["step", "stride"])
@pytest.mark.parametrize("flow", ["cavity", "couette"])
def test_lattices_retire_one_after_another(check_every, residual, flow):
    """A recorded run whose list of lattices shrinks: each stands where its own count of updates says."""
    sizes = [(24, 24), (133, 20), (50, 41), (96, 64), (301, 30)]
    tau, u = [1.1, 0.9, 1.0, 0.7, 0.8], [0.02, 0.03, 0.01, 0.05, 0.02]
    b = create(sizes, tau, u, FLOWS[flow])
    most = 3000
    assert S.smrt_batch_run(b, 3e-4, check_every, most, residual) == 0
    steps, _, state = S.smrt_batch_status(b)
    assert len(set(steps.tolist())) >= 2 and (state != S.SMRT_BATCH_DIVERGED).all()
    assert (state == S.SMRT_BATCH_CONVERGED).sum() >= 2
    for k, (nx, ny) in enumerate(sizes):
        assert steps[k] % check_every == 0
        h = make(nx, ny, tau[k], u[k], FLOWS[flow], "f32")
        S.smrt_step(h, int(steps[k]))
        assert np.array_equal(get_f(h), batch_f(b, k, nx, ny)), (nx, ny, int(steps[k]))
        S.smrt_destroy(h)
    S.smrt_batch_destroy(b)


@pytest.mark.parametrize("flow", ["cavity", "periodic"])
def test_a_diverged_lattice_leaves_the_others_alone(flow):
    sizes = [(131, 70), (250, 91), (64, 40)]
    b = create(sizes, [0.6] * 3, [0.08] * 3, FLOWS[flow])
    for k, (nx, ny) in enumerate(sizes):
        rho, u = start_fields(nx, ny, 10 + k)
        if k == 1:
            rho[90, 249] = np.nan
        S.smrt_batch_init_macros(b, k, rho, u)
    S.smrt_batch_step(b, 6)
    S.smrt_batch_step(b, 5)
    assert S.smrt_batch_status(b)[2].tolist() == [S.SMRT_BATCH_ACTIVE, S.SMRT_BATCH_DIVERGED, S.SMRT_BATCH_ACTIVE]
    for k in (0, 2):
        nx, ny = sizes[k]
        h = make(nx, ny, 0.6, 0.08, FLOWS[flow], "f32")
        S.smrt_init_macros(h, *start_fields(nx, ny, 10 + k))
        S.smrt_step(h, 11)
        assert np.array_equal(get_f(h), batch_f(b, k, nx, ny))
        S.smrt_destroy(h)
    S.smrt_batch_destroy(b)
