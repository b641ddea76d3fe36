"""smrt_macros in 64 bits where 1 / rho is no ordinary number: the quotients j / rho of IEEE arithmetic."""
import numpy as np
import pytest

import paper_2409_01076_gb300 as S
from gpu_util import get_macros, make
from paper_2409_01076_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def moments(f):
    """rho and u by divisions, the sums in the order of the kernels."""
    g = f - WT
    with np.errstate(all="ignore"):
        drho = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8]
        jx = (g[1] - g[3]) + ((g[5] - g[7]) - (g[6] - g[8]))
        jy = (g[2] - g[4]) + ((g[5] - g[7]) + (g[6] - g[8]))
        rho = 1.0 + drho
        return rho, jx / rho, jy / rho


def massless():
    """Populations of a node whose rho is exactly zero and whose momentum is not."""
    f = np.array([0.0, 0.25, 0.125, -0.5, 0.0, 0.0, 0.0, 0.0, 0.0])
    f[0] = -f[1:].sum()
    for _ in range(100):
        rho = moments(f)[0]
        if rho == 0.0:
            return f
        f[0] -= rho
    raise AssertionError("no such node")


def node(**kw):
    f = WT.copy()
    for k, v in kw.items():
        f[int(k[1:])] = v
    return f


NODES = [massless(), node(f0=np.inf, f1=0.3), node(f1=1.7e308, f3=-1.7e308), node(f0=8e307, f1=8e307),
         node(f0=2.0 ** 1021, f2=2.0 ** 1019), node(f0=-3.0, f1=0.2), node(f2=np.nan), node(f0=1e-3, f6=0.4), WT * 1.25]


@pytest.mark.parametrize("layout", ["ab", "aa"])
def test_velocity_is_the_quotient(layout):
    nx, ny = 24, 20
    f = np.repeat(WT, nx * ny).reshape(9, ny, nx).copy()
    at = [(1 + 2 * (k // 3), 2 + 5 * (k % 3)) for k in range(len(NODES))]
    at[0] = (0, 0)                              # one at the seam, the others inside
    for (j, i), q in zip(at, NODES):
        f[:, j, i] = q
    h = make(nx, ny, 0.8, 0.0, W.ALL_PERIODIC, "f64", layout)
    S.smrt_set_f(h, f)
    rho, u = get_macros(h)
    S.smrt_destroy(h)
    for (j, i), q in zip(at, NODES):
        r, ux, uy = moments(q)
        assert np.array_equal(rho[j, i], r, equal_nan=True), (j, i)
        for got, want in ((u[0, j, i], ux), (u[1, j, i], uy)):
            if np.isfinite(want):
                assert abs(got - want) <= 2.3e-16 * abs(want), (j, i, got, want)    # one unit in the last place
            else:
                assert np.array_equal(got, want, equal_nan=True), (j, i, got, want)
