"""FP64 state of long STRANG_XY and MAGNUS4 runs against the same steps in long double: the error is the
rounding of the updates, which does not add up in one direction."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def product(scheme, a, dt, px, py):
    """First column (alpha, beta) of U_N ... U_1 for one momentum, from the steps' dt P as the FP64
    kernels round it; multiplied in pairs."""
    if scheme == "magnus4":
        kappa = -np.sqrt(3.0) / 6.0
        Px = dt * px + dt * (0.5 * (a[:, 0] + a[:, 2]))
        Py = dt * py + dt * (0.5 * (a[:, 1] + a[:, 3]))
        dx, dy = kappa * (dt * (a[:, 2] - a[:, 0])), kappa * (dt * (a[:, 3] - a[:, 1]))
        x, y = Px.astype(L), Py.astype(L)
        z = x * dy.astype(L) - y * dx.astype(L)
        r = np.sqrt(x * x + y * y + z * z)
        s = np.sin(r) / r
        ar, ai, br, bi = np.cos(r), -s * z, s * y, -s * x
    else:
        x, y = (dt * px + dt * a[:, 0]).astype(L), (dt * py + dt * a[:, 1]).astype(L)
        cx, sx, cy, sy = np.cos(x), np.sin(x), np.cos(y), np.sin(y)
        ar, ai, br, bi = cx * cy, 0 * cx, sy, -cy * sx
    while len(ar) > 1:
        if len(ar) % 2:
            ar, ai, br, bi = (np.append(v, L(e)) for v, e in ((ar, 1), (ai, 0), (br, 0), (bi, 0)))
        ar1, ai1, br1, bi1 = ar[0::2], ai[0::2], br[0::2], bi[0::2]
        ar2, ai2, br2, bi2 = ar[1::2], ai[1::2], br[1::2], bi[1::2]
        # alpha = alpha2 alpha1 - conj(beta2) beta1, beta = beta2 alpha1 + conj(alpha2) beta1
        ar, ai, br, bi = (ar2 * ar1 - ai2 * ai1 - br2 * br1 - bi2 * bi1,
                          ar2 * ai1 + ai2 * ar1 - br2 * bi1 + bi2 * br1,
                          br2 * ar1 - bi2 * ai1 + ar2 * br1 + ai2 * bi1,
                          br2 * ai1 + bi2 * ar1 + ar2 * bi1 - ai2 * br1)
    return ar[0], ai[0], br[0], bi[0]


# series degrees (4, 3), (5, 5), (5, 5), (6, 6)
@pytest.mark.parametrize("scheme", ["strang_xy", "magnus4"])
@pytest.mark.parametrize("steps,theta", [(100000, 0.015), (100000, 0.06), (20000, 0.1),
                                         (20000, 0.18)])
def test_long_runs_against_long_double(scheme, steps, theta):
    """1e5 steps at theta 0.06 (and others).  A step rounds each component of the state once at its size (0.6 of
    2^-53 times about 0.5, 3.3e-17) and the diagonal once at 1 (3.2e-17, shared): about 5e-17 a step
    and component, 1.6e-14 over the run as a random walk; three times that is allowed.  (With
    the small parts as pairs of floats, off by 2^-50 of theta^2/2 in one direction, it came to
    5.4e-14 and 6.0e-14 here, and to 1.6e-13 for momenta that are at theta 0.06 throughout.)"""
    nx, ny = 4, 2
    sample = B.sample_pulse_gauss if scheme == "magnus4" else B.sample_pulse
    a, a_in, a_out, _ = sample(W.sin2_pulse(1.0, 1.55, 5.0, 0.5), steps)
    dt = theta / np.hypot(4.0 + np.abs(a[:, 0::2]).max(), 4.0 + np.abs(a[:, 1::2]).max())
    h = B.create_grid(nx, ny, (-4.0, 4.0), (-4.0, 4.0), "fp64", scheme)
    B.set_pulse(h, a, dt, a_in, a_out)
    first, last = (np.zeros(B.state_bytes(nx, ny, "fp64"), np.uint8) for _ in range(2))
    B.save_state(h, first)
    B.evolve(h, steps)
    B.save_state(h, last)
    B.destroy_grid(h)
    n = nx * ny
    p0, p1 = (v.view(np.float64).reshape(2, n, 2) for v in (first, last))  # planes a, b
    err = []
    for k in range(n):
        px, py = -4.0 + (k % nx + 0.5) * 2.0, -4.0 + (k // nx + 0.5) * 4.0  # exact
        ar, ai, br, bi = product(scheme, a, dt, px, py)
        (xr, xi), (yr, yi) = p0[0, k].astype(L), p0[1, k].astype(L)
        ref = (ar * xr - ai * xi - br * yr - bi * yi, ar * xi + ai * xr - br * yi + bi * yr,
               br * xr - bi * xi + ar * yr + ai * yi, br * xi + bi * xr + ar * yi - ai * yr)
        err += [float(v - w.astype(L)) for v, w in zip(ref, np.r_[p1[0, k], p1[1, k]])]
    assert np.sqrt(np.mean(np.square(err))) <= 5e-14 * np.sqrt(steps / 1e5)
