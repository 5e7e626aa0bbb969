"""Tables made to be hard for the expansion of step groups: what it drops has to be counted, so that
the run is either taken from the expansion within the FP32-mixed tolerance or goes step by step.

Tolerance: 1e-5 against the FP64 oracle, FP32-mixed's target (the expansion's bound on what it
drops, 4e-6, plus the rounding of either path, below 1e-6 at these step counts)."""
import math

import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def solve(size, px, py, a, dt, a_in, a_out, scheme):
    g = B.Grid(size[0], size[1], px, py, "fp32_mixed", scheme)
    g.set_pulse(a, dt, a_in, a_out)
    groups = B.get_groups(g.h)[0]
    m, n = g.solve()
    torch.cuda.synchronize()
    out = m.double().cpu().numpy().copy()
    g.close()
    return out, n, groups


# D: of a step, |D| = (sqrt(3)/6) dt |A2 - A1|
@pytest.mark.parametrize("D,groups", [(1.8e-5, 4), (3e-5, 0)])
def test_magnus4_commutators_at_the_precession_frequency(orc, D, groups):
    """MAGNUS4 steps whose two samples differ in A_y (their mean is zero), with opposite signs in the
    two halves of every group of four and a size that follows the precession of the momenta at p_x =
    8.6: the plane's fourth-order term in D then adds up over the run (left out, it came to 3e-5 in
    the operator and 1.3e-5 and 2.1e-5 in the map at these sizes).  A slow A_x of 1e-3 keeps P from
    being the same in every step, where any FP32 rounding adds up too."""
    steps, dt, p0 = 20000, 0.01, 8.6
    n = np.arange(steps)
    sign = np.where(n % 4 < 2, -1.0, 1.0) * np.cos(2 * dt * p0 * (n - n % 4 + 1.5))
    a = np.zeros((steps, 4))
    a[:, 1] = D / (dt * math.sqrt(3) / 3) * sign
    a[:, 3] = -a[:, 1]
    a[:, 0] = a[:, 2] = 1e-3 * np.sin(2 * np.pi * n / 977)
    a_in, a_out = np.array([0.0, 8.0]), np.array([0.0, -8.0])
    px, py = (-9.2, 9.2), (-0.6, 0.6)  # nodes at p_x = +-8.6, p_y = 0
    m, _, taken = solve((46, 3), px, py, a, dt, a_in, a_out, "magnus4")
    ref = orc.solve_grid(46, 3, px, py, a, dt, a_in, a_out, scheme="magnus4")[0]
    assert taken == groups
    assert np.abs(m - ref).max() <= TOL


@pytest.mark.parametrize("scheme", ["exact", "strang_xy", "magnus4"])
@pytest.mark.parametrize("kind", ["noise", "step", "spikes", "D"])
@pytest.mark.parametrize("dt,steps", [(0.0008, 20003), (0.003, 8005), (0.012, 4003)])
def test_rough_tables_of_every_scheme(orc, scheme, kind, dt, steps):
    """Group sizes 16, 8 or 4 (theta_max 0.005, 0.02, 0.07), over potentials too rough for the
    expansion, just smooth enough, and smooth; D: noise that cancels within every step."""
    rng = np.random.default_rng(5)
    width = 4 if scheme == "magnus4" else 2
    taken = []
    for amp in (1e-4, 3e-3, 0.1, 1.0):
        a = np.zeros((steps, width))
        if kind == "noise":
            a = amp * rng.standard_normal((steps, width)).clip(-3, 3)
        elif kind == "step":
            a[steps // 3:] = amp
        elif kind == "spikes":
            a[rng.integers(0, steps, 40)] = amp
        else:
            a[:, :2] = amp * rng.standard_normal((steps, 2)).clip(-3, 3)
            a[:, 2:] = -a[:, :2] if width == 4 else 0.0
        a_in, a_out = np.array([0.5, -1.0]), np.array([-2.0, 0.25])
        px, py = (-4.0, 5.0), (-3.5, 3.0)
        m, _, groups = solve((33, 9), px, py, a, dt, a_in, a_out, scheme)
        ref = orc.solve_grid(33, 9, px, py, a, dt, a_in, a_out, scheme=scheme)[0]
        taken.append(groups)
        assert np.abs(m - ref).max() <= TOL, (amp, groups)
    assert taken[0] > 0 and taken == sorted(taken, reverse=True)
