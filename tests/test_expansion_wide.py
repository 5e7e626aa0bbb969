"""The expansion's widest level (group angles above 0.32) keeps the small part v of a group's rotation
S + v apart from S; the operator's vector part is then sinc|w| (S + v), v's own share included.

Tolerance: 1e-5 against the FP64 oracle, FP32-mixed's target."""
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
    groups = B.get_groups(g.h)
    m, _ = g.solve()
    torch.cuda.synchronize()
    out = m.double().cpu().numpy().copy()
    g.close()
    return out, groups


# the run's length and A_in, A_out: what shows the term best in each scheme
@pytest.mark.parametrize("scheme,steps,a_in,a_out", [
    ("exact", 40000, (0.0, 0.01), (0.0, 8.0)), ("magnus4", 40000, (0.0, 0.01), (0.0, 8.0)),
    ("strang_xy", 20000, (0.0, 8.0), (0.0, -8.0))])
def test_field_at_the_precession_frequency(orc, scheme, steps, a_in, a_out):
    """A weak A_y at the precession frequency of the momenta at p_x = 8.6, in groups of 16 at the
    angle 0.66: what it adds to a group is as small as 1e-6, but adds up over the run (with v's share
    left out of sinc|w| v the map was off by 5e-5, 5e-5 and 1.5e-5).  A slow A_x of 1e-3 keeps P from
    being the same in every step, where any FP32 rounding adds up too."""
    dt, p0 = 0.0045, 8.6
    px, py = (-9.2, 9.2), (-0.6, 0.6)  # nodes at p_x = +-8.6, p_y = 0
    half = np.sqrt(3) / 6 if scheme == "magnus4" else 0.0
    t = dt * (np.arange(steps)[:, None] + 0.5 + half * np.array([-1.0, 1.0]))
    a = np.zeros((steps, 2, 2))
    a[:, :, 0] = 1e-3 * np.sin(2 * np.pi * t / (977 * dt))
    a[:, :, 1] = 3e-3 * np.cos(2 * p0 * t)
    a = a.reshape(steps, 4) if scheme == "magnus4" else a[:, 0]
    a_in, a_out = np.array(a_in), np.array(a_out)
    m, groups = solve((46, 3), px, py, a, dt, a_in, a_out, scheme)
    ref = orc.solve_grid(46, 3, px, py, a, dt, a_in, a_out, scheme=scheme)[0]
    assert groups == (16, 2)
    assert np.abs(m - ref).max() <= TOL


# group angle 0.59 in groups of 16 and of 8
@pytest.mark.parametrize("dt,steps,G", [(0.006, 4003, 16), (0.012, 2405, 8)])
def test_split_steps_in_a_nearly_constant_field(orc, dt, steps, G):
    """STRANG_XY's own part of v is there without any change of A (left out of sinc|w| v it came to
    1.2e-5 and 5e-5 here)."""
    rng = np.random.default_rng(5)
    a = 1e-4 * rng.standard_normal((steps, 2))
    a_in, a_out = np.array([0.5, -1.0]), np.array([-2.0, 0.25])
    px, py = (-4.0, 5.0), (-3.5, 3.0)
    m, groups = solve((33, 9), px, py, a, dt, a_in, a_out, "strang_xy")
    ref = orc.solve_grid(33, 9, px, py, a, dt, a_in, a_out, scheme="strang_xy")[0]
    assert groups == (G, 2)
    assert np.abs(m - ref).max() <= TOL
