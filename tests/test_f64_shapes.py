"""The FP64 kernels' shapes -- 32 columns x 4 rows or 32 consecutive points per warp, or 8 points per
warp pair, one warp forming the operators and one applying them -- give bitwise the same map, density
and state.  The tiling hook forces the first two; sizes up to a few thousand points take pairs."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def solve(size, table, scheme, tiling, valley=1, pieces=()):
    a, a_in, a_out, dt = table
    g = B.Grid(size[0], size[1], (-3.0, 5.0), (-2.5, 3.5), "fp64", scheme, valley)
    B.test_tiling(g.h, tiling)
    g.set_pulse(a, dt, a_in, a_out)
    for p in pieces:
        g.evolve(p)
    m, n = g.solve()
    torch.cuda.synchronize()
    out = m.cpu().numpy().copy(), n, g.state.cpu().numpy().view(np.uint32).copy()  # its bits
    g.close()
    return out


# one point; warps not full; one pair per scheduler; several; several warps per scheduler
@pytest.mark.parametrize("size", [(1, 1), (7, 3), (64, 65), (131, 90), (300, 257)])
@pytest.mark.parametrize("scheme", ["exact", "strang_xy", "magnus4"])
@pytest.mark.parametrize("steps", [1, 67, 130])
def test_shapes_agree_bitwise(orc, size, scheme, steps):
    pulse = W.sin2_pulse(2.0, 1.2, 0.003 * steps, eps=0.6)
    sample = B.sample_pulse_gauss if scheme == "magnus4" else B.sample_pulse
    tab = sample(pulse, steps)
    m, n, s = solve(size, tab, scheme, 1, valley=-1)
    for tiling in (0, 2):
        m1, n1, s1 = solve(size, tab, scheme, tiling, valley=-1)
        assert np.array_equal(m, m1) and n == n1 and np.array_equal(s, s1)
    if steps > 1:  # any split of FP64 steps
        m1, n1, s1 = solve(size, tab, scheme, 1, valley=-1, pieces=(1, steps - 5, 2))
        assert np.array_equal(m, m1) and n == n1 and np.array_equal(s, s1)
    a, a_in, a_out, dt = (orc.pulse_table_gauss if scheme == "magnus4" else orc.pulse_table)(
        pulse, steps)
    ref, _, _, nref = orc.solve_grid(size[0], size[1], (-3.0, 5.0), (-2.5, 3.5), a, dt, a_in,
                                     a_out, scheme=scheme, valley=-1)
    assert np.abs(m - ref).max() <= 1e-9 and abs(n - nref) <= 1e-10 * nref
