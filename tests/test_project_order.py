"""Projection of a large FP32-mixed grid, whose granules are dealt in another order than a small
one's: the map has the bits of its row bands'."""
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


# whole rows of granules, four rounds of the chip and more (with a ragged last round); just
# below; and rows that are not whole granules
@pytest.mark.parametrize("nx,ny", [(2048, 2048), (3072, 1337), (256, 14999), (2048, 1200),
                                   (2049, 1999)])
@pytest.mark.parametrize("expand", [True, False])
def test_bands_have_the_full_grid_s_bits(nx, ny, expand):
    steps = 48
    a, a_in, a_out, dt = B.sample_pulse(W.sin2_pulse(1.0, 1.55, 5.0, 0.5), 2000)

    def solve(rows=None):
        g = B.Grid(nx, ny, (-6.0, 6.0), (-6.0, 6.0), "fp32_mixed", rows=rows)
        B.test_expansion(g.h, expand)
        g.set_pulse(a[900:900 + steps].copy(), dt, a_in, a_out)
        g.evolve(steps)
        g.project()
        torch.cuda.synchronize()
        m = g.map.cpu().numpy().reshape(-1, nx).copy()
        g.solve()  # and in one call
        torch.cuda.synchronize()
        np.testing.assert_array_equal(g.map.cpu().numpy().reshape(-1, nx), m)
        g.close()
        return m

    full = solve()
    cuts = [ny * k // 5 for k in range(6)]
    for lo, hi in zip(cuts, cuts[1:]):
        np.testing.assert_array_equal(solve((lo, hi)), full[lo:hi])
