"""The step-by-step FP32-mixed kernels where the library would evaluate groups expanded: row strips,
their last wave in 2-row strips, contiguous tiles and the projection in the evolve launch, with the
expansion switched off, and left to its own bound on tables it refuses."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# steps -> step group (theta_max ~ 128 / steps on [-4, 4]^2): 16, 8, 4, 2
STEPS = {"exact": {16: 10000, 8: 5000, 4: 2500, 2: 1300},
         "strang_xy": {16: 10000, 8: 5000, 4: 2500, 2: 1300},
         "magnus4": {16: 12000, 8: 6000, 4: 3000, 2: 1600}}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def sample(scheme, steps):
    f = B.sample_pulse_gauss if scheme == "magnus4" else B.sample_pulse
    return f(W.sin2_pulse(1.0, 1.55, 5.0, eps=0.4), steps)


def solve(size, tab, scheme="exact", tiling=1, expand=False, pieces=None, project=False, **kw):
    a, a_in, a_out, dt = tab
    g = B.Grid(size[0], size[1], (-4.0, 4.0), (-4.0, 4.0), "fp32_mixed", scheme, **kw)
    B.test_expansion(g.h, expand)
    B.test_tiling(g.h, tiling)
    g.set_pulse(a, dt, a_in, a_out)
    assert B.get_groups(g.h)[0] == 0
    info = B.get_info(g.h)
    if project:  # the projection in a launch of its own
        g.evolve(len(a))
        m, n = g.project(), g.density()
    else:
        for p in pieces or []:
            g.evolve(p)
        m, n = g.solve()
    torch.cuda.synchronize()
    out = m.cpu().numpy().copy(), n
    g.close()
    return out, info


def same(a, b):
    return np.array_equal(a[0], b[0]) and a[1] == b[1]


@pytest.mark.parametrize("scheme", ["exact", "strang_xy", "magnus4"])
@pytest.mark.parametrize("G", [16, 8, 4, 2])
def test_strips_equal_contiguous_tiles(orc, G, scheme):
    """Every step group: row strips (10 rows: the last strip hangs over), 4-row strips only, contiguous
    tiles and a projection of its own give the same bits, whole and in pieces, and meet the oracle."""
    tab = sample(scheme, STEPS[scheme][G])
    ref, info = solve((512, 10), tab, scheme)
    assert info["group_steps"] == G and info["row_strips"] == 1
    for kw in ({"tiling": 2}, {"tiling": 0}, {"project": True}, {"tiling": 0, "project": True},
               {"pieces": [16, 640]}):
        assert same(ref, solve((512, 10), tab, scheme, **kw)[0]), kw
    f = orc.pulse_table_gauss if scheme == "magnus4" else orc.pulse_table
    a, a_in, a_out, dt = f(W.sin2_pulse(1.0, 1.55, 5.0, eps=0.4), STEPS[scheme][G])
    m = orc.solve_grid(512, 10, (-4.0, 4.0), (-4.0, 4.0), a, dt, a_in, a_out, scheme=scheme)[0]
    assert np.abs(ref[0] - m).max() <= 1e-5


@pytest.mark.parametrize("scheme", ["exact", "strang_xy", "magnus4"])
def test_last_wave_in_two_row_strips(scheme):
    """512 x 700: the 350 strip tiles leave a last wave that is split (rows 608 and up)."""
    tab = sample(scheme, 12000)
    ref, _ = solve((512, 700), tab, scheme)
    assert same(ref, solve((512, 700), tab, scheme, tiling=2)[0])
    assert same(ref, solve((512, 700), tab, scheme, tiling=0)[0])


def test_bands_and_valleys_on_strips():
    tab = sample("exact", 5000)
    ref, _ = solve((256, 23), tab, valley=-1)
    for tiling in (0, 1):
        band, _ = solve((256, 23), tab, tiling=tiling, valley=-1, rows=(7, 19))
        assert np.array_equal(band[0], ref[0][7:19])


# noise in every group is seen on the host; jumps in a quarter of them only in the groups' sums
@pytest.mark.parametrize("kind", ["noise", "jumps"])
@pytest.mark.parametrize("size", [(512, 10), (512, 700), (300, 9)])
@pytest.mark.parametrize("keep", [True, False])
def test_tables_that_the_expansion_refuses(orc, size, keep, kind):
    """Tables over the expansion's bound, expansion on: the run goes step by step, as it does when the
    expansion is off, the final state kept or not."""
    rng = np.random.default_rng(4)
    a = rng.standard_normal((3001, 2)).clip(-3, 3)
    if kind == "jumps":
        a = np.repeat(rng.choice([-2.0, 2.0], (3001 // 16 + 1, 2)), 16, axis=0)[1:3002]
    tab = (a, np.zeros(2), np.array([0.5, 0.0]), 0.002)
    ref, info = solve(size, tab)
    assert info["group_steps"] > 1
    g = B.Grid(size[0], size[1], (-4.0, 4.0), (-4.0, 4.0), "fp32_mixed")
    B.set_keep_final_state(g.h, keep)
    g.set_pulse(tab[0], tab[3], tab[1], tab[2])
    assert B.get_groups(g.h)[0] == 0
    g.evolve(1600)
    m, n = g.solve()
    torch.cuda.synchronize()
    # the two make the step table in different ways (half an ulp of its running sum apart)
    assert np.abs(m.cpu().numpy() - ref[0]).max() <= 2e-6 and abs(n - ref[1]) <= 1e-6 * n
    assert np.abs(m.cpu().numpy().astype(np.float64)
                  - orc.solve_grid(size[0], size[1], (-4.0, 4.0), (-4.0, 4.0), a, tab[3], tab[1],
                                   tab[2])[0]).max() <= 1e-5 or size[1] > 100
    if keep:  # the projection of the state that was left has the same bits
        first = m.cpu().numpy().copy()
        m2 = g.project()
        torch.cuda.synchronize()
        assert np.array_equal(m2.cpu().numpy(), first)
    else:
        with pytest.raises(B.DSPError) as e:
            g.project()
        assert e.value.code == -4
    g.close()


@pytest.mark.parametrize("size,steps,expanded", [
    ((256, 256), 511, False), ((256, 256), 512, True), ((1024, 512), 63, False),
    ((1024, 512), 64, True), ((512, 2), 511, False), ((512, 2), 512, True), ((64, 64), 4, True),
    ((1100, 1000), 31, False), ((1100, 1000), 32, True)])
def test_pulses_too_short_to_expand(size, steps, expanded):
    """The line by grid and length, and a band on the full grid's side of it, bit for bit."""
    a, a_in, a_out, _ = sample("exact", steps)
    out = []
    for rows in (None, (1, 2)):
        g = B.Grid(size[0], size[1], (-4.0, 4.0), (-4.0, 4.0), "fp32_mixed", rows=rows)
        g.set_pulse(a, 0.002, a_in, a_out)
        assert (B.get_groups(g.h)[0] > 0) == expanded
        m, _ = g.solve()
        torch.cuda.synchronize()
        out.append(m.cpu().numpy().copy())
        g.close()
    assert np.array_equal(out[1], out[0][1:2])
