"""Pieces that end on multiples of 16 steps give the bits of one launch however few steps are left for the
last piece, and a served request has the same result alone and in chunks."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import serve
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def solve(scheme, steps, pieces):
    sample = B.sample_pulse_gauss if scheme == "magnus4" else B.sample_pulse
    a, a_in, a_out, _ = sample(W.sin2_pulse(1.0, 1.55, 5.0, eps=0.4), steps)
    g = B.Grid(37, 21, (-4.0, 4.0), (-3.0, 4.0), "fp32_mixed", scheme)
    g.set_pulse(a, 0.003, a_in, a_out)
    taken = B.get_groups(g.h)[0]
    for p in pieces:
        g.evolve(p)
    m, n = g.solve()
    torch.cuda.synchronize()
    out = m.cpu().numpy().copy(), n, g.state.cpu().numpy().view(np.uint32).copy()
    g.close()
    return out, taken


@pytest.mark.parametrize("scheme", ["exact", "strang_xy", "magnus4"])
@pytest.mark.parametrize("left", [1, 2, 3, 4, 5, 15])
def test_short_last_piece(scheme, left):
    steps = 160 + left
    (m, n, s), taken = solve(scheme, steps, [])
    assert taken > 0
    for pieces in ([160], [16, 144], [48, 112, left]):
        (m2, n2, s2), _ = solve(scheme, steps, pieces)
        assert np.array_equal(m, m2) and n == n2 and np.array_equal(s, s2), pieces


def test_served_in_chunks_or_at_once():
    """Chunks that leave 1, 2 and 3 steps for the last one."""
    reqs = serve.prepare([{"grid": {"nx": 40, "ny": 24, "px": (-4.0, 4.0), "py": (-4.0, 4.0)},
                           "pulse": W.sin2_pulse(0.5 + 0.2 * k, 1.55, 5.0, eps=0.4),
                           "steps": 4800 + k, "arrival_s": 0.0} for k in range(1, 4)])
    once, chunks = (serve.run(reqs, hbm_budget_bytes=1 << 30, max_active=n, chunk_steps=c,
                              keep_map=True, realtime=False)["results"]
                    for n, c in ((1, 1 << 30), (3, 480)))
    for k in range(3):
        assert np.array_equal(once[k]["map"], chunks[k]["map"])
        assert once[k]["density"] == chunks[k]["density"]
