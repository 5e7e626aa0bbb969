"""The server's budget counts what a request takes on the device, its expanded step groups included; a
request that fits only without them goes step by step, whatever else is active."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import serve
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 30000
PLAIN = 32 * 64 * 64 + 8 * STEPS + 4 * 64 * 64 + 2048  # state, table, map, the small arrays
GROUPS = 52 * STEPS  # FP64 table 16, running sums 1, entries 80 (1/16 + 1/8 + 1/4) bytes a step


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def requests(count):
    """Long pulses on small grids: groups of 16 may be expanded."""
    return serve.prepare([{"grid": {"nx": 64, "ny": 64, "px": (-4.0, 4.0), "py": (-4.0, 4.0)},
                           "pulse": W.sin2_pulse(0.5 + 0.1 * k, 1.55, 5.0, eps=0.4),
                           "steps": STEPS, "arrival_s": 0.0} for k in range(count)])


def run(reqs, budget, max_active=6):
    seen = []
    out = serve.run(reqs, hbm_budget_bytes=int(budget), max_active=max_active, chunk_steps=6400,
                    keep_map=True, realtime=False, on_step=lambda a, q, f: seen.append(a + f))
    assert all(v["state"] == "done" for v in out["results"].values())
    return out["results"], max(seen)


def solve(r, expand):
    a, a_in, a_out, dt = r["table"]
    g = B.Grid(64, 64, (-4.0, 4.0), (-4.0, 4.0), "fp32_mixed")
    B.test_expansion(g.h, expand)
    g.set_pulse(a, dt, a_in, a_out)
    assert (B.get_groups(g.h)[0] == 16) == expand
    m, n = g.solve()
    torch.cuda.synchronize()
    out = m.cpu().numpy().copy(), n
    g.close()
    return out


def test_budget_counts_the_expanded_groups():
    """Room for two and a half requests with their groups (ten without): never more than two."""
    reqs = requests(6)
    res, most = run(reqs, 2.5 * (PLAIN + GROUPS))
    assert most == 2
    m, n = solve(reqs[3], True)
    assert np.array_equal(res[3]["map"], m) and res[3]["density"] == n


def test_a_budget_without_room_for_the_groups():
    """A request that fits without its groups is served step by step, alone or beside others."""
    reqs = requests(3)
    m, n = solve(reqs[1], False)
    for budget in (1.2 * PLAIN, 0.99 * (PLAIN + GROUPS)):
        res, most = run(reqs, budget)
        assert most == (1 if budget < 2 * PLAIN else 3)
        assert np.array_equal(res[1]["map"], m) and res[1]["density"] == n
    with pytest.raises(B.DSPError) as e:
        run(reqs, 0.9 * PLAIN)
    assert e.value.code == -2
