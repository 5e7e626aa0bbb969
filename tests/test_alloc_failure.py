"""A device without room for a pulse's expanded step groups: a grid's pulse goes step by step (and says
so), a served request waits, so that its result does not depend on what else is on the device.  The
allocations fail in the library's own hook; nothing is driven out of memory."""
import numpy as np
import pytest
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GRID = {"nx": 70, "ny": 33, "px": (-4.0, 4.0), "py": (-3.0, 4.0)}
STEPS = 6001


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1607_03062_gb300 import build
    build.build()
    B.lib()
    torch.cuda.set_device(0)


def table(k=0):
    return B.sample_pulse(W.sin2_pulse(1.0 + 0.2 * k, 1.55, 5.0, eps=0.4), STEPS)


def grid():
    return B.Grid(GRID["nx"], GRID["ny"], GRID["px"], GRID["py"], "fp32_mixed")


def set_pulse(g, tab):
    g.set_pulse(tab[0], tab[3], tab[1], tab[2])


def solve(g):
    m, n = g.solve()
    torch.cuda.synchronize()
    return m.cpu().numpy().copy(), n


def plain(tab, expand):
    g = grid()
    B.test_expansion(g.h, expand)
    set_pulse(g, tab)
    out = solve(g)
    g.close()
    return out


# the groups' memory; the table's behind it; and on a grid that has both, for a longer pulse
@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("again", [False, True])
def test_no_room_for_the_groups(skip, again):
    tab = table()
    g = grid()
    if again:
        short = B.sample_pulse(W.sin2_pulse(1.0, 1.55, 5.0, eps=0.4), STEPS // 2)
        set_pulse(g, short)
    B.test_fail_alloc(g.h, skip, 1)
    set_pulse(g, tab)
    assert B.get_groups(g.h)[0] == 0
    m, n = solve(g)
    ms, ns = plain(tab, False)
    assert np.array_equal(m, ms) and n == ns
    set_pulse(g, tab)  # room again
    assert B.get_groups(g.h)[0] > 0
    m, n = solve(g)
    ms, ns = plain(tab, True)
    assert np.array_equal(m, ms) and n == ns
    g.close()


def test_no_room_for_the_table():
    """DSP_E_NOMEM, the pulse before is gone, and the grid takes the next one."""
    g = grid()
    set_pulse(g, B.sample_pulse(W.sin2_pulse(1.0, 1.55, 5.0), 100))
    B.test_fail_alloc(g.h, 0, 2)
    with pytest.raises(B.DSPError) as e:
        set_pulse(g, table())
    assert e.value.code == -2
    with pytest.raises(B.DSPError) as e:
        g.evolve(1)
    assert e.value.code == -4
    set_pulse(g, table())
    m, n = solve(g)
    ms, ns = plain(table(), True)
    assert np.array_equal(m, ms) and n == ns
    g.close()


def submit(srv, tab):
    return B.server_submit(srv, B.make_request(GRID, STEPS, tab[3], tab[1], tab[2], keep_map=True),
                           tab[0])


def finish(srv):
    for _ in range(100):
        if B.server_step(srv)[:2] == (0, 0):
            return


def result(srv, rid):
    m = np.zeros((GRID["ny"], GRID["nx"]), np.float32)
    state, n, _ = B.server_query(srv, rid, m)
    return state, m, n


def test_a_request_waits_for_room():
    """The second request's allocation fails while the first is active: it stays queued, and its
    result is the one it has alone."""
    srv = B.server_create(1 << 30, 8, 640)
    a = submit(srv, table(0))
    B.server_step(srv)
    B.server_test_fail_alloc(srv, 0, 1)
    b = submit(srv, table(1))
    active, queued, _ = B.server_step(srv)
    assert (active, queued) == (1, 1)
    finish(srv)
    for k, rid in ((0, a), (1, b)):
        state, m, n = result(srv, rid)
        ms, ns = plain(table(k), True)
        assert state == "done" and np.array_equal(m, ms) and n == ns
    B.server_destroy(srv)


@pytest.mark.parametrize("fails,state", [(1, "done"), (2, "failed")])
def test_a_request_alone_without_room(fails, state):
    """Nothing to wait for but what finished: tried again once, then failed; the next is served."""
    srv = B.server_create(1 << 30, 8, 640)
    B.server_test_fail_alloc(srv, 0, fails)
    a, b = submit(srv, table(0)), submit(srv, table(1))
    finish(srv)
    assert result(srv, a)[0] == state
    s, m, n = result(srv, b)
    ms, ns = plain(table(1), True)
    assert s == "done" and np.array_equal(m, ms) and n == ns
    B.server_destroy(srv)
