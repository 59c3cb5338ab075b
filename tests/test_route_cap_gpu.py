"""Trip planning and written states under a device-memory cap (sim_params.max_device_bytes)."""
import time

import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .parity import run_lockstep
from .test_seg_gpu import _grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1807_01148_gb300 import gbtraffic
    return gbtraffic


def _capped(sc, cap):
    return dict(sc, params=dict(sc["params"], max_device_bytes=cap))


def _least(G, sc, lo=1 << 10, hi=1 << 28):
    """The least cap under which the handle can be created."""
    while hi - lo > 1:
        mid = (lo + hi) // 2
        try:
            G.Sim(_capped(sc, mid)).close()
            hi = mid
        except G.SimError:
            lo = mid
    return hi


def _planning(sc, trees):
    """Bytes that planning needs at least: link arrays of 4 words per link, the nodes' tables, 32
    bytes per node and tree in flight, 96 links per trip."""
    nn, nl, nt = sc["network"]["n_nodes"], len(sc["network"]["link_from"]), sc["demand"]["n_trips"]
    n_org = len(np.unique(sc["demand"]["origin"]))
    n_cta = min(n_org, trees)
    return (4 * (4 * nl + 3 * (nn + 1) + n_org + 1 + 2 * nt) + n_cta * (32 * nn + 8) + 4
            + 4 * max(1024, 96 * nt))


@pytest.mark.parametrize("room", [0, 4, 1 << 20], ids=["links by id", "by id, a little more", "pairs"])
def test_least_room(G, room):
    import oracle
    sc = S.small_grid(n=20, n_trips=200, steps=100)
    g, o = G.Sim(_capped(sc, _least(G, sc) + _planning(sc, 1 << 30) + room)), oracle.OracleSim(sc)
    g.route()
    o.route()
    (go, gl), (oo, ol) = g.routes(), o.routes()
    assert np.array_equal(go, oo) and np.array_equal(gl, ol)


def test_assignment_keeps_the_segments(G):
    # beside the segments (about 20 MB) there is room for four trees per SM, not for eight: the
    # running state stays in the segments (2 launches a step, 7 in the sorted form)
    import torch
    sc = S.small_grid(n=40, n_trips=8000, steps=100)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert len(np.unique(sc["demand"]["origin"])) > 8 * sms
    g = G.Sim(_capped(sc, _least(G, sc) + _planning(sc, 4 * sms) + (30 << 20)))
    g.route()
    g.step(4)
    n0 = g.launch_count()
    g.step(4)
    assert g.launch_count() - n0 == 2 * 4
    g.assign_static(np.full(len(sc["network"]["link_from"]), 1800.0), max_iter=1)
    n0 = g.launch_count()
    g.step(4)
    assert g.launch_count() - n0 == 2 * 4


def _launches(g):
    n0 = g.launch_count()
    g.step(4)
    return g.launch_count() - n0


def _write_time(G, sc, cap):
    """Seconds of a written state, and the launches of four steps after it."""
    n = sc["demand"]["n_trips"]
    st = dict(status=np.zeros(n, np.uint8), link=np.zeros(n, np.int32), lane=np.zeros(n, np.int32),
              cursor=np.zeros(n, np.int32), x=np.zeros(n, np.float32), v=np.zeros(n, np.float32))
    g = G.Sim(_capped(sc, cap))
    g.set_routes(sc["routes"]["offsets"], sc["routes"]["links"])
    took = []
    for _ in range(12):
        t = time.perf_counter()
        g.write_state(st)
        took.append(time.perf_counter() - t)
    return np.median(took), _launches(g)


def test_written_state_without_room_for_segments(G):
    # finding no room for the segments costs a written state no more than laying them out does
    sc = _grid(n=128, lanes=3, n_trips=2000)
    free, launches = _write_time(G, sc, 0)
    assert launches == 2 * 4 + 1
    capped, launches = _write_time(G, sc, _least(G, sc) + (4 << 20))
    assert launches == 7 * 4
    assert capped < 2.0 * free, (capped, free)


def test_written_state_with_just_room_for_segments(G):
    # the segments are not made where the arrays of a written state would push them out again
    sc = _grid(n=128, lanes=3, n_trips=20000)
    lo = hi = _least(G, sc)
    hi += 1 << 30
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        g = G.Sim(_capped(sc, mid))
        try:
            g.set_routes(sc["routes"]["offsets"], sc["routes"]["links"])
            segments = _launches(g) == 2 * 4 + 1
        except G.SimError:
            segments = False
        g.close()
        lo, hi = (lo, mid) if segments else (mid, hi)
    free, _ = _write_time(G, sc, 0)
    capped, _ = _write_time(G, sc, hi)
    assert capped < 2.0 * free, (capped, free)


def test_routes_that_do_not_fit_leave_none(G):
    # the old routes are gone by then: stepping is refused until there are new ones
    import oracle
    sc = _grid(n=24, n_trips=3000)
    short = sc["routes"]
    off, links = S.random_walk_routes(sc, 400, 600, seed=S.BASE_SEED)
    g = G.Sim(_capped(sc, _least(G, sc) + (1 << 20)))
    g.set_routes(short["offsets"], short["links"])
    g.step(10)
    with pytest.raises(G.SimError) as e:
        g.set_routes(off, links)
    assert e.value.code == G.SIM_ENOMEM
    with pytest.raises(G.SimError) as e:
        g.step(1)
    assert e.value.code == G.SIM_ESTATE
    g.set_routes(short["offsets"], short["links"])
    o = oracle.OracleSim(sc)
    o.set_routes(short["offsets"], short["links"])
    run_lockstep(g, o, 20, 10, check_occ=False)
