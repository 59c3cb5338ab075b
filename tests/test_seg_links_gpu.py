"""Links in segments whose vehicles come and go all at once, bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .parity import compare, run_lockstep, setup_pair
from .test_outputs_gpu import compare_outputs
from .test_seg_gpu import _grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1807_01148_gb300 import gbtraffic
    return gbtraffic


def emptied_link(n, second):
    """100 vehicles at the end of their last link (more than a warp stages) and one that comes
    two steps later: a departure, or a vehicle that crosses into the link.  Nothing else is on
    the road, so nobody works on the link in between."""
    sc = _grid(n=n, n_trips=101)
    net = sc["network"]
    lf, lt = net["link_from"].astype(np.int64), net["link_to"].astype(np.int64)
    # a link and one before it, straight on, in another group of 32 lanes (2 lanes each)
    L, F, out = next((b, a, c) for b in range(40, len(lf)) for a in np.flatnonzero(lt == lf[b])
                     if lt[b] - lf[b] == lt[a] - lf[a] and a // 16 != b // 16
                     for c in np.flatnonzero(lf == lt[b])[:1] if lt[c] != lf[b])
    if second == "departs":
        legs = [[L]] * 100 + [[L, out]]
    else:
        legs = [[L]] * 100 + [[F, L, out]]
    sc["routes"] = dict(offsets=np.r_[0, np.cumsum([len(q) for q in legs])].astype(np.int32),
                        links=np.concatenate(legs).astype(np.int32))
    sc["demand"]["depart_step"][:] = 0
    sc["demand"]["depart_step"][100] = 2
    k = np.arange(101)
    st = dict(status=np.ones(101, np.uint8), link=np.full(101, L, np.int32), lane=(k % 2).astype(np.int32),
              cursor=np.zeros(101, np.int32), x=np.full(101, net["link_length_m"][L], np.float32),
              v=np.full(101, 9.0, np.float32))
    if second == "departs":
        st["status"][100] = st["link"][100] = st["x"][100] = st["v"][100] = 0
    else:
        st["link"][100], st["x"][100] = F, net["link_length_m"][F] - 13.0
    st["lane"][100] = 0
    sc["init_state"] = st
    return sc, L


@pytest.mark.parametrize("n", [24, 160], ids=["parts", "packed"])
@pytest.mark.parametrize("second", ["departs", "crosses"])
@pytest.mark.parametrize("mode", [0, 1])
def test_link_emptied_by_a_block_bitexact(G, n, second, mode):
    import oracle
    sc, L = emptied_link(n, second)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if mode:
        g.set_exec(mode=1, threads=256, blocks_per_sm=1)
    run_lockstep(g, o, 1, 1)
    assert o.counters()["arrived"] == 100   # the link is empty
    run_lockstep(g, o, 1, 1)
    assert not (o.state()["link"][o.state()["status"] == 1] == L).any()
    run_lockstep(g, o, 1, 1)
    assert (o.state()["link"][o.state()["status"] == 1] == L).sum() == 1   # comes in the third step
    run_lockstep(g, o, 20, 5)


def filling_link(most, depart):
    """A link that holds as many vehicles (overlapping) as its segment or a block's staging area
    takes, and one more from step `depart` + 1 on."""
    sc = _grid(n=24, n_trips=most + 1)
    net = sc["network"]
    lf, lt = net["link_from"].astype(np.int64), net["link_to"].astype(np.int64)
    # an east-west link whose head stays green north-south for the first 12 steps
    phase = -net["signal_offset_ds"] % net["signal_cycle_ds"]
    red = (phase + 12 * 5 < net["signal_green_ds"])[lt]
    ew = net["node_y_dm"][lf] == net["node_y_dm"][lt]
    L = int(np.flatnonzero(red & ew)[5])
    out = int(np.flatnonzero((lf == lt[L]) & (lt != lf[L]))[0])
    n = most + 1
    sc["routes"] = dict(offsets=2 * np.arange(n + 1, dtype=np.int32), links=np.tile([L, out], n).astype(np.int32))
    sc["demand"]["depart_step"][:] = 0
    sc["demand"]["depart_step"][most] = depart
    k = np.arange(n)
    st = dict(status=np.ones(n, np.uint8), link=np.full(n, L, np.int32), lane=(k % 2).astype(np.int32),
              cursor=np.zeros(n, np.int32), x=(199.0 - 170.0 * (k // 2) / (most // 2)).astype(np.float32),
              v=np.zeros(n, np.float32))
    for q in ("status", "link", "lane", "x"):
        st[q][most] = 0
    sc["init_state"] = st
    return sc, L


# 200 m of 2 lanes hold 84 vehicles of 5 m and 2 more that a step may bring; a block stages 1,024
@pytest.mark.parametrize("most", [84, 1022])
@pytest.mark.parametrize("depart", [0, 1])
@pytest.mark.parametrize("how", ["graph", "persistent", "timed"])
def test_sample_of_a_step_that_did_not_fit(G, most, depart, how):
    import oracle
    sc, L = filling_link(most, depart)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    for q in (g, o):
        q.set_outputs(7, sample_every=1, per_window=3, max_windows=4)
    if how == "persistent":
        g.set_exec(mode=1, threads=256, blocks_per_sm=1)
    o.step(depart + 1)
    assert (o.state()["link"] == L).sum() == most + 1   # the next step does not fit
    o.step(12 - depart - 1)
    g.step_timed(12) if how == "timed" else g.step(12)
    compare(g, o, "filled")
    compare_outputs(g, o, 7, "filled")


# a segment that ran full in a call that times, taps or tries steps does not keep later steps out
# of the segments (2 launches a step there, 7 in the sorted form)
@pytest.mark.parametrize("call", ["timed", "adjoint", "autotune"])
def test_full_segment_is_forgotten(G, call):
    import oracle
    sc, L = filling_link(1022 if call == "autotune" else 84, 7 if call == "autotune" else 1)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if call == "timed":
        g.step_timed(4)
        o.step(4)
    elif call == "adjoint":
        tgt = np.full((2, sc["demand"]["n_trips"]), 100.0)
        grad, loss = g.adjoint(10, 5, tgt, 1)
        og, oloss = o.adjoint(10, 5, tgt, 1)
        assert abs(loss - oloss) <= 1e-12 * oloss
        assert np.allclose(grad, np.reshape(og, (1, 5)), rtol=1e-9, atol=1e-9 * np.abs(og).max())
    else:
        g.autotune(10)   # back to the state before the link runs full
        g.set_exec(mode=0)
    n0 = g.launch_count()
    g.step(4)
    assert g.launch_count() - n0 == 2 * 4
    o.step(4)
    compare(g, o, call)
