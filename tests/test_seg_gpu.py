"""Stepping in link segments (networks of 2,048 lanes and more, and the persistent launch):
bit-exact against the oracle where the form can go wrong: stop signs, signals, merges and
departures on a mixed network, loop routes, links filled beyond their segment and beyond a
block's staging area, overlapping vehicles (lanes out of order), changes of the execution
mode mid-run, and a device-memory cap that leaves no room for the segments."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .parity import compare, run_lockstep, setup_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1807_01148_gb300 import gbtraffic
    return gbtraffic


def _grid(n=24, n_trips=3000, loop=False, lanes=2, seed=5):
    """A signalised grid of 2 lanes x 4 n (n - 1) links with explicit walks; loop: there and back."""
    sc = S.small_grid(n=n, n_trips=n_trips, lanes=lanes, seed=S.BASE_SEED + seed, window_steps=200)
    net = sc["network"]
    off, links = S.random_walk_routes(sc, 3, 9, seed=S.BASE_SEED + seed)
    if loop:
        nn = net["n_nodes"]
        key = net["link_from"].astype(np.int64) * nn + net["link_to"]
        by = np.argsort(key)
        twin = by[np.searchsorted(key[by], net["link_to"].astype(np.int64) * nn + net["link_from"])]
        legs = [np.r_[links[a:b], twin[links[a:b]][::-1]] for a, b in zip(off[:-1], off[1:])]
        off = np.r_[0, np.cumsum([len(q) for q in legs])].astype(np.int32)
        links = np.concatenate(legs).astype(np.int32)
        sc["params"]["loop_routes"] = 1
    sc["routes"] = dict(offsets=off, links=links)
    return sc


def _state(sc, on_link, per_lane, spacing):
    """Every trip whose walk begins on on_link is on it, per_lane vehicles in each of the first lanes."""
    off, links = sc["routes"]["offsets"], sc["routes"]["links"]
    n = sc["demand"]["n_trips"]
    lanes = int(sc["network"]["link_lanes"][on_link])
    put = np.flatnonzero(links[off[:-1]] == on_link)[: per_lane * lanes]
    st = dict(status=np.zeros(n, np.uint8), link=np.zeros(n, np.int32), lane=np.zeros(n, np.int32),
              cursor=np.zeros(n, np.int32), x=np.zeros(n, np.float32), v=np.zeros(n, np.float32))
    k = np.arange(len(put))
    st["status"][put], st["link"][put], st["lane"][put] = 1, on_link, k % lanes
    st["x"][put] = np.minimum(199.0, spacing * (k // lanes)).astype(np.float32)
    st["v"][put] = (3.0 * (k % 3)).astype(np.float32)
    return st


def _crowd(sc, link, n):
    """The first n trips walk from the given link on."""
    off, links = sc["routes"]["offsets"].copy(), sc["routes"]["links"]
    legs = [links[a:b] for a, b in zip(off[:-1], off[1:])]
    to, lf = sc["network"]["link_to"], sc["network"]["link_from"]
    nxt = int(np.flatnonzero((lf == to[link]) & (to != lf[link]))[0])
    for i in range(n):
        legs[i] = np.array([link, nxt], np.int32) if i % 3 else np.array([link], np.int32)
    sc["routes"] = dict(offsets=np.r_[0, np.cumsum([len(q) for q in legs])].astype(np.int32),
                        links=np.concatenate(legs).astype(np.int32))
    return sc


@pytest.mark.parametrize("mode", ["graph", "persistent", "switching"])
def test_mixed_network_bitexact(G, mode):
    import oracle
    sc = S.small_metro(nx=44, ny=34, n_trips=9000, steps=900, seed=S.BASE_SEED + 91)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if mode == "persistent":
        g.set_exec(mode=1, threads=512, blocks_per_sm=1)
    for k in range(6):
        if mode == "switching":
            g.set_exec(**([dict(mode=0), dict(mode=1, threads=256, blocks_per_sm=2)][k % 2]))
        run_lockstep(g, o, 150, 75)
    assert o.counters()["arrived"] > 100


@pytest.mark.parametrize("lanes", [1, 3, 8])
def test_loop_routes_bitexact(G, lanes):
    import oracle
    sc = _grid(loop=True, lanes=lanes, n=34 if lanes == 1 else 24)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    run_lockstep(g, o, 400, 100)


# more groups of lanes than resident warps: packed lists kept for several steps.  Chunks of 1, 7,
# 8, 9 and more steps begin and end at every age of the lists; walks enter links that are not
# in them, trips depart up to step 200, one link is left to a whole block.
@pytest.mark.parametrize("n,lanes,mode", [(128, 2, 0), (104, 3, 0), (128, 2, 1)])
def test_packed_lists_bitexact(G, n, lanes, mode):
    import oracle
    sc = _crowd(_grid(n=n, lanes=lanes, n_trips=5000, loop=mode == 1), 77, 120)
    sc["params"]["loop_routes"] = 0
    sc["init_state"] = _state(sc, 77, 47, 4.2)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if mode:
        g.set_exec(mode=1, threads=256, blocks_per_sm=2)
    for total, chunk in [(3, 1), (14, 7), (8, 8), (18, 9), (21, 21), (100, 50), (130, 130)]:
        run_lockstep(g, o, total, chunk)
    assert o.counters()["arrived"] > 20


# a dense network, several runs per warp, with links that hold as many vehicles as a whole block
# is set to, or a few more, and lose some: no second warp may take them in the same step
@pytest.mark.parametrize("mode", [0, 1])
def test_links_about_the_staging_area_bitexact(G, mode):
    import oracle
    sc = S.small_grid(n=128, n_trips=580000, lanes=3, seed=S.BASE_SEED + 6, window_steps=200)
    net = sc["network"]
    lf, lt = net["link_from"].astype(np.int64), net["link_to"].astype(np.int64)
    n_links, n = len(lf), sc["demand"]["n_trips"]
    out = np.argsort(lf, kind="stable")
    k = np.searchsorted(lf[out], lt)
    nxt = np.where(lt[out[k]] == lf, out[np.minimum(k + 1, n_links - 1)], out[k])   # not back
    crowded = np.arange(50, n_links, 97)
    many = 93 + np.arange(len(crowded)) % 4
    at = np.concatenate([np.repeat(crowded, many), np.tile(np.setdiff1d(np.arange(n_links), crowded), 9)])[:n]
    sc["routes"] = dict(offsets=3 * np.arange(n + 1, dtype=np.int32),
                        links=np.stack([at, nxt[at], nxt[nxt[at]]], 1).reshape(-1).astype(np.int32))
    order = np.argsort(at, kind="stable")
    rank = np.empty(n, np.int64)
    rank[order] = np.arange(n) - np.searchsorted(at[order], at[order])
    x = 199.0 - 6.0 * (rank // 3)
    sc["init_state"] = dict(status=np.ones(n, np.uint8), link=at.astype(np.int32), lane=(rank % 3).astype(np.int32),
                            cursor=np.zeros(n, np.int32), x=x.astype(np.float32), v=np.full(n, 9.0, np.float32))
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if mode:
        g.set_exec(mode=1, threads=256, blocks_per_sm=1)
    run_lockstep(g, o, 12, 4)


# vehicles per lane of a 200 m link: up to a warp's staging area, past it, past the link's
# segment (84 + 2 vehicles), past a block's staging area
@pytest.mark.parametrize("per_lane,spacing", [(40, 5.0), (46, 4.3), (47, 4.2), (120, 1.5), (560, 0.3), (60, 0.0)])
def test_crowded_link_bitexact(G, per_lane, spacing):
    import oracle
    sc = _crowd(_grid(), 77, 2 * per_lane)
    sc["init_state"] = _state(sc, 77, per_lane, spacing)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    run_lockstep(g, o, 60, 12)
    g.set_exec(mode=1, threads=256, blocks_per_sm=1)
    run_lockstep(g, o, 40, 20)


def test_memory_cap_keeps_stepping(G):
    # a cap that the handle and its routes just fit: the segments do not, the results are the same
    import oracle
    sc = _grid(n_trips=800)
    lo, hi = 1 << 16, 1 << 24
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        try:
            G.setup(dict(sc, params=dict(sc["params"], max_device_bytes=mid))).close()
            hi = mid
        except G.SimError:
            lo = mid
    cap = hi + 65536   # what reading the state takes
    g, o = setup_pair(dict(sc, params=dict(sc["params"], max_device_bytes=cap)), G.Sim, oracle.OracleSim)
    run_lockstep(g, o, 60, 30, check_occ=False)
    compare(g, o, "capped", check_occ=False)
