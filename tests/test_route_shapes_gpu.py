"""Trip planning on networks that reach the edges of the search kernel: a chain (paths longer
than a group's share of the note space), a hub with more spokes than the near queue holds in
shared memory and more in-links than a group of threads tests at once, parallel links of
equal cost, one destination next to the origin and one at the far end.  Routes equal the
oracle's link by link."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


def _scenario(n, lf, lt, length, o, d):
    net = S._net(n, np.arange(n) * 10, (np.arange(n) * 37) % 1000, np.zeros(n), np.zeros(n), np.full(n, 600),
                 np.full(n, 300), lf, lt, np.asarray(length, float), np.full(len(lf), 10.0), np.ones(len(lf)),
                 np.zeros(len(lf)))
    return dict(name="shape", network=net, demand=S._demand(o, d, np.zeros(len(o))), params=S.default_params(1))


def _chain(n):
    a = np.arange(n - 1)
    lf, lt = np.r_[a, a + 1], np.r_[a + 1, a]
    return _scenario(n, lf, lt, 50.0 + (np.arange(len(lf)) * 7919) % 400, [0, 0, n - 1, n // 2], [n - 1, 1, 0, n - 2])


def _hub(spokes):
    # hub 0 <-> middle nodes (in-degree limit 255) <-> leaves, every road twice with equal cost
    mid = 60
    m = 1 + np.arange(mid)
    leaf = 1 + mid + np.arange(spokes)
    up = 1 + np.arange(spokes) % mid
    lf = np.r_[np.zeros(mid), m, up, leaf, up, leaf].astype(int)
    lt = np.r_[m, np.zeros(mid), leaf, up, leaf, up].astype(int)
    length = np.r_[np.full(2 * mid, 100.0), np.full(4 * spokes, 200.0)]
    o = [0, leaf[0], leaf[5], leaf[7], 0]
    d = [leaf[-1], leaf[-2], 0, leaf[7 + mid], leaf[3]]
    return _scenario(1 + mid + spokes, lf, lt, length, o, d)


@pytest.mark.parametrize("make", [lambda: _chain(9), lambda: _chain(700), lambda: _hub(100), lambda: _hub(6000)],
                         ids=["chain9", "chain700", "hub100", "hub6000"])
def test_routes_equal_oracle(make):
    import oracle
    from paper_1807_01148_gb300 import gbtraffic as G
    sc = make()
    g, o = G.Sim(sc), oracle.OracleSim(sc)
    g.route()
    o.route()
    (go, gl), (oo, ol) = g.routes(), o.routes()
    assert np.array_equal(go, oo) and np.array_equal(gl, ol)
