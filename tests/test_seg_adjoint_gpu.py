"""The calibration adjoint on a network large enough for packed lists of busy links (more groups
of lanes than the resident warps of the move phase): whatever the checkpoint interval, every
replayed segment packs its lists before its first step, so the gradient equals the oracle's,
on a fresh handle and again on the same one."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .test_seg_gpu import _grid

pytestmark = pytest.mark.gpu
KEYS = ("v0", "T", "a", "b", "s0")


@pytest.fixture(scope="module")
def case():
    import oracle
    steps, every = 600, 20
    sc = _grid(n=160, n_trips=4000)   # 6,360 groups; 3 blocks of 8 warps on each of 152 SMs are 3,648
    r = sc["routes"]
    p = {k: np.array(sc["params"][k], np.float64) for k in KEYS}
    o = oracle.OracleSim(sc)
    o.set_routes(r["offsets"], r["links"])
    o.set_class_params(p["v0"], 1.2 * p["T"], 1.1 * p["a"], p["b"], p["s0"])
    tgt = o.observe(steps, every)
    o = oracle.OracleSim(sc)
    o.set_routes(r["offsets"], r["links"])
    grad, loss = o.adjoint(steps, every, tgt, 1)
    return sc, steps, every, tgt, np.asarray(grad).reshape(1, 5), loss


@pytest.mark.parametrize("seg", [5, 10, 64])
def test_adjoint_on_packed_lists(case, seg):
    from paper_1807_01148_gb300 import gbtraffic as G
    sc, steps, every, tgt, og, oloss = case
    n = sc["demand"]["n_trips"]
    g = G.Sim(sc)
    g.set_routes(sc["routes"]["offsets"], sc["routes"]["links"])
    start = dict(status=np.zeros(n, np.uint8), link=np.zeros(n, np.int32), lane=np.zeros(n, np.int32),
                 cursor=np.zeros(n, np.int32), x=np.zeros(n, np.float32), v=np.zeros(n, np.float32))
    for again in range(2):
        if again:
            g.write_state(start)
        grad, loss = g.adjoint(steps, every, tgt, 1, checkpoint_every=seg)
        assert abs(loss - oloss) <= 1e-12 * abs(oloss)
        # summation order only, as in the adjoint's test on a small network
        assert np.allclose(grad, og, rtol=1e-9, atol=1e-9 * np.abs(og).max()), (again, grad, og)
    n0 = g.launch_count()
    g.step(8)
    assert g.launch_count() - n0 == 2 * 8 + 1   # lists were packed: this network is in packed form
