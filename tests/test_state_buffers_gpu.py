"""sim_read_state into device buffers that start on any element: trip counts around the
vectors of four and buffers off their alignment read the same as the oracle's state, in both
forms of the state (sorted: small grid; segments: persistent launch)."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .parity import STATE_KEYS, setup_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("n_trips", [1, 3, 4, 5, 602, 1023])
def test_any_alignment(n_trips, persistent):
    import oracle
    import torch
    from paper_1807_01148_gb300 import gbtraffic as G
    sc = S.small_grid(n=5, n_trips=n_trips, steps=100, seed=S.BASE_SEED + n_trips, window_steps=120)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    if persistent:
        g.set_exec(mode=1, threads=256, blocks_per_sm=1)
    g.step(70)
    o.step(70)
    want = o.state()
    for shift in (0, 1, 2):
        raw = {k: torch.full((n_trips + 4,), 77, dtype=torch.from_numpy(want[k]).dtype, device="cuda")
               for k in STATE_KEYS}
        g.state_device({k: t[shift:] for k, t in raw.items()}, G.F_ALL)
        for k, t in raw.items():
            got = t.cpu().numpy()
            assert np.array_equal(got[shift:shift + n_trips], want[k]), (k, shift)
            assert (got[:shift] == 77).all() and (got[shift + n_trips:] == 77).all(), (k, shift)
