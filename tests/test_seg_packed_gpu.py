"""Packed lists of busy links with measured outputs and vehicle types, over several packings: the
network has half as many groups of lanes again as the device's warps could hold at four blocks of
the move phase per SM, and the launches per step show that the lists are what runs."""
import numpy as np
import pytest

from paper_1807_01148_gb300 import scenarios as S

from .parity import compare, setup_pair
from .test_outputs_gpu import compare_outputs
from .test_seg_gpu import _grid

pytestmark = pytest.mark.gpu
FLEET = [(4.5, 1.0, 40.0), (12.0, 0.6, 22.0), (18.0, 0.5, 18.0)]


@pytest.mark.parametrize("types", [False, True])
@pytest.mark.parametrize("mode", [0, 1])
def test_outputs_and_types_on_packed_lists(types, mode):
    import oracle
    import torch
    from paper_1807_01148_gb300 import gbtraffic as G
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = int(np.ceil(np.sqrt(1.5 * 4 * 8 * sms * 32 / (4 * 2)))) + 1   # 4 n (n - 1) links of 2 lanes
    sc = _grid(n=n, n_trips=4000)
    g, o = setup_pair(sc, G.Sim, oracle.OracleSim)
    ty = np.random.default_rng(S.BASE_SEED).choice(3, sc["demand"]["n_trips"], p=(0.7, 0.2, 0.1)).astype(np.uint8)
    for q in (g, o):
        if types:
            q.set_vehicle_types(FLEET, ty)
        q.set_outputs(7, sample_every=5, per_window=3, max_windows=20)
    if mode:
        g.set_exec(mode=1, threads=256, blocks_per_sm=2)
    chunks = (1, 7, 9, 60, 100)
    n0, steps = g.launch_count(), sum(chunks)
    for k in chunks:
        g.step(k)
        o.step(k)
        compare(g, o, f"{k} steps", check_occ=False)
    if not mode:   # front and move, a sample every fifth step, a packing every eighth at least
        assert g.launch_count() - n0 - 2 * steps - len(range(0, steps, 5)) >= steps // 8
    compare_outputs(g, o, 7, "packed")
    assert o.counters()["arrived"] > 100
