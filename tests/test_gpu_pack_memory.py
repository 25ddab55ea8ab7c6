"""A device without room for the packed form's pools: the campaign runs on the light and heavy
kernels, as it does when they are named, and on the packed form again once there is room."""
import numpy as np
import pytest

from paper_2508_16376_gb300 import synth
from paper_2508_16376_gb300.rtlfs import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(), dict(no_drop=1), dict(use_graph=1)])
def test_run_without_room_for_the_pools(opts):
    import torch
    from paper_2508_16376_gb300 import build
    build.build()
    d = synth.gen_datapath_fsm(5, 1000, 300, 16, 16, [8], 0.8, 8, 64)
    u = synth.fault_universe(d)
    f = u.take(np.resize(np.arange(len(u)), 60000))   # 7 pools of 16M register diffs, 12 bytes each: 1.4 GB
    stim = synth.stimulus(d, 70, 3, 0.1)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        ref, rl = sim.run(want_load=True, heavy_form=1, no_drop=opts.get("no_drop", 0))   # its memory stays with the context
        free, _ = torch.cuda.mem_get_info()
        keep = 600 << 20
        hog = torch.empty(max(0, free - keep), dtype=torch.uint8, device="cuda")
        try:
            got, gl = sim.run(want_load=True, **opts)
            form = sim.stats()["heavy_form"]
        finally:
            del hog
            torch.cuda.empty_cache()
        again, al = sim.run(want_load=True, **opts)
        assert form in (1, 2, 3) and sim.stats()["heavy_form"] == 4
    for r, l in ((got, gl), (again, al)):
        assert np.array_equal(r[0], ref[0]) and np.array_equal(l[0], rl[0])


def test_run_without_room_for_the_crowds():
    """Room for the packed form but not for a slot per resident warp of the heavy kernel: the tiers take every fault."""
    import torch
    from paper_2508_16376_gb300 import build
    build.build()
    d = synth.gen_datapath_fsm(5, 60000, 64, 16, 16, [8], 0.8, 24, 64)
    u = synth.fault_universe(d)
    f = u.take(np.sort(np.random.default_rng(2).choice(len(u), 3000, replace=False)))
    stim = synth.stimulus(d, 70, 3, 0.1)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        ref, rl = sim.run(want_load=True, heavy_form=1)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(max(0, free - (1200 << 20)), dtype=torch.uint8, device="cuda")   # the slots take 3 GB
        try:
            got, gl = sim.run(want_load=True)
            form = sim.stats()["heavy_form"]
            again, al = sim.run(want_load=True, use_graph=1, window=64)
        finally:
            del hog
            torch.cuda.empty_cache()
        roomy, ml = sim.run(want_load=True, use_graph=1, window=64)
        assert form == 4 and sim.stats()["heavy_form"] == 4
    for r, l in ((got, gl), (again, al), (roomy, ml)):
        assert np.array_equal(r[0], ref[0]) and np.array_equal(l[0], rl[0])
