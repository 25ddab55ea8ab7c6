"""Stop, save, load and resume of the packed form where faults outgrow its last tier: such a fault
is a heavy one, whatever it was before the cycle that no tier held, and the checkpoint keeps all
its register diffs. Whole numbers: equal to the uninterrupted run and the oracle, or wrong."""
import numpy as np
import pytest

from paper_2508_16376_gb300.rtlfs import RTLFS_PENDING, Simulator, split
from test_gpu_checkpoint import _layout
from test_gpu_pack import _built, _case, _general  # noqa: F401  (_built: builds the library)

pytestmark = pytest.mark.gpu
COUNTERS = ("node_evals", "fault_cycles", "light_evals", "light_fault_cycles", "heavy_evals", "heavy_fault_cycles")


def _result(sim, **opts):
    res, loads = sim.run(want_load=True, **opts)
    return res[0], loads[0], sim.stats(), sim.mismatch_counts(0) if opts.get("no_drop") else None


@pytest.mark.parametrize("no_drop", [0, 1])
@pytest.mark.parametrize("light_cap", [1, 3])
@pytest.mark.parametrize("name", ["fan1100", "fan4200"])
def test_faults_beyond_the_last_tier_stop_and_resume(name, light_cap, no_drop):
    d, stim, f = _case(name)
    exp, _ = _general(name, bool(no_drop))
    opts = dict(window=64, light_cap=light_cap, heavy_frac=0.0, no_drop=no_drop)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        res, load, st, mism = _result(sim, **opts)
        assert st["heavy_form"] == 4 and st["promoted"] > 0
        for a, b in zip(split(res), exp[:3]):
            assert np.array_equal(a, b)
    deepest = 0
    for stop in (64, 128):
        with Simulator(0) as sim:
            sim.add(d, stim, f)
            first, _ = sim.run(stop_cycle=stop, **opts)
            blob = sim.checkpoint()
            done = first[0]["detected"] != RTLFS_PENDING
            assert np.array_equal(first[0][done], res[done])
            same = _result(sim, resume=1, **opts)
        off, F, n_live, n_carry, _ = _layout(blob)
        live = np.frombuffer(blob, np.uint32, n_live, off["live"])
        nreg = np.frombuffer(blob, np.uint8, F, off["st_nreg"])[live]
        assert n_live == 0 or nreg.max() <= (4 if light_cap == 1 else 8)
        if n_carry:
            deepest = max(deepest, int(np.frombuffer(blob, np.uint32, 4 * n_carry, off["carry"])[1::4].max()))
        with Simulator(0) as sim:
            sim.add(d, stim, f)
            sim.restore(blob)
            loaded = _result(sim, resume=1, **opts)
        for r, l, s, m in (same, loaded):
            assert np.array_equal(r, res) and np.array_equal(l, load)
            assert [s[k] for k in COUNTERS] == [st[k] for k in COUNTERS]
            if no_drop:
                assert np.array_equal(m, mism) and np.array_equal(m, exp[3])
    if no_drop:   # the case the test is for: more register diffs than the light form's state or a byte holds
        assert deepest > (1000 if name == "fan1100" else 8)
