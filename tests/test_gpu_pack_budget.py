"""The work budget in the packed form stops a fault after the cycle that exceeds it, also where
that cycle ends one of the packed form's own windows: results, loads and counters are those of the light and
heavy kernels with the same options, for budgets that run out all over the stimulus."""
import numpy as np
import pytest

from paper_2508_16376_gb300.rtlfs import Simulator, make_opts, rtlfs_run
from test_gpu_pack import _built, _case  # noqa: F401  (_built: builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("no_drop", [0, 1])
@pytest.mark.parametrize("window", [0, 48, 64, 128])
@pytest.mark.parametrize("name", ["fan5", "fan40", "fan1100", "fan4200", "fsm"])
def test_budget_at_every_cycle(name, window, no_drop):
    d, stim, f = _case(name)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        _, full, _ = rtlfs_run(sim.ctx, sim.n_faults, make_opts(heavy_form=1, no_drop=no_drop), True)
        # a budget between any two loads that the faults reach, spread over their range
        budgets = np.unique(np.geomspace(1, max(2, int(full[0].max())), 24).astype(np.int64))
        hits = 0
        for budget in budgets.tolist():
            out = []
            for form in (1, 0):
                r, l, rc = rtlfs_run(sim.ctx, sim.n_faults, make_opts(fault_budget=budget, heavy_form=form, window=window,
                                                                      no_drop=no_drop), True, check=False)
                out.append((r[0], l[0], rc, sim.mismatch_counts(0) if no_drop else np.zeros(1)))
            assert out[0][2] == out[1][2]
            for a, b in zip(out[0][:2] + out[0][3:], out[1][:2] + out[1][3:]):
                assert np.array_equal(a, b), budget
            hits += int((out[0][0]["detected"] == 255).sum())
        assert hits > 0


def test_budget_under_graph_replay():
    """One context, the same budget under windows that share the packed form's own: each run stops faults as
    the light and heavy kernels do under its window, captured or replayed."""
    d, stim, f = _case("fan5")
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        _, full, _ = rtlfs_run(sim.ctx, sim.n_faults, make_opts(heavy_form=1), True)
        budget = max(1, int(np.median(full[0][full[0] > 0])) // 2)
        for window in (0, 128, 0, 64, 128):
            ref, rl, _ = rtlfs_run(sim.ctx, sim.n_faults, make_opts(fault_budget=budget, heavy_form=1, window=window), True, check=False)
            got, gl, _ = rtlfs_run(sim.ctx, sim.n_faults, make_opts(fault_budget=budget, window=window, use_graph=1), True, check=False)
            assert np.array_equal(got[0], ref[0]) and np.array_equal(gl[0], rl[0]), window
