"""More faults in the packed form's last tiers than they take at a time: those go to the heavy
kernel, window by window. Results, loads, no-drop counts and budgets equal the light and heavy
kernels', and the division of the evaluations into light and heavy does not depend on where a
campaign was stopped and resumed. Whole numbers: equal or wrong."""
import functools

import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import synth
from paper_2508_16376_gb300.rtlfs import Simulator, make_opts, rtlfs_run, split
from paper_2508_16376_gb300.synth import ADD, OR, SLICE, XOR, _Builder
from test_gpu_pack import _built  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


def ladder(width, levels, couple):
    """`levels` rows of `width` nodes between registers; one node in `couple` also reads its neighbour (0: none)."""
    b = _Builder([8] * 4, [8] * width)
    row = [b.reg_net(i) for i in range(width)]
    for k in range(levels):
        row = [b.add((XOR, ADD, OR, XOR)[(i + k) % 4], 8, row[i],
                     row[(i + 1) % width] if couple and (k * 7 + i) % couple == 0 else (i + k) % 4) for i in range(width)]
    for i in range(width):
        b.reg_d[i] = row[i]
    return b.finish("ladder", [b.add(SLICE, 1, row[i], imm=3) for i in range(0, width, max(1, width // 4))])


# Narrow levels (the last two tiers take 2 and 32 faults per SM) and wide ones (4 and 64): faults beyond
# the third tier's 64 x 152, between the two, and just beyond the last tier's.
CASES = {"narrow": (ladder, (4, 60, 3), 12000), "narrow_few": (ladder, (4, 60, 3), 700), "wide": (ladder, (140, 12, 2), 12000),
         "wide_few": (ladder, (140, 12, 2), 1500)}


@functools.lru_cache(maxsize=None)
def _case(name):
    make, args, F = CASES[name]
    d = make(*args)
    T = 150
    u = synth.fault_universe(d, include_inputs=True)
    f = u.take(np.sort(np.random.default_rng(4).choice(len(u), F - 100, replace=F - 100 > len(u))))
    return d, synth.stimulus(d, T, 7, 0.2), synth.Faults.concat([f, synth.transient_faults(d, 100, T, 8)])


@functools.lru_cache(maxsize=None)
def _general(name, no_drop):
    d, stim, f = _case(name)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        res, loads = sim.run(want_load=True, heavy_form=1, no_drop=no_drop)
        mism = sim.mismatch_counts(0) if no_drop else None
    pick = np.sort(np.random.default_rng(9).choice(len(f), 150, replace=False))
    exp = oracle.fault_sim_ex(d, stim, f.take(pick), threads=8, no_drop=bool(no_drop))
    for a, b in zip(split(res[0]), exp[:3]):
        assert np.array_equal(a[pick], b)
    if no_drop:
        assert np.array_equal(mism[pick], exp[3])
    return res[0], loads[0], mism


@pytest.mark.parametrize("no_drop", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_crowds_equal_general_path(name, no_drop):
    res, load, mism = _general(name, no_drop)
    d, stim, f = _case(name)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        for opts in (dict(), dict(window=48, light_cap=1), dict(window=128, use_graph=1), dict(window=128, use_graph=1),
                     dict(heavy_block=64, heavy_ctas=40), dict(window=64, heavy_frac=0.3)):
            r, l = sim.run(want_load=True, no_drop=no_drop, **opts)
            assert sim.stats()["heavy_form"] == 4
            assert np.array_equal(r[0], res) and np.array_equal(l[0], load), opts
            if no_drop:
                assert np.array_equal(sim.mismatch_counts(0), mism), opts


@pytest.mark.parametrize("no_drop", [0, 1])
@pytest.mark.parametrize("name", ["narrow", "wide_few"])
def test_crowds_stop_and_resume(name, no_drop):
    res, load, _ = _general(name, no_drop)
    d, stim, f = _case(name)
    opts = dict(window=64, light_cap=1, heavy_frac=0.0, no_drop=no_drop)
    keys = ("node_evals", "fault_cycles", "light_evals", "light_fault_cycles", "heavy_evals", "heavy_fault_cycles")
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        sim.run(**opts)
        full = sim.stats()
        sim.run(stop_cycle=64, **opts)
        blob = sim.checkpoint()
        for again in (False, True):
            if again:
                sim.restore(blob)
            r, l = sim.run(want_load=True, resume=1, **opts)
            st = sim.stats()
            assert np.array_equal(r[0], res) and np.array_equal(l[0], load)
            assert [st[k] for k in keys] == [full[k] for k in keys]


def test_crowds_budget():
    d, stim, f = _case("narrow")
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        for budget in (40, 300, 2000, 9000):
            for window in (0, 128):
                (a, la, ra), (b, lb, rb) = [rtlfs_run(sim.ctx, sim.n_faults, make_opts(fault_budget=budget, window=window, heavy_form=form),
                                                      True, check=False) for form in (1, 0)]
                assert ra == rb and np.array_equal(a[0], b[0]) and np.array_equal(la[0], lb[0]), (budget, window)
