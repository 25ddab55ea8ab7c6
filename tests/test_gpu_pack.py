"""The packed faulty-machine form against the light and heavy kernels (the general path, chosen by
naming a heavy form) and the oracle: results, evaluation counts and no-drop counts, on designs
whose cones, fan-outs and latched registers sit at the edges of the tiers' tables. Everything
is whole numbers: equal or wrong."""
import functools

import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import synth
from paper_2508_16376_gb300.rtlfs import Simulator, split
from paper_2508_16376_gb300.synth import AND, EQ, LT, MUX2, NOT, SLICE, XOR, _Builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_16376_gb300 import build
    build.build()
    oracle.build()


def fan(k, r):
    """A control register whose bit selects k MUX2 nodes; the first r of them are latched, and the
    registers feed back through the datapath. One node in sixteen reaches the output, so that
    faults live on for some cycles with k dirty nodes and up to r register diffs."""
    b = _Builder([8, 8, 1], [1] + [8] * r)
    s = b.reg_net(0)
    m = [b.add(MUX2, 8, s, i % 2, b.reg_net(1 + i % r) if r else (i + 1) % 2) for i in range(k)]
    x = [b.add(XOR, 8, m[i], b.reg_net(1 + (7 * i) % r) if r else 1) for i in range(min(k, 40))]
    acc = x[0]
    for i in range(16, len(x), 16):
        acc = b.add(AND, 8, acc, x[i])
    hit = b.add(EQ, 1, b.add(SLICE, 2, acc, imm=1), b.add(SLICE, 2, 0, imm=3))
    b.reg_d[0] = b.add(XOR, 1, 2, b.add(LT, 1, 0, 1))
    for i in range(r):
        b.reg_d[1 + i] = m[i % k]
    return b.finish(f"fan{k}_{r}", [hit])


def deep(n):
    """n levels: one more than the tags name takes the light and heavy kernels."""
    b = _Builder([4], [4])
    x = b.reg_net(0)
    for i in range(n):
        x = b.add(NOT if i % 3 else XOR, 4, x, 0)
    b.reg_d[0] = x
    return b.finish(f"deep{n}", [b.add(SLICE, 1, x, imm=2)])


DESIGNS = {"fan1": lambda: fan(1, 1), "fan4": lambda: fan(4, 4), "fan5": lambda: fan(5, 5), "fan8": lambda: fan(8, 3),
           "fan9": lambda: fan(9, 0), "fan40": lambda: fan(40, 33), "fan130": lambda: fan(130, 129),
           "fan520": lambda: fan(520, 130), "fan1100": lambda: fan(1100, 1030), "fan4200": lambda: fan(4200, 40),
           "deep4094": lambda: deep(4093), "deep4096": lambda: deep(4096),
           "fsm": lambda: synth.gen_datapath_fsm(8, 1500, 150, 16, 16, [8], 0.8, 12, 64)}


@functools.lru_cache(maxsize=None)
def _case(name):
    d = DESIGNS[name]()
    T = 9 if name.startswith("deep") else 141   # two whole windows of 64 cycles and a rest
    stim = synth.stimulus(d, T, 5, 0.2)
    u = synth.fault_universe(d, include_inputs=True)
    rng = np.random.default_rng(3)
    idx = np.sort(rng.choice(len(u), min(len(u), 240), replace=False))
    ctl = np.nonzero(u.net == d.n_in)[0]        # the control register's own faults are always there
    f = synth.Faults.concat([u.take(np.unique(np.concatenate([idx, ctl]))), synth.port_faults(d),
                             synth.transient_faults(d, 40, T, 6)])
    return d, stim, f


@functools.lru_cache(maxsize=None)
def _general(name, no_drop):
    d, stim, f = _case(name)
    exp = oracle.fault_sim_ex(d, stim, f, threads=8, no_drop=no_drop)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        res, loads = sim.run(want_load=True, heavy_form=1, no_drop=int(no_drop))
        assert sim.stats()["heavy_form"] == 1
    for a, b in zip(split(res[0]), exp[:3]):
        assert np.array_equal(a, b)
    return exp, loads[0]


@pytest.mark.parametrize("no_drop", [False, True])
@pytest.mark.parametrize("name", sorted(DESIGNS))
def test_packed_form_equals_general_path(name, no_drop):
    d, stim, f = _case(name)
    exp, gload = _general(name, no_drop)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        for opts in (dict(), dict(window=128, light_cap=1), dict(window=48), dict(window=64, use_graph=1, scheduler=0),
                     dict(window=192, light_cap=3, heavy_frac=0.3, good_first=1)):
            res, loads = sim.run(want_load=True, no_drop=int(no_drop), **opts)
            assert (sim.stats()["heavy_form"] == 4) == (name != "deep4096")
            for a, b in zip(split(res[0]), exp[:3]):
                assert np.array_equal(a, b), opts
            assert np.array_equal(loads[0], gload), opts
            if no_drop:
                assert np.array_equal(sim.mismatch_counts(0), exp[3]), opts


def test_packed_form_many_designs_and_more_faults_than_slots():
    """Designs of several sizes and cycle counts in one run (one without faults), with enough
    faults that lanes are refilled, against the general path."""
    parts = []
    for i, (n, T, F) in enumerate([(900, 150, 90000), (1500, 65, 4000), (1000, 200, 0), (1200, 1, 500)]):
        d = synth.gen_datapath_fsm(60 + i, n, max(48, n // 10), 16, 16, [8], 0.8, 8, 64)
        u = synth.fault_universe(d)
        f = u.take(np.resize(np.arange(len(u)), F)) if F else u.take(np.zeros(0, np.int64))
        parts.append((d, synth.stimulus(d, T, i, 0.1), f))
    with Simulator(0) as sim:
        for p in parts:
            sim.add(*p)
        ref, rl = sim.run(want_load=True, heavy_form=1, window=64)
        for opts in (dict(), dict(window=128, use_graph=1)):
            got, gl = sim.run(want_load=True, **opts)
            for a, b, x, y in zip(got, ref, gl, rl):
                assert np.array_equal(a, b) and np.array_equal(x, y), opts


def test_budget_in_the_packed_form():
    d, stim, f = _case("fan130")
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        out = []
        for form in (1, 0):
            from paper_2508_16376_gb300.rtlfs import make_opts, rtlfs_run
            r, l, rc = rtlfs_run(sim.ctx, sim.n_faults, make_opts(fault_budget=300, heavy_form=form), True, check=False)
            out.append((r[0], l[0], rc))
    assert out[0][2] == out[1][2]
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert int((out[0][0]["detected"] == 255).sum()) > 0
