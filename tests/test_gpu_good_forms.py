"""The good trace in every form (one CTA, clusters of 2 to 16, chosen and forced) against the
oracle's trace, net by net, where its schedules and loops have edges: more inputs than threads,
more registers than a thread keeps, one node latched by every register (homes in other CTAs),
64-bit words through every op, and windows that resume."""
import dataclasses
import functools

import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import synth
from paper_2508_16376_gb300.rtlfs import Simulator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_16376_gb300 import build
    build.build()
    oracle.build()


@functools.lru_cache(maxsize=None)
def _case(which):
    if which == "wide":
        d = synth.gen_random_dag(5, 900, 3300, 700, 16, 40, 64, 1, 64, "wide")
    elif which == "one_d":
        d = synth.gen_random_dag(6, 700, 640, 8, 8, 8, 64, 8, 64, "one_d")
        d = dataclasses.replace(d, reg_d=np.full_like(d.reg_d, d.n_in + d.n_reg + d.n_node - 1))
    else:
        d = synth.gen_random_dag(7, 3000, 40, 8, 8, 64, 64, 8, 64, "ops")
    stim = synth.stimulus(d, 70, 9, 0.1)
    _, trace = oracle.good_run(d, stim, with_trace=True)
    return d, stim, synth.sample_faults(d, 64, 1), trace


@pytest.mark.parametrize("opts", [dict(), dict(good_cluster=2), dict(good_cluster=4, window=64), dict(good_cluster=16),
                                  dict(window=33)])
@pytest.mark.parametrize("which", ["wide", "one_d", "ops"])
def test_good_trace_forms(which, opts):
    d, stim, f, trace = _case(which)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        sim.run(**opts)
        assert np.array_equal(sim.good_trace(0), trace)
