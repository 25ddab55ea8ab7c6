"""A design of registers alone that is too large for one CTA's shared memory: its good trace runs on
clusters whose schedule has no steps, and its campaigns on designs without levels."""
import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import synth
from paper_2508_16376_gb300.rtlfs import Simulator, split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(), dict(good_cluster=4), dict(window=64)])
def test_registers_only_on_clusters(opts):
    from paper_2508_16376_gb300 import build
    build.build()
    oracle.build()
    d = synth.delay_chain(29500, 8)
    assert d.n_node == 0
    stim = synth.stimulus(d, 70, 3)
    f = synth.sample_faults(d, 40, 2)
    _, trace = oracle.good_run(d, stim, with_trace=True)
    exp = oracle.fault_sim(d, stim, f, threads=8)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        res, _ = sim.run(**opts)
        assert np.array_equal(sim.good_trace(0), trace)
    for a, b in zip(split(res[0]), exp):
        assert np.array_equal(a, b)
