"""The allocation-free call against the oracle where its warp-per-fault kernel has edges: levels
wider than one look at the bitmap (1024 nodes), nets with more than eight consumers and several
latches, registers fed by registers, a fault on every kind of net, more faults than warps, cycle
counts around 32, and out-of-range faults among good ones."""
import functools

import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import rtlfs, synth
from paper_2508_16376_gb300.rtlfs import Simulator, split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_16376_gb300 import build
    build.build()
    oracle.build()


@functools.lru_cache(maxsize=None)
def _case(which):
    if which == "wide":      # 2,500 nodes on its first level
        d = synth.gen_datapath_fsm(2, 12000, 900, 16, 16, [8], 0.4, 6, 64, "wide")
        T, F = 65, 6000
    elif which == "chain":
        d, T, F = synth.delay_chain(9, 13), 31, None
    elif which == "regs":    # registers latch common nets: several latches per net
        d, T, F = synth.gen_random_dag(8, 150, 400, 6, 6, 16, 64, 1, 64, "regs"), 33, None
    else:
        d, T, F = synth.tiny_design(3), 97, None
    stim = synth.stimulus(d, T, 5, 0.3)
    f = synth.fault_universe(d, include_inputs=True) if F is None else synth.sample_faults(d, F, 3)
    return d, stim, f, oracle.fault_sim(d, stim, f, threads=16)


@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("which", ["wide", "chain", "regs", "tiny"])
def test_static_call_equals_oracle(which, bad):
    import torch
    d, stim, f, exp = _case(which)
    fa = rtlfs.fault_array(f).copy()
    n = len(fa)
    at = np.arange(0, n, 7) if bad else np.zeros(0, np.int64)
    fa["bit"][at] = 64
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        sim.good_outputs(0)
        dev = torch.from_numpy(fa.view(np.uint8).copy()).cuda()
        out = torch.full((n * rtlfs.RESULT_DTYPE.itemsize,), 0xA5, dtype=torch.uint8, device="cuda")
        call = lambda: rtlfs.rtlfs_fault_sim_static(sim.ctx, 0, dev.data_ptr(), n, out.data_ptr(),
                                                    torch.cuda.current_stream().cuda_stream)
        rc = call()
        assert (rc != rtlfs.RTLFS_OK) == bad
    got = out.cpu().numpy().view(rtlfs.RESULT_DTYPE)
    assert (got["detected"][at] == 254).all()
    ok = np.setdiff1d(np.arange(n), at)
    for a, b in zip(split(got), exp):
        assert np.array_equal(a[ok], b[ok])
