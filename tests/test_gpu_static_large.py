"""The allocation-free call on a design whose bitmaps do not fit in a CTA's shared memory: a thread per
fault, in waves of as many as the scratch array holds, against the oracle, with out-of-range faults among
them."""
import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import rtlfs, synth
from paper_2508_16376_gb300.rtlfs import Simulator, split

pytestmark = pytest.mark.gpu


def large(levels=24, width=40000, regs=64):
    """Rows of two-operand nodes over the row before; the registers also feed a late row, and latch and
    are observed in the last, so faults of the late rows have small cones that live on."""
    rng = np.random.default_rng(7)
    I, R, N = 4, regs, levels * width
    row = np.repeat(np.arange(levels), width)
    first = I + R + (row - 1) * width
    a = np.where(row == 0, rng.integers(0, I + R, N), first + rng.integers(0, width, N)).astype(np.uint32)
    b = np.where((row == 0) | ((row == levels - 5) & (rng.random(N) < 0.01)), rng.integers(0, I + R, N),
                 first + rng.integers(0, width, N)).astype(np.uint32)
    last = I + R + N - width
    return synth.Design("large", np.full(I, 16, np.uint8), np.full(R, 16, np.uint8),
                        rng.integers(last, last + width, R).astype(np.uint32),
                        rng.choice([synth.XOR, synth.ADD, synth.SUB, synth.OR], N).astype(np.uint8), np.full(N, 16, np.uint8),
                        a, b, np.zeros(N, np.uint32), np.zeros(N, np.uint64), (last + np.arange(0, 400, 50)).astype(np.uint32))


def test_thread_per_fault_form():
    import torch
    from paper_2508_16376_gb300 import build
    build.build()
    oracle.build()
    d = large()
    T = 4
    words = lambda n: (n + 31) // 32
    assert 4 * (words(d.n_node) + words(d.n_net)) > 227 * 1024            # no warp's bitmaps fit
    wave = (64 * 2 ** 20 - 4 * d.n_net) // (12 * d.n_net + 8 * d.n_node)
    assert 0 < wave < 5
    stim = synth.stimulus(d, T, 5, 0.2)
    rng = np.random.default_rng(1)
    first = d.n_in + d.n_reg
    # late nodes (one that an output observes among them) and a register
    net = np.concatenate([d.n_net - 1 - rng.integers(0, 4 * 40000, 10), [d.outputs[3], d.n_in + 5, first + 20 * 40000 + 77]])
    f = synth.Faults(net.astype(np.uint32), rng.integers(0, 16, len(net)).astype(np.uint8), rng.integers(0, 2, len(net)).astype(np.uint8))
    exp = oracle.fault_sim(d, stim, f, threads=8)
    fa = rtlfs.fault_array(f).copy()
    bad = np.array([2, 7])
    fa["bit"][bad] = 16
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        sim.good_outputs(0)
        dev = torch.from_numpy(fa.view(np.uint8).copy()).cuda()
        out = torch.full((len(fa) * rtlfs.RESULT_DTYPE.itemsize,), 0xA5, dtype=torch.uint8, device="cuda")
        rc = rtlfs.rtlfs_fault_sim_static(sim.ctx, 0, dev.data_ptr(), len(fa), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc != rtlfs.RTLFS_OK
    got = out.cpu().numpy().view(rtlfs.RESULT_DTYPE)
    assert (got["detected"][bad] == 254).all()
    ok = np.setdiff1d(np.arange(len(fa)), bad)
    assert exp[0][ok].any() and not exp[0][ok].all()
    for a, b in zip(split(got), exp):
        assert np.array_equal(a[ok], b[ok])
