"""The allocation-free call on designs with a few nodes per level, whose chains one lane walks, against
the oracle: chains through every op, whose value feeds one operand, several or a select, chains that
meet, chains longer than one look at the bitmap, latches and ports along the way."""
import functools

import numpy as np
import pytest

import oracle
from paper_2508_16376_gb300 import rtlfs, synth
from paper_2508_16376_gb300.rtlfs import Simulator, split
from paper_2508_16376_gb300.synth import ADD, AND, CONCAT, EQ, LT, MUX2, NOT, OR, SHL, SHR, SLICE, SUB, XOR, _Builder

pytestmark = pytest.mark.gpu


def thin(chains, length, meet, seed):
    """`chains` chains of `length` nodes, one in `meet` of whose nodes reads another chain too."""
    rng = np.random.default_rng(seed)
    b = _Builder([16, 16, 1, 4], [16] * (chains + 3))
    regs = [b.reg_net(i) for i in range(chains + 3)]
    tail = regs[:chains]
    seen = []
    for k in range(length):
        for c in range(chains):
            x = tail[c]
            y = tail[int(rng.integers(chains))] if rng.random() * meet < 1 else int(rng.choice([0, 1, 3] + regs))
            r = int(rng.integers(16))
            if r < 5: n = b.add((AND, OR, XOR, ADD, SUB)[r], 16, x, y)
            elif r < 8: n = b.add((ADD, XOR, SUB)[r - 5], 16, y, x)
            elif r == 8: n = b.add(ADD, 16, x, x)              # both operands
            elif r == 9: n = b.add(MUX2, 16, x, y, 1)          # the select
            elif r == 10: n = b.add(MUX2, 16, 2, x, y)
            elif r == 11: n = b.add(MUX2, 16, x, x, y)         # select and operand
            elif r == 12: n = b.add(NOT, 16, x)
            elif r == 13: n = b.add((SHL, SHR)[k & 1], 16, x, imm=int(rng.integers(0, 5)))
            elif r == 14: n = b.add(CONCAT, 16, b.add(SLICE, 8, x, imm=4), b.add(SLICE, 8, x, imm=0))
            else: n = b.add(XOR, 16, x, b.add((EQ, LT)[k & 1], 1, x, y))
            tail[c] = n
            seen.append(n)
    for i in range(chains):
        b.reg_d[i] = tail[i]
    for i in range(3):
        b.reg_d[chains + i] = seen[int(rng.integers(len(seen)))]
    return b.finish("thin", [tail[0], seen[len(seen) // 2], seen[len(seen) // 3]])


CASES = {"one": (1, 40, 99), "long": (1, 2600, 99), "two": (2, 700, 6), "six": (6, 300, 9), "apart": (6, 60, 1e9)}


@functools.lru_cache(maxsize=None)
def _case(name):
    d = thin(*CASES[name], seed=len(name))
    T = 40
    stim = synth.stimulus(d, T, 5, 0.3)
    u = synth.fault_universe(d, include_inputs=True)
    f = u.take(np.sort(np.random.default_rng(1).choice(len(u), min(len(u), 3000), replace=False)))
    return d, stim, f, oracle.fault_sim(d, stim, f, threads=16)


@pytest.mark.parametrize("name", sorted(CASES))
def test_thin_designs_equal_oracle(name):
    import torch
    oracle.build()
    d, stim, f, exp = _case(name)
    with Simulator(0) as sim:
        sim.add(d, stim, f)
        assert d.n_node <= 8 * rtlfs.rtlfs_design_info(sim.ctx, 0)[1]
        sim.good_outputs(0)
        dev = torch.from_numpy(rtlfs.fault_array(f).view(np.uint8).copy()).cuda()
        out = torch.full((len(f) * rtlfs.RESULT_DTYPE.itemsize,), 0xA5, dtype=torch.uint8, device="cuda")
        rtlfs.rtlfs_fault_sim_static(sim.ctx, 0, dev.data_ptr(), len(f), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    for a, b in zip(split(out.cpu().numpy().view(rtlfs.RESULT_DTYPE)), exp):
        assert np.array_equal(a, b)
