"""What a user of this framework has it do, as measurable cases.

A case is one pass through the public entry points: a fault-simulation campaign (new
stimulus and fault lists handed over from host memory, every fault simulated, results back
in host memory), a good-machine simulation, a scoring pass of the load predictor, one
gradient of its training, or the allocation-free call on device buffers. Designs are the
seeded synthetic shapes of `synth` (the repository's own configurations: tiny, medium, the
batch's 1k-50k nodes, large); a design is loaded once, as a user's program keeps it, while
the stimulus and the fault list are new with every seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2508_16376_gb300 import rtlfs, synth

# Options of the tuned campaigns (the ones the benchmark runs its workloads with).
MEDIUM = {"window": 128, "light_cap": 1, "light_block": 256, "heavy_frac": 0.02}
BATCH = {"window": 128, "light_cap": 1, "light_block": 64, "heavy_frac": 0.0, "use_graph": 1}
LARGE = {"window": 128, "light_cap": 1, "light_block": 256, "heavy_frac": 0.0}
LEARNED = {"window": 512, "light_cap": 1, "heavy_frac": 0.0, "scheduler": rtlfs.SCHED_MLP, "use_graph": 1,
           "order_classes": 8}
PLAIN_OPTS = {"window": 256, "light_cap": 1}


def _campaign(name, shape, nodes, cycles, faults, opts, **kw):
    c = {"kind": "campaign", "shape": shape, "nodes": nodes, "design_seed": 2, "designs": 1, "cycles": cycles,
         "faults": faults, "hold": 0.1, "model": "stuck", "loads": False}
    c.update({"opt_" + k: v for k, v in opts.items()})
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: the tiny design's whole fault list with default options, as in a
        # unit-level regression; launches, copies and host work count.
        _campaign("tiny_default", "tiny", 200, 100, 5926, {}, design_seed=1, hold=0.0),
        # A block-level design screened quickly with default options (odd sizes).
        _campaign("block_default", "datapath", 2777, 777, 3001, {}, hold=0.0),
        # Load recording for the predictor's training data: the one-pass form, loads wanted.
        _campaign("record_loads", "medium", 20000, 1511, 5003, {"scheduler": rtlfs.SCHED_PLAIN}, design_seed=11,
                  loads=True),
        # The medium campaign at full size: 20k nodes, 10k cycles, 100k sampled stuck-at faults.
        _campaign("medium_campaign", "medium", 20000, 10000, 100000, MEDIUM),
        # Transient faults (SEU/SET) mixed with output-port and stuck-at faults, same design.
        _campaign("transient_mixed", "medium", 20000, 2501, 30011, PLAIN_OPTS, model="mixed"),
        # The evaluation protocol without fault dropping, with n-detection counts.
        _campaign("no_drop", "datapath", 9973, 1003, 4001, dict(PLAIN_OPTS, no_drop=1)),
        # Many designs in one graph-replayed campaign (1k-50k nodes, ragged cycle counts).
        _campaign("batch_graph", "batch", 50000, 1500, 5000, BATCH, design_seed=1000, designs=12, hold=0.0),
        # The large design (200k nodes, 256 ports, 8 FSMs) over a shorter stimulus.
        _campaign("large_campaign", "large", 200000, 512, 20000, LARGE, design_seed=4, hold=0.0),
        # Good machine only: new stimulus in, golden outputs out, a design of 48k nodes.
        {"name": "good_outputs", "kind": "good", "shape": "datapath", "nodes": 48000, "design_seed": 5, "cycles": 3000,
         "hold": 0.0},
        # Predictor in use: features of a fault list and its scores (sharding, queue order).
        {"name": "predict_scores", "kind": "score", "shape": "medium", "nodes": 20000, "design_seed": 2, "cycles": 300,
         "faults": 400000, "hold": 0.1},
        # One gradient of the predictor's training over a large batch.
        {"name": "train_gradient", "kind": "grad", "samples": 65537},
        # The allocation-free call on caller-owned device buffers.
        {"name": "static_call", "kind": "static", "shape": "datapath", "nodes": 1200, "design_seed": 7, "cycles": 300,
         "faults": 1500, "hold": 0.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["campaign"] * 7 + ["good", "score", "grad", "static"])
    seed = rng.randrange(1, 1 << 20)
    if kind == "grad":
        return {"kind": kind, "samples": _log(rng, 300, 200000)}
    if kind == "static":
        return {"kind": kind, "shape": "datapath", "nodes": _log(rng, 1000, 3000), "design_seed": seed,
                "cycles": _log(rng, 50, 300), "faults": _log(rng, 100, 1500), "hold": 0.0}
    nodes = _log(rng, 1000, 60000)
    if kind == "good":
        return {"kind": kind, "shape": "datapath", "nodes": nodes, "design_seed": seed,
                "cycles": min(_log(rng, 100, 10000), 144_000_000 // nodes), "hold": rng.choice([0.0, 0.1])}
    if kind == "score":
        return {"kind": kind, "shape": "datapath", "nodes": nodes, "design_seed": seed, "cycles": _log(rng, 64, 600),
                "faults": min(_log(rng, 2000, 400000), 20 * nodes), "hold": 0.1}
    if rng.random() < 0.12:
        return _campaign("", "tiny", 200, _log(rng, 20, 400), 5926, {}, design_seed=seed, hold=0.0)
    cycles = _log(rng, 100, 8000)
    faults = min(_log(rng, 500, 60000), 100_000_000 // cycles)
    opts = {"window": rng.choice([0, 64, 128, 256, 512]), "light_cap": rng.choice([0, 1, 1]),
            "scheduler": rng.choice([rtlfs.SCHED_PLAIN, rtlfs.SCHED_HEURISTIC, rtlfs.SCHED_MLP]),
            "use_graph": rng.choice([0, 1])}
    kw = {"design_seed": seed, "hold": rng.choice([0.0, 0.1]), "model": rng.choice(["stuck", "stuck", "mixed"])}
    if rng.random() < 0.25:   # without dropping every fault runs every cycle
        opts["no_drop"] = 1
        faults = min(faults, 20_000_000 // cycles)
    if rng.random() < 0.25:
        kw["designs"] = rng.randint(2, 12)
        return _campaign("", "batch", nodes, min(cycles, 1500), min(faults, 5000), opts, **kw)
    return _campaign("", "datapath", nodes, cycles, faults, opts, **kw)


# ---- inputs -------------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _design(shape, nodes, seed):
    if shape == "tiny":
        return synth.tiny_design(seed)
    if shape == "medium":
        return synth.medium_design(seed)
    if shape == "large":
        return synth.large_design(seed)
    # the batch's rule for registers and stages
    return synth.gen_datapath_fsm(seed, nodes, max(48, nodes // 10), 64, 64, [32], 0.8,
                                  int(max(8, min(40, nodes // 250))), 64, "datapath")


def _sizes(case):
    """Per design of the case: (shape, nodes, design seed, cycles, faults)."""
    if case.get("shape") != "batch":
        return [(case["shape"], case["nodes"], case["design_seed"], case["cycles"], case.get("faults", 0))]
    rng = np.random.default_rng(case["design_seed"])   # ragged: nodes log-uniform, cycles and faults uniform
    out = []
    for i in range(case["designs"]):
        n = int(round(math.exp(rng.uniform(math.log(1000), math.log(case["nodes"])))))
        out.append(("datapath", n, case["design_seed"] + i, int(rng.integers(max(1, case["cycles"] // 5), case["cycles"] + 1)),
                    int(rng.integers(max(1, case["faults"] // 5), case["faults"] + 1))))
    return out


def _faults(design, model, cycles, n, seed):
    if model == "mixed":   # half stuck-at, a tenth output-port stuck-at, the rest transient
        ports = synth.port_faults(design)
        ports = ports.take(np.sort(np.random.default_rng(seed).choice(len(ports), min(len(ports), n // 10), replace=False)))
        return synth.Faults.concat([synth.sample_faults(design, n // 2, seed), ports,
                                    synth.transient_faults(design, n - n // 2 - len(ports), cycles, seed)])
    return synth.sample_faults(design, n, seed)


class _State:
    """The context a user's program keeps (closed with the object) and the host inputs."""

    def __init__(self):
        self.sim = rtlfs.Simulator(0)

    def __del__(self):
        sim = getattr(self, "sim", None)
        if sim is not None:
            sim.close()


def _samples(n, seed):
    """Feature rows and log-loads with the spread the recorded training data has."""
    rng = np.random.default_rng(seed)
    X = np.stack([rng.uniform(0.0, 1.5, n), rng.uniform(0.0, 1.0, n), rng.integers(0, 17, n) / 16.0,
                  rng.integers(1, 65, n) / 64.0, rng.uniform(0.0, 0.6, n)], 1).astype(np.float32)
    t = (4.0 + 5.0 * X[:, 0] * X[:, 4] + rng.normal(0.0, 1.5, n)).clip(0.0, 16.0).astype(np.float32)
    return X, t


def _weights(seed):
    """BF16 parameters of the predictor's shape, as after some training."""
    rng = np.random.default_rng(seed + 77)
    w = np.zeros(rtlfs.MLP_PARAMS, np.float32)
    w[:320] = rng.normal(0, math.sqrt(2 / 5), 320)
    w[320:384] = rng.normal(0, 0.05, 64)
    w[384:4480] = rng.normal(0, math.sqrt(2 / 64), 4096)
    w[4480:4544] = rng.normal(0, 0.05, 64)
    w[4544:4608] = rng.normal(0, math.sqrt(1 / 64), 64)
    w[4608] = 4.0
    return torch.from_numpy(w).to(torch.bfloat16)


def prepare(case, seed):
    s = _State()
    s.kind = case["kind"]
    ctx = s.sim.ctx
    if s.kind in ("grad", "score") or case.get("opt_scheduler") == rtlfs.SCHED_MLP:
        rtlfs.rtlfs_mlp_set_weights(ctx, _weights(seed).view(torch.int16).numpy().view(np.uint16))
    if s.kind == "grad":
        s.X, s.t = _samples(case["samples"], seed)
        return s
    s.stim, s.faults, s.n_faults, s.cycles, s.n_out = [], [], [], [], []
    for i, (shape, nodes, dseed, cycles, n) in enumerate(_sizes(case)):
        d = _design(shape, nodes, dseed)
        rtlfs.rtlfs_load_design(ctx, *rtlfs.design_arrays(d))
        s.stim.append(synth.stimulus(d, cycles, 1_000_000 + 97 * seed + i, case["hold"]))
        f = _faults(d, case.get("model", "stuck"), cycles, n, 2_000_000 + 89 * seed + i) if n else None
        s.faults.append(None if f is None else rtlfs.fault_array(f) if f.cycle is None else rtlfs.fault_array_ex(f))
        s.n_faults.append(0 if f is None else len(f))
        s.cycles.append(cycles)
        s.n_out.append(d.n_out)
    if s.kind == "campaign":
        s.loads = case["loads"]
        opts = {k[4:]: v for k, v in case.items() if k.startswith("opt_")}
        s.no_drop = bool(opts.get("no_drop"))
        s.opts = rtlfs.make_opts(**opts) if opts else None
    if s.kind == "score":   # the good trace is there from an earlier call
        rtlfs.rtlfs_set_stimulus(ctx, 0, s.stim[0])
        rtlfs.rtlfs_good_outputs(ctx, 0, s.cycles[0], s.n_out[0])
    if s.kind == "static":
        rtlfs.rtlfs_set_stimulus(ctx, 0, s.stim[0])
        rtlfs.rtlfs_good_outputs(ctx, 0, s.cycles[0], s.n_out[0])
        s.dev_faults = torch.from_numpy(s.faults[0].view(np.uint8).copy()).cuda()
        s.dev_results = torch.zeros(s.n_faults[0], 3, dtype=torch.int32, device="cuda")
    return s


def run(s):
    ctx = s.sim.ctx
    if s.kind == "grad":
        return rtlfs.rtlfs_mlp_grad(ctx, s.X, s.t)
    if s.kind == "good":
        rtlfs.rtlfs_set_stimulus(ctx, 0, s.stim[0])
        return rtlfs.rtlfs_good_outputs(ctx, 0, s.cycles[0], s.n_out[0]).view(np.int64)
    if s.kind == "score":
        rtlfs.rtlfs_set_faults(ctx, 0, s.faults[0])
        X = rtlfs.rtlfs_features(ctx, 0, s.n_faults[0])
        return X, rtlfs.rtlfs_mlp_forward(ctx, X)
    if s.kind == "static":
        rc = rtlfs.rtlfs_fault_sim_static(ctx, 0, s.dev_faults.data_ptr(), s.n_faults[0], s.dev_results.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream)
        return rc, s.dev_results
    for i, (stim, faults) in enumerate(zip(s.stim, s.faults)):
        rtlfs.rtlfs_set_stimulus(ctx, i, stim)
        (rtlfs.rtlfs_set_faults if faults.dtype == rtlfs.FAULT_DTYPE else rtlfs.rtlfs_set_faults_ex)(ctx, i, faults)
    res, loads, _ = rtlfs.rtlfs_run(ctx, s.n_faults, s.opts, s.loads)
    out = [[r["detected"], r["cycle"], r["port"]] for r in res]
    if s.loads:
        out.append([x.view(np.int64) for x in loads])
    if s.no_drop:
        out.append([rtlfs.rtlfs_mismatch_counts(ctx, i, n).view(np.int32) for i, n in enumerate(s.n_faults)])
    return out


def work(case):
    """Inputs read once and outputs written once; operations: every good-machine node once
    a cycle (what the faulty machines need beyond that depends on the values)."""
    if case["kind"] == "grad":
        n = case["samples"]
        return {"bytes": 24 * n + 6 * rtlfs.MLP_PARAMS + 4, "flops": 6 * n * (5 * 64 + 64 * 64 + 64)}
    nbytes = flops = 0
    for shape, nodes, _, cycles, faults in _sizes(case):
        n_in = 8 if shape == "tiny" else 256 if shape == "large" else 64
        graph = 40 * nodes   # the operator graph: descriptors and fan-out lists
        if case["kind"] == "score":
            nbytes += graph + faults * (8 + 20 + 4) + 8 * min(cycles, 256) * min(nodes, faults)
            flops += 2 * faults * (5 * 64 + 64 * 64 + 64)
        elif case["kind"] == "static":
            nbytes += graph + 8 * nodes * cycles + faults * (8 + 12)
        else:
            n_out = 8 * n_in * cycles if case["kind"] == "good" else faults * (12 + 8 * bool(case["loads"]))
            nbytes += graph + 8 * n_in * cycles + 8 * faults + n_out
            flops += nodes * cycles
    return {"bytes": nbytes, "flops": flops}


# ---- exact values of the computed floats -----------------------------------------------------

def _mlp64(X, seed):
    w = _weights(seed).to(torch.float64)
    W1, b1, W2, b2 = w[:320].view(5, 64), w[320:384], w[384:4480].view(64, 64), w[4480:4544]
    w3, b3 = w[4544:4608], w[4608]
    p = [x.clone().requires_grad_(True) for x in (W1, b1, W2, b2, w3, b3)]
    h = torch.relu(torch.relu(torch.from_numpy(X).double() @ p[0] + p[1]) @ p[2] + p[3])
    return h @ p[4] + p[5], p


def exact(case, seed):
    if case["kind"] == "grad":
        X, t = _samples(case["samples"], seed)
        y, p = _mlp64(X, seed)
        loss = ((y - torch.from_numpy(t).double()) ** 2).mean()
        loss.backward()
        return float(loss.detach()), torch.cat([x.grad.reshape(-1) for x in p])
    return None   # whole numbers, or (scores) values of the recorded trace
