"""The bench line's kernel entry for the packed form: its tiers run side by side, so their summed
times are no time of the step; the faulty machines' span (under graph replay the step's time) is."""
import numpy as np

from paper_2508_16376_gb300 import roofline, synth


def _stats(form, faulty):
    return dict(good_ms=3.0, light_ms=5.0, heavy_ms=40.0, faulty_ms=faulty, heavy_form=form, node_evals=10, fault_cycles=20)


def test_packed_kernels_are_taken_together():
    assert roofline.dominant(roofline.kernel_times([_stats(1, 12.0)], 15.0)) == ("heavy", 40.0)
    assert roofline.dominant(roofline.kernel_times([_stats(4, 12.0), _stats(4, 14.0)], 15.0)) == ("packed", 13.0)
    mean = roofline.kernel_times([_stats(4, 0.0)], 15.0)
    assert roofline.dominant(mean) == ("packed", 15.0)
    d = synth.counter4()
    parts = [(d, np.zeros((20, 1), np.uint64), synth.Faults(np.array([1], np.uint32), np.zeros(1, np.uint8), np.zeros(1, np.uint8)))]
    r = roofline.step_roofline(parts, None, _stats(4, 0.0), mean, {"window": 8}, {"hbm_gbs": 1000.0}, 30, 15.0,
                               roofline.int_peak({}, 2000.0, 100))
    assert r["kernel_ms_per_step"] <= 15.0 and r["launches"] == 30 and abs(r["avg_launch_ms"] - 0.5) < 1e-12
    assert abs(r["achieved"] - r["step_achieved"]) < 1e-12
