"""The autotuner where the library runs the packed form, against a fake campaign timer: no repeated trials
of knobs that form does not read, and the light and heavy kernels tuned beside it."""
import pytest

from paper_2508_16376_gb300 import autotune
from test_autotune_cpu import FakeSim


class PackedSim(FakeSim):
    def stats(self):
        return dict(super().stats(), heavy_form=self.last.get("heavy_form", 0) or 4)


def _cost(packed_ms, general_ms):
    def cost(o):
        if o.get("heavy_form"):   # the light and heavy kernels read every knob
            return general_ms + 10.0 * (o["window"] != 128) + 10.0 * (o["light_block"] != 64)
        return packed_ms + 5.0 * (o["good_first"] != 1)
    return cost


@pytest.mark.parametrize("packed_ms,general_ms", [(100.0, 300.0), (300.0, 100.0)])
def test_the_faster_form_wins_and_blind_knobs_are_not_swept(tmp_path, packed_ms, general_ms):
    sim = PackedSim(_cost(packed_ms, general_ms))
    best = autotune.tune(sim, cache_path=str(tmp_path / "c.json"))
    packed_runs = [r for r in sim.runs if "heavy_form" not in r]
    for k in autotune.BLIND:
        assert {r[k] for r in packed_runs} == {autotune.BASE[k]}
    knobs = dict(autotune.KNOBS)
    assert len(packed_runs) == 1 + sum(len(v) - 1 for k, v in knobs.items() if k not in autotune.BLIND)
    if packed_ms < general_ms:
        assert "heavy_form" not in best and best["good_first"] == 1
    else:
        assert best["heavy_form"] == 1 and best["window"] == 128 and best["light_block"] == 64
