"""The autotuner on plans whose Legendre steps run on the tensor cores: it times only the knobs their kernels
read, and nothing twice where there is nothing to choose (fake plans and timers, no GPU)."""
import numpy as np

from paper_1106_0159_gb300 import autotune, sht
from paper_1106_0159_gb300.autotune import ALM2MAP, MAP2ALM


class FakePlan:
    nrings, npix, lmax, mmax = 1023, 786432, 512, 512
    fp64_tensor = True

    def __init__(self, mode=sht.MODE_FP64):
        self.mode = mode
        self.knobs = {sht.TUNE_SYNTH_MAPS: 4, sht.TUNE_ANAL_MAPS: 2, sht.TUNE_ANAL_SLOTS: 4, sht.TUNE_DF_MAPS: 8,
                      sht.TUNE_TC_MAPS: 16, sht.TUNE_PREC_ANAL: 1}

    def set_tuning(self, k, v):
        assert v in sht.TUNE_VALUES[k]
        self.knobs[k] = v

    def tuning(self, k):
        return self.knobs[k]


def _tune(plan, direction, nmaps):
    calls = []

    def timer(p, d, src, dst):
        calls.append(dict(p.knobs))
        return 5.0 + 0.1 * len(calls) - (p.knobs[sht.TUNE_TC_MAPS] == 8)
    return autotune.Autotuner(timer=timer).tune(plan, direction, np.zeros((nmaps, 4)), None), calls


def test_only_the_knobs_of_the_tensor_core_kernels_are_timed():
    for mode in (sht.MODE_FP64, sht.MODE_SPLIT_BF16):
        p = FakePlan(mode)
        rec, calls = _tune(p, ALM2MAP, 16)
        assert rec["knobs"] == {str(sht.TUNE_TC_MAPS): 8} and p.knobs[sht.TUNE_TC_MAPS] == 8
        assert [c[sht.TUNE_TC_MAPS] for c in calls] == [8, 16, 16]
        assert {c[sht.TUNE_SYNTH_MAPS] for c in calls} == {4}
        rec, calls = _tune(FakePlan(mode), ALM2MAP, 3)      # up to 8 maps both values act alike
        assert rec["knobs"] == {str(sht.TUNE_TC_MAPS): 16} and len(calls) == 1
    rec, calls = _tune(FakePlan(), MAP2ALM, 16)             # the FP64 analysis there reads no knob
    assert rec["knobs"] == {} and len(calls) == 1 and rec["ms"] == rec["default_ms"] and rec["tried"] == []
    assert autotune.knobs_for(MAP2ALM, sht.MODE_SPLIT_BF16, True) == [sht.TUNE_PREC_ANAL, sht.TUNE_DF_MAPS]
    assert autotune.knobs_for(ALM2MAP, sht.MODE_FP64, False) == [sht.TUNE_SYNTH_MAPS]


class FakeBatch:
    def __init__(self, tiles):
        self.n = tiles
        self.k = {sht.BATCH_SYNTH_MAPS: 4, sht.BATCH_LEG_CTAS: 8, sht.BATCH_RING_CTAS: 4, sht.BATCH_ANAL_MAPS: 2,
                  sht.BATCH_ANAL_SLOTS: 4}
        self.touched = set()

    def tiles(self, stage):
        return self.n if stage == 0 else 100

    def tuning(self, knob):
        return self.k[knob]

    def set_tuning(self, knob, value):
        self.k[knob] = value
        self.touched.add(knob)


def test_a_batch_without_queued_legendre_work_tunes_its_ring_grid_only():
    for d in (ALM2MAP, MAP2ALM):
        b = FakeBatch(0)
        rec = autotune.tune_batch(b, d, timer=lambda bb: 10.0 + abs(bb.k[sht.BATCH_RING_CTAS] - 2))
        assert b.touched == {sht.BATCH_RING_CTAS} and b.k[sht.BATCH_RING_CTAS] == 2
        assert rec["knobs"] == {str(sht.BATCH_RING_CTAS): 2}
    b = FakeBatch(7)
    autotune.tune_batch(b, ALM2MAP, timer=lambda bb: 1.0)
    assert b.touched == set(autotune.batch_knobs(ALM2MAP))
