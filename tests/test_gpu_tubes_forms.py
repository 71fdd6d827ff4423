"""GPU test of the tube batch's choice between its two forms, around the lengths, steps
and sizes of the rule: the form that runs, and the same bits from both at lengths around the
pair chunks of the resident form's blocks."""
import numpy as np
import pytest

from test_gpu_tubes import _batch, _fields
from test_gpu_tubes_resident import _run, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,steps,resident", [
    ([1024, 60], 2, True), ([1024, 60], 1, False), ([1025, 60], 2, False), ([1025, 60], 3, True),
    ([2048] * 3, 3, True), ([2049] * 3, 64, False), ([3600] * 8, 64, False),
    ([2049] * 75, 4, True), ([2049] * 75, 3, False), ([3600] * 153, 8, False), ([3600] * 180, 8, True),
    ([3601], 64, False)])
def test_form(lengths, steps, resident):
    from paper_0908_3749_gb300 import lbm
    B = _batch(lengths, seed=1)
    b = lbm.lbm_batch_create(B["nx"], B["dx"], B["dt"], B["s"], B["left"], B["right"])
    try:
        assert lbm.lbm_batch_plan(b, steps)[0] == resident
        lbm.lbm_batch_set_tiling(b, 512, 128)
        assert lbm.lbm_batch_plan(b, steps) == (False, 1)
    finally:
        lbm.lbm_batch_destroy(b)


SHORT = [2, 3, 4, 127, 128, 129, 255, 256, 257, 258, 385, 511, 512, 513, 767, 1023, 1024, 1025, 1537, 2047, 2048]
LONG = [2049, 2500, 3071, 3072, 3073, 3599, 3600]


@pytest.mark.parametrize("lengths,chunks", [
    (SHORT, [20]), (SHORT * 10, [3, 17]), (SHORT[:17] * 9, [2, 1, 17]),
    (SHORT + LONG * 8, [4, 16]), (SHORT * 10 + LONG * 30, [8, 12])])
def test_resident_equals_streamed(lengths, chunks):
    from paper_0908_3749_gb300 import lbm
    B = _batch(lengths, seed=11)
    b = lbm.lbm_batch_create(B["nx"], B["dx"], B["dt"], B["s"], B["left"], B["right"])
    assert lbm.lbm_batch_plan(b, max(chunks))[0]
    lbm.lbm_batch_destroy(b)
    _same(_run(B, chunks, False), _run(B, [sum(chunks)], True))
