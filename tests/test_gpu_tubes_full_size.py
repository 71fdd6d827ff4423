"""GPU test of the 4096-tube batch at its full size in both forms: the one that the
library takes and the streamed one with the autotuned tiling give the same fields and
the same first bad levels, bit for bit, over 30 steps."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_both_forms_at_full_size():
    from paper_0908_3749_gb300 import lbm
    B = W.tube_batch()
    nt, n, got = len(B["nx"]), 30, []
    b = lbm.lbm_batch_create(B["nx"], B["dx"], B["dt"], B["s"], B["left"], B["right"])
    try:
        for form in ("resident", "streamed"):
            lbm.lbm_batch_set_init(b, *W.tube_fields(B))
            if form == "streamed":
                lbm.lbm_batch_set_tiling(b, *lbm.lbm_batch_autotune(b, 5, None))
            assert lbm.lbm_batch_plan(b, n)[0] == (form == "resident")
            lbm.lbm_batch_step(b, n)
            out = [np.empty(lbm.lbm_batch_total_nodes(b)) for _ in range(4)]
            lbm.lbm_batch_moments(b, *out)
            got.append((out, lbm.lbm_batch_status(b, nt)))
    finally:
        lbm.lbm_batch_destroy(b)
    for p, q in zip(got[0][0], got[1][0]):
        np.testing.assert_array_equal(p, q)
    assert got[0][1][0] == got[1][1][0] == lbm.LBM_OK
    np.testing.assert_array_equal(got[0][1][1], got[1][1][1])
