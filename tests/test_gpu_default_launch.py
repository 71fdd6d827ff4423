"""GPU test of the default launch of large FP32 and double-word grids (several tiles per
block) against one tile per block, bit for bit: populations, audit log and watchdog,
around the number of tiles from which it is taken, with ragged edges."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

BC = (("eq", (1.2, 0.25, -0.1, 1.1)), ("extrap", None), ("reflect", None), ("outflow", None))


def _run(w, arith, blocks):
    from paper_0908_3749_gb300 import lbm
    ctx = lbm.lbm_create(lbm.make_config(w.nx, w.ny, w.dx, w.dy, w.dt, w.s, w.bc, arith, 3))
    try:
        if blocks:
            lbm.lbm_set_step_blocks(ctx, blocks)
        lbm.lbm_set_init(ctx, *[np.ascontiguousarray(a) for a in w.fields()])
        lbm.lbm_step(ctx, 7)
        f = np.empty((16, w.ny, w.nx), np.float32 if arith == "fp32" else np.float64)
        step = lbm.lbm_get_populations(ctx, f)
        return f.view(np.uint32), step, lbm.lbm_audit_log(ctx), lbm.lbm_status(ctx)
    finally:
        lbm.lbm_destroy(ctx)


# 32 x 8 tiles: 4 x 999 and 4 x 1000 (double-word), 50 x 100 - 1 column, 50 x 100 (FP32),
# 64 x 96 (6 would return to the same column), 47 x 113 ragged.
@pytest.mark.parametrize("arith,nx,ny", [("df64", 128, 8 * 999), ("df64", 128, 8 * 1000), ("df64", 1030, 1001),
                                         ("fp32", 32 * 49, 800), ("fp32", 32 * 50, 800), ("fp32", 2048, 768),
                                         ("fp32", 1501, 899)])
def test_default_launch_equals_one_tile_per_block(arith, nx, ny):
    w = W.random_state(nx, ny, seed=nx + ny, bc=BC)
    a, b = (_run(w, arith, blocks) for blocks in (0, 1 << 20))
    np.testing.assert_array_equal(a[0], b[0])
    assert a[1:] == b[1:]
