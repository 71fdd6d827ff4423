"""GPU test of lbm_step_blocks: the blocks of the launch that runs, and a value that
selects the same launch when it is set again, for every default: four threads per
node (small FP64 grids), one tile per block, several tiles per block (large FP32 and
double-word grids), and after the autotuner."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TILE_ROWS = {"fp64": 2, "fp32": 8, "df64": 8}


def _ctx(arith, nx, ny):
    from paper_0908_3749_gb300 import lbm
    w = W.random_state(nx, ny, seed=nx + ny)
    ctx = lbm.lbm_create(lbm.make_config(w.nx, w.ny, w.dx, w.dy, w.dt, w.s, w.bc, arith, 0))
    lbm.lbm_set_init(ctx, *[np.ascontiguousarray(a) for a in w.fields()])
    return ctx


def _tiles(arith, nx, ny):
    return -(-nx // 32) * -(-ny // TILE_ROWS[arith])


@pytest.mark.parametrize("arith,nx,ny,per_tile", [
    ("fp64", 200, 4, 8.0), ("fp64", 2048, 64, 1.0), ("fp32", 600, 200, 1.0),
    ("fp32", 1600, 1600, 1 / 6), ("df64", 1030, 1001, 1 / 3)])
def test_reported_blocks_are_the_launch_and_round_trip(arith, nx, ny, per_tile):
    from paper_0908_3749_gb300 import lbm
    n = _tiles(arith, nx, ny)
    ctx = _ctx(arith, nx, ny)
    try:
        g = lbm.lbm_step_blocks(ctx)
        if per_tile < 1:
            assert g < n and abs(g - n * per_tile) <= 0.2 * n * per_tile  # 6 or 7 tiles, 3 tiles
        else:
            assert g == n * per_tile
        lbm.lbm_set_step_blocks(ctx, g)
        assert lbm.lbm_step_blocks(ctx) == g
        lbm.lbm_set_step_blocks(ctx, 1 << 20)
        assert lbm.lbm_step_blocks(ctx) == n
        lbm.lbm_set_step_blocks(ctx, 0)
        assert lbm.lbm_step_blocks(ctx) == g
        tuned = lbm.lbm_autotune(ctx, 3)
        lbm.lbm_set_step_blocks(ctx, tuned)
        assert lbm.lbm_step_blocks(ctx) == tuned
    finally:
        lbm.lbm_destroy(ctx)
