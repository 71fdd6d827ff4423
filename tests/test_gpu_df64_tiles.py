"""GPU test of the double-word step's two tile shapes, 32 x 4 (few tiles, or one to one
and a half 32 x 8 tiles per multiprocessor) and 32 x 8: a state that repeats along a
periodic y gives the same populations on a grid of one period (32 x 4) as on one of
several (32 x 8), bit for bit, period by period; with ragged edges, ghosts on the x
sides, one and several tiles per block, and audits. The audits' totals are FP32 pairs
(48 bits) summed in FP64, in another order: within 2^-40 of the sum of magnitudes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

PER = ("periodic", None)
EQ = ("eq", (1.2, 0.25, -0.1, 1.1))


def _run(w, fields, ny, audit, blocks):
    from paper_0908_3749_gb300 import lbm
    ctx = lbm.lbm_create(lbm.make_config(w.nx, ny, w.dx, w.dy, w.dt, w.s, w.bc, "df64", audit))
    try:
        tiles = lbm.lbm_step_blocks(ctx)
        if blocks:
            lbm.lbm_set_step_blocks(ctx, max(1, tiles // blocks))
        lbm.lbm_set_init(ctx, *[np.ascontiguousarray(a) for a in fields])
        lbm.lbm_step(ctx, 70)
        f = np.empty((16, ny, w.nx))
        lbm.lbm_get_populations(ctx, f)
        return tiles, f.view(np.uint64), lbm.lbm_audit_log(ctx), lbm.lbm_status(ctx)
    finally:
        lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("nx,ny,periods", [(200, 40, 3), (33, 9, 60), (1, 7, 300), (255, 180, 2), (600, 62, 4)])
@pytest.mark.parametrize("bc,audit,blocks", [((PER,) * 4, 0, 0), ((EQ, ("extrap", None), PER, PER), 3, 0),
                                             ((EQ, ("reflect", None), PER, PER), 1, 3)])
def test_tile_shapes_give_the_same_bits(nx, ny, periods, bc, audit, blocks):
    w = W.random_state(nx, ny, seed=nx + ny, bc=bc)
    fields = w.fields()
    a = _run(w, fields, ny, audit, blocks)
    b = _run(w, [np.tile(f, (periods, 1)) for f in fields], ny * periods, audit, blocks)
    tx = -(-nx // 32)
    assert a[0] == tx * -(-ny // 4) and b[0] == tx * -(-ny * periods // 8)
    np.testing.assert_array_equal(np.tile(a[1], (1, periods, 1)), b[1])
    assert a[2][1] == b[2][1] and a[3] == b[3]
    size = 50.0 * nx * ny * periods * w.dx * w.dy     # above the sum of the moments' magnitudes
    for p, q in zip(a[2][0], b[2][0]):
        np.testing.assert_allclose(np.array(p) * periods, q, rtol=0, atol=2.0 ** -40 * size)
