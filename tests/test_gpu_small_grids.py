"""GPU test of the FP64 form with four threads per node around the largest grids that
take it: which launch runs, and the same bits as one thread per node, with audits
on no, some and every step (overlapped and plain launches)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

PER = ("periodic", None)
EQ = ("eq", (1.2, 0.25, -0.1, 1.1))
WALLS = (EQ, ("extrap", None), ("reflect", None), ("wall", (1.0, 0.2, 0.0, 0.9)))


def _run(w, blocks, audit):
    from paper_0908_3749_gb300 import lbm
    ctx = lbm.lbm_create(lbm.make_config(w.nx, w.ny, w.dx, w.dy, w.dt, w.s, w.bc, "fp64", audit))
    try:
        if blocks:
            lbm.lbm_set_step_blocks(ctx, blocks)
        g = lbm.lbm_step_blocks(ctx)
        lbm.lbm_set_init(ctx, *[np.ascontiguousarray(a) for a in w.fields()])
        lbm.lbm_step(ctx, 66)
        f = np.empty((16, w.ny, w.nx))
        step = lbm.lbm_get_populations(ctx, f)
        return g, f, step, lbm.lbm_audit_log(ctx), lbm.lbm_status(ctx)
    finally:
        lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("audit", [0, 1, 5])
@pytest.mark.parametrize("nx,ny,bc,lanes", [
    (9728, 1, (PER,) * 4, True), (2432, 4, (PER,) * 4, True), (2433, 4, (PER,) * 4, False),
    (97, 100, WALLS, True), (140, 100, WALLS, False), (200, 150, (PER,) * 4, False)])
def test_launch_and_bits_around_the_largest_small_grid(nx, ny, bc, lanes, audit):
    w = W.random_state(nx, ny, seed=nx + ny, bc=bc)
    a, b = (_run(w, blocks, audit) for blocks in (0, 1 << 20))
    assert b[0] == -(-nx // 32) * -(-ny // 2)
    assert a[0] == (8 if lanes else 1) * b[0]
    assert np.isfinite(a[1]).all()
    np.testing.assert_array_equal(a[1], b[1])
    assert a[2:] == b[2:]
