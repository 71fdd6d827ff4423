"""GPU test of the FP64 step with four lanes per node (small grids) against the
one with a thread per node, bit for bit: populations, audit log and watchdog, on
grids around its tiles of 8 nodes of a 32 x 2 tile, with every boundary kind, a
side that switches kind, unequal spacings and a state that goes unphysical."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

PER = ("periodic", None)
EQ = ("eq", (1.2, 0.25, -0.1, 1.1))
SIDES = {
    "periodic": (PER, PER, PER, PER),
    "mixed": (EQ, ("extrap", None), ("reflect", None), ("wall", (1.0, 0.2, 0.0, 0.9))),
    "open": (("outflow", None), ("extrap", None), ("outflow", None), ("extrap", None)),
    "x_only": (("reflect", None), EQ, PER, PER),
    "y_only": (PER, PER, ("wall", (1.0, -0.3, 0.1, 1.2)), ("reflect", None)),
    "split": (EQ, ("extrap", None), ("eq", EQ[1], ("reflect", 0.05, 0.0)),
              ("eq", EQ[1], ("extrap", 0.04, 300.0))),
}


def _run(w, blocks, nsteps, audit, dy=None):
    from paper_0908_3749_gb300 import lbm
    cfg = lbm.make_config(w.nx, w.ny, w.dx, dy or w.dy, w.dt, w.s, w.bc, "fp64", audit)
    ctx = lbm.lbm_create(cfg)
    try:
        if blocks:
            lbm.lbm_set_step_blocks(ctx, blocks)
        lbm.lbm_set_init(ctx, *[np.ascontiguousarray(a) for a in w.fields()])
        lbm.lbm_step(ctx, nsteps)
        f = np.empty((16, w.ny, w.nx))
        step = lbm.lbm_get_populations(ctx, f)
        return f, step, lbm.lbm_audit_log(ctx), lbm.lbm_status(ctx)
    finally:
        lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (2, 2), (7, 5), (8, 2), (31, 3), (32, 2),
                                   (33, 7), (65, 16), (200, 4)])
def test_lanes_equal_one_thread_per_node(sides, nx, ny):
    w = W.random_state(nx, ny, seed=nx * 100 + ny, bc=SIDES[sides])
    dy = 0.013 if (nx + ny) % 2 else None
    a, b = (_run(w, blocks, 70, 3, dy) for blocks in (0, 1 << 20))
    assert np.isfinite(a[0]).all()
    np.testing.assert_array_equal(a[0], b[0])
    assert a[1:] == b[1:]


def test_unphysical_state_is_reported_alike():
    w = W.sod_config1("literal")             # rho <= 0 at time level 1122 (oracle)
    a, b = (_run(w, blocks, 1200, 0) for blocks in (0, 1 << 20))
    assert a[3] == b[3] and a[3][0] != 0 and abs(a[3][1] - 1122) <= 5
    np.testing.assert_array_equal(a[0], b[0])
