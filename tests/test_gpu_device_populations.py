"""GPU test of the populations' copies to and from device arrays, bit for bit against the
host ones: rows joined into flat arrays, 16-byte pieces, single elements, and arrays
that are not aligned to 16 bytes, to an element, or (pairs of floats at an odd
offset) to the element size."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

HOST = {"fp64": np.float64, "fp32": np.float32, "df64": np.float64}


@pytest.mark.parametrize("arith", ["fp32", "fp64", "df64"])
@pytest.mark.parametrize("offset", [0, 1, 2, 4])     # 4-byte words
@pytest.mark.parametrize("nx,ny", [(64, 12), (32, 1), (96, 5), (36, 7), (33, 9), (1, 3), (520, 40)])
def test_device_arrays_equal_host_arrays(arith, nx, ny, offset):
    import torch
    from paper_0908_3749_gb300 import lbm
    w = W.random_state(nx, ny, seed=nx * ny + offset)
    cfg = lbm.make_config(w.nx, w.ny, w.dx, w.dy, w.dt, w.s, w.bc, arith, 0)
    words = 16 * ny * nx * np.dtype(HOST[arith]).itemsize // 4
    a, b = lbm.lbm_create(cfg), lbm.lbm_create(cfg)
    try:
        lbm.lbm_set_init(a, *[np.ascontiguousarray(x) for x in w.fields()])
        lbm.lbm_step(a, 3)
        host = np.empty((16, ny, nx), HOST[arith])
        assert lbm.lbm_get_populations(a, host) == 3
        buf = torch.full((words + 8,), -7.0, device="cuda", dtype=torch.float32)
        assert lbm.lbm_get_populations(a, buf[offset:offset + words]) == 3
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[offset:offset + words].view(np.uint32), host.reshape(-1).view(np.uint32))
        assert (got[:offset] == -7).all() and (got[offset + words:] == -7).all()
        lbm.lbm_set_populations(b, buf[offset:offset + words], 3)
        back = np.empty_like(host)
        assert lbm.lbm_get_populations(b, back) == 3
        np.testing.assert_array_equal(back.view(np.uint8), host.view(np.uint8))
        lbm.lbm_step(a, 2)
        lbm.lbm_step(b, 2)
        lbm.lbm_get_populations(a, host)
        lbm.lbm_get_populations(b, back)
        np.testing.assert_array_equal(back.view(np.uint8), host.view(np.uint8))
    finally:
        lbm.lbm_destroy(a)
        lbm.lbm_destroy(b)


def test_managed_and_pinned_memory_go_through_the_copy_engine():
    import torch
    from paper_0908_3749_gb300 import lbm
    w = W.random_state(40, 6, seed=5)
    ctx = lbm.lbm_create(lbm.make_config(w.nx, w.ny, w.dx, w.dy, w.dt, w.s, w.bc, "fp64", 0))
    try:
        lbm.lbm_set_init(ctx, *[np.ascontiguousarray(x) for x in w.fields()])
        host = np.empty((16, 6, 40))
        lbm.lbm_get_populations(ctx, host)
        pinned = torch.zeros((16, 6, 40), dtype=torch.float64).pin_memory()
        import ctypes
        step = ctypes.c_longlong()
        rc = lbm.load().lbm_get_populations(ctx, ctypes.c_void_p(pinned.data_ptr()), ctypes.byref(step), 1)
        assert rc == lbm.LBM_OK and step.value == 0
        np.testing.assert_array_equal(pinned.numpy(), host)
    finally:
        lbm.lbm_destroy(ctx)
