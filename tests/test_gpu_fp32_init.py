"""GPU test of the FP32 initial state against the FP64 one rounded to FP32, bit for
bit: values on both sides of the range that the double-word form takes, zeros, tiny
velocities, infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _populations(arith, fields):
    from paper_0908_3749_gb300 import lbm
    ny, nx = fields[0].shape
    per = ("periodic", None)
    ctx = lbm.lbm_create(lbm.make_config(nx, ny, 0.01, 0.01, 1e-4, np.full(16, 1e3), (per,) * 4, arith))
    try:
        lbm.lbm_set_init(ctx, *fields)
        f = np.empty((16, ny, nx), np.float32 if arith == "fp32" else np.float64)
        lbm.lbm_get_populations(ctx, f)
        return f
    finally:
        lbm.lbm_destroy(ctx)


def _state(kind, shape, rng):
    rho = np.exp(rng.uniform(-2, 2, shape))
    u, v = rng.uniform(-3, 3, (2, *shape))
    T = np.exp(rng.uniform(-2, 2, shape))
    if kind == "at rest":
        u, v = np.zeros((2, *shape))
    elif kind == "x only":
        v = np.zeros(shape)
    elif kind == "cold":                    # groups whose terms cancel or vanish
        T = rng.choice([0.0, -0.5, 0.5, 1.0, 18.0], shape)
        u = rng.choice([0.0, 1.0, -6.0, 1e-9], shape)
    elif kind == "wide":                    # past both ends of the double-word form's range
        rho, u, v, T = (a * np.exp2(rng.uniform(-60, 25, shape)) for a in (rho, u, v, T))
    elif kind == "rounded":                 # FP32 values: empty second words
        rho, u, v, T = (a.astype(np.float32).astype(float) for a in (rho, u, v, T))
    return [np.ascontiguousarray(a) for a in (rho, u, v, T)]


@pytest.mark.parametrize("kind", ["any", "at rest", "x only", "cold", "wide", "rounded"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 5), (512, 256)])
def test_fp32_state_is_the_rounded_fp64_state(kind, nx, ny):
    fields = _state(kind, (ny, nx), np.random.default_rng(nx))
    with np.errstate(over="ignore"):
        want = _populations("fp64", fields).astype(np.float32)
    np.testing.assert_array_equal(_populations("fp32", fields), want)


def test_special_values():
    one = np.ones((4, 8))
    for k, x in enumerate((np.inf, -np.inf, np.nan, 0.0)):
        fields = [one.copy(), 0.1 * one, -0.2 * one, one.copy()]
        fields[k][1, 3] = x
        want = _populations("fp64", fields).astype(np.float32)
        np.testing.assert_array_equal(_populations("fp32", fields), want)
