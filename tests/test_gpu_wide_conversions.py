"""GPU test of the conversions between FP64 and the narrower population formats, bit
for bit: the FP32-pair initial state against the FP64 one split on the host, and the
moments of FP32 and FP32-pair populations against those of the same numbers in FP64;
values with ties, carries into the exponent, zeros and numbers outside the range of
the integer conversions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NY, NX = 37, 131


def _ctx(arith):
    from paper_0908_3749_gb300 import lbm
    return lbm.lbm_create(lbm.make_config(NX, NY, 0.01, 0.01, 1e-4, np.full(16, 1e3),
                                          (("periodic", None),) * 4, arith))


def _initial(arith, fields):
    from paper_0908_3749_gb300 import lbm
    ctx = _ctx(arith)
    try:
        lbm.lbm_set_init(ctx, *fields)
        f = np.empty((16, NY, NX), np.float32 if arith == "fp32" else np.float64)
        lbm.lbm_get_populations(ctx, f)
        return f
    finally:
        lbm.lbm_destroy(ctx)


def _moments(arith, f):
    from paper_0908_3749_gb300 import lbm
    ctx = _ctx(arith)
    try:
        lbm.lbm_set_populations(ctx, f, 0)
        out = [np.empty((NY, NX)) for _ in range(4)]
        lbm.lbm_moments(ctx, *out)
        return np.stack(out)
    finally:
        lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("scale", [0, -30, 30, -70, 58, 64, -130])
def test_double_word_state_is_the_nearest_split(scale):
    rng = np.random.default_rng(scale + 200)
    rho, T = np.exp(rng.uniform(-2, 2, (2, NY, NX))) * 2.0 ** (scale // 2)
    u, v = rng.choice([0.0, 1.0, -6.0, 0.37], (2, NY, NX)) * rng.choice([1.0, 2.0 ** -24, 1 / 3], (2, NY, NX))
    fields = [np.ascontiguousarray(a) for a in (rho, u, v, T)]
    f = _initial("fp64", fields)
    assert np.isfinite(f.astype(np.float32)).all()
    h = f.astype(np.float32)
    want = np.stack([h, (f - h).astype(np.float32)], -1)
    got = _initial("df64", fields).view(np.float32).reshape(want.shape)
    np.testing.assert_array_equal(got.view(np.uint32), want.view(np.uint32))


def _numbers(rng, shape):
    m = rng.choice([1.0, 1.5, 2.0 - 2.0 ** -23, 1.0 + 2.0 ** -23, np.pi / 2], shape)
    x = (m * rng.choice([0.0, 1.0, -1.0], shape) * np.exp2(rng.integers(-20, 20, shape))).astype(np.float32)
    x[rng.random(shape) < 0.01] = np.float32(1e-41)          # subnormal
    x[rng.random(shape) < 0.001] = np.inf
    x[rng.random(shape) < 0.001] = np.nan
    return x


@pytest.mark.parametrize("arith", ["fp32", "df64"])
def test_moments_are_those_of_the_widened_populations(arith):
    rng = np.random.default_rng(5)
    h = _numbers(rng, (16, NY, NX))
    if arith == "fp32":
        f, wide = h, h.astype(np.float64)
    else:
        with np.errstate(invalid="ignore"):
            l = np.where(np.isfinite(h), _numbers(rng, h.shape) * np.float32(2.0 ** -26) * np.abs(h), np.float32(0))
            wide = h.astype(np.float64) + l.astype(np.float64)
        f = np.ascontiguousarray(np.stack([h, l], -1)).view(np.float64)[..., 0]
    np.testing.assert_array_equal(_moments(arith, np.ascontiguousarray(f)), _moments("fp64", wide))
