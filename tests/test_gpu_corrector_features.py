"""GPU test of the corrector's logarithms: the features log rho and log T are
the FP64 logarithms rounded to FP32, bit for bit, whatever the magnitude.

lbm_cnn_residual_rms returns sqrt(mean (t - x)^2) of the FP32 features: against
coarse fields of 1 (features exactly 0) on a one-pixel image it is |log32(rho)|
exactly (one square and one square root, each correctly rounded: below 2^-52)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _values():
    rng = np.random.default_rng(3)
    v = [np.exp(rng.uniform(-2.4, 2.4, 3000)), np.exp(rng.uniform(-700, 700, 1000)),
         1 + rng.uniform(-1, 1, 1000) * 10.0 ** rng.uniform(-16, -2, 1000),
         np.array([1.0, 0.5, 2.0, np.sqrt(0.5), np.nextafter(np.sqrt(0.5), 0), np.sqrt(2.0),
                   np.nextafter(1, 0), np.nextafter(1, 2), 2.0 ** -1022, 5e-324, 1.7e308]),
         np.arange(90, 184) / 128.0, (np.arange(90, 184) + 0.5) / 128.0]
    return np.concatenate(v)


def test_log_features_are_the_rounded_fp64_logarithms():
    import torch
    from paper_0908_3749_gb300 import lbm
    vals = _values()
    ref = np.log(vals).astype(np.float32).astype(np.float64)
    one = torch.ones((4, 1, 1), dtype=torch.float64, device="cuda")
    one[1:3] = 0.0
    net = lbm.lbm_cnn_create(1, 1)
    got = np.empty((len(vals), 2))
    try:
        dev = torch.ones((len(vals), 4, 1, 1), dtype=torch.float64, device="cuda")
        dev[:, 1:3] = 0.0
        dev[:, 0, 0, 0] = torch.tensor(vals, device="cuda")
        dev[:, 3, 0, 0] = torch.tensor(vals[::-1].copy(), device="cuda")
        for k in range(len(vals)):
            r = lbm.lbm_cnn_residual_rms(net, one, dev[k])
            got[k] = r[0], r[3]
    finally:
        lbm.lbm_cnn_destroy(net)
    np.testing.assert_allclose(got[:, 0], np.abs(ref), rtol=2.0 ** -51, atol=0)
    np.testing.assert_allclose(got[::-1, 1], np.abs(ref), rtol=2.0 ** -51, atol=0)


@pytest.mark.parametrize("bad", [0.0, -1.0, np.inf, np.nan])
def test_log_features_of_invalid_values_are_log_s(bad):
    import torch
    from paper_0908_3749_gb300 import lbm
    f = torch.ones((4, 1, 1), dtype=torch.float64, device="cuda")
    f[1:3] = 0.0
    g = f.clone()
    g[0] = bad
    net = lbm.lbm_cnn_create(1, 1)
    try:
        r = lbm.lbm_cnn_residual_rms(net, f, g)
    finally:
        lbm.lbm_cnn_destroy(net)
    with np.errstate(all="ignore"):
        ref = np.abs(np.log(bad))
    assert np.isnan(r[0]) if np.isnan(ref) else r[0] == ref


def test_corrected_fields_are_the_exponentials_of_the_features():
    """With zero parameters the corrected density and temperature are exp of the
    FP32 logarithms: within 0.6 units in the last place of the true value, numpy's
    exp within one, so 2 x 2^-52 relative between them; the sums of the density
    agree with the fallback's mass test (no fallback at 1e-6: the logarithm's FP32
    rounding changes the density by at most 2^-24 |log|)."""
    import torch
    from paper_0908_3749_gb300 import lbm
    vals = _values()
    vals = vals[(vals > 1e-307) & (vals < 1e307)]
    for part in (vals, np.exp(np.random.default_rng(4).uniform(-2, 2, 70000))):
        f = np.stack([part, np.linspace(-1, 1, len(part)), np.zeros(len(part)), part[::-1]])[:, None, :]
        coarse = torch.tensor(f, device="cuda")
        out = torch.empty_like(coarse)
        net = lbm.lbm_cnn_create(1, len(part))
        try:
            fallback = lbm.lbm_cnn_correct(net, coarse, out, mass_tol=700 * 2.0 ** -24)
            again = torch.empty_like(coarse)
            lbm.lbm_cnn_correct(net, coarse, again, mass_tol=700 * 2.0 ** -24)
        finally:
            lbm.lbm_cnn_destroy(net)
        assert not fallback and torch.equal(out, again)
        ref = np.exp(np.log(part).astype(np.float32).astype(np.float64))
        got = out.cpu().numpy()
        np.testing.assert_allclose(got[0, 0], ref, rtol=2.0 ** -51, atol=0)
        np.testing.assert_allclose(got[3, 0], ref[::-1], rtol=2.0 ** -51, atol=0)
        np.testing.assert_array_equal(got[1, 0], f[1, 0].astype(np.float32))


def test_a_non_finite_output_falls_back():
    import torch
    from paper_0908_3749_gb300 import lbm
    coarse = torch.ones((4, 3, 300), dtype=torch.float64, device="cuda")
    coarse[1, 2, 299] = float("inf")
    out = torch.zeros_like(coarse)
    net = lbm.lbm_cnn_create(3, 300)
    try:
        assert lbm.lbm_cnn_correct(net, coarse, out)
        assert torch.equal(out, coarse)
        coarse[1, 2, 299] = 0.0
        assert not lbm.lbm_cnn_correct(net, coarse, out)
    finally:
        lbm.lbm_cnn_destroy(net)
