"""GPU test of the batched 16 x 16 eigenvalue solver over the batch sizes at
which it changes its threads per matrix (16, 8 or 4: two, four or eight matrices
per warp, in step) and over matrices that behave differently in one warp:
random, triangular, scaled to the ends of the range, with tiny and zero entries,
defective, not finite.

Bars: 1e-11 x norm for well-conditioned (random) spectra, as for single
matrices; for a Jordan block the eigenvalue moves by up to (norm x rounding)^(1/16)
= (16 x 2^-50)^(1/16) = 0.14, so that only its trace is compared (within 16 x
16 x 2^-52 x norm)."""
import numpy as np
import pytest

from test_gpu_stability import _match

pytestmark = pytest.mark.gpu


def _lines():
    import torch
    warps = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    return [1, 7, 8, 9, 2 * warps, 2 * warps + 1, 4 * warps, 4 * warps + 1, 4 * warps + 13]


@pytest.mark.parametrize("which", range(9))
def test_batch_sizes(which):
    from paper_0908_3749_gb300 import lbm
    n = _lines()[which]
    rng = np.random.default_rng(which)
    A = rng.normal(size=(n, 16, 16)) + 1j * rng.normal(size=(n, 16, 16))
    omega, radius, nf = lbm.lbm_eig16(A)
    assert nf == 0
    ref = np.linalg.eigvals(A)
    norm = np.linalg.norm(A, 2, axis=(1, 2))
    assert np.all(np.abs(radius - np.abs(ref).max(1)) <= 1e-11 * norm)
    assert np.all(np.abs(omega.sum(1) - np.trace(A, axis1=1, axis2=2)) <= 1e-11 * norm)
    for i in {0, n // 2, n - 1}:
        assert _match(omega[i], ref[i]) <= 1e-11 * norm[i]


@pytest.mark.parametrize("copies", [1, 80, 160])
def test_unlike_matrices_in_one_warp(copies):
    """The same 20 matrices in batches with 16, 8 and 4 threads per matrix."""
    from paper_0908_3749_gb300 import lbm
    rng = np.random.default_rng(9)
    kinds = []
    for k in range(8):
        A = rng.normal(size=(16, 16)) + 1j * rng.normal(size=(16, 16))
        kinds.append(A * 10.0 ** rng.integers(-3, 4))
    kinds += [np.triu(kinds[0]), np.tril(kinds[1]), np.diag(np.diag(kinds[2])), np.zeros((16, 16)),
              np.eye(16) * (2 + 1j), kinds[3] * 1e300, kinds[4] * 1e-300]
    T = kinds[5].copy()
    T[np.tril_indices(16, -2)] *= 1e-200        # Hessenberg but for tiny entries
    B = np.zeros((16, 16), complex)
    B[:8, :8], B[8:, 8:] = kinds[6][:8, :8], kinds[7][:8, :8]   # two decoupled blocks
    J = np.eye(16) * 0.5 + np.diag(np.ones(15), 1)              # one Jordan block
    N = kinds[0].copy()
    N[3, 5] = np.inf
    kinds += [T, B, J.T, N, J]
    kinds = np.array(kinds)
    n = len(kinds)
    omega, radius, nf = lbm.lbm_eig16(np.tile(kinds, (copies, 1, 1)))
    assert nf == copies
    for c in {0, copies // 2, copies - 1}:
        for i, A in enumerate(kinds):
            w, r = omega[c * n + i], radius[c * n + i]
            if not np.isfinite(A).all():
                assert np.isnan(w).all() and np.isnan(r)
                continue
            norm = np.linalg.norm(A, 2)
            if i in (n - 3, n - 1):
                assert abs(w.sum() - np.trace(A)) <= 256 * 2.0 ** -52 * norm
            else:
                assert _match(w, np.linalg.eigvals(A)) <= 1e-11 * norm, (c, i)
