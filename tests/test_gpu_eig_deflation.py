"""GPU test of the eigenvalue solver's deflation beside diagonal entries at the lower end
of the range: decoupled entries and blocks of 2^-940 to 2^-1060 next to ones of
order 1 deflate at once (a zero below the diagonal is negligible however small the
diagonal is). Eigenvalues of diagonal matrices are their entries, to a relative
2^-50 where these are normal numbers after the solver's scaling."""
import numpy as np
import pytest

from test_gpu_stability import _match

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [1, 100, 300])     # 16, 8 and 4 threads per matrix
def test_tiny_decoupled_entries(copies):
    from paper_0908_3749_gb300 import lbm
    rng = np.random.default_rng(4)
    mats = []
    for e in (940, 970, 975, 980, 1000, 1019, 1030, 1060):
        d = rng.uniform(1, 2, 16) * 2.0 ** -float(e)
        d[rng.integers(0, 16)] = 1.0
        mats.append(np.diag(d).astype(complex))
        A = np.diag(d).astype(complex)                # a block of order 1 among them
        A[:5, :5] = rng.normal(size=(5, 5)) + 1j * rng.normal(size=(5, 5))
        mats.append(A)
        mats.append(np.triu(A))
    A = np.array(mats)
    n = len(A)
    omega, radius, nf = lbm.lbm_eig16(np.tile(A, (copies, 1, 1)))
    assert nf == 0
    for i in range(n):
        w = omega[(copies - 1) * n + i]
        assert _match(w, np.linalg.eigvals(A[i])) <= 1e-11 * np.linalg.norm(A[i], 2), i
        if i % 3 == 0:
            want = np.sort(np.diag(A[i]).real)
            np.testing.assert_allclose(np.sort(w.real), want, rtol=2.0 ** -50, atol=2.0 ** -1060)
            assert (w.imag == 0).all()
