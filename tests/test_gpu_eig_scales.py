"""GPU test of the eigenvalue solver on matrices whose entries differ in size by many
orders: columns below the diagonal scaled by 2^-400 to 2^-560, where sums of squares go
through the thresholds of the reflections and below the range of normal numbers. Bar:
1e-11 x norm, as for random matrices (numpy's eigenvalues of the same matrices)."""
import numpy as np
import pytest

from test_gpu_stability import _match

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [1, 10, 40])     # 16, 8 and 4 threads per matrix
@pytest.mark.parametrize("columns", [[0], [5], [13], [0, 1, 2], [2, 7, 11]])
def test_tiny_columns_below_the_diagonal(columns, copies):
    from paper_0908_3749_gb300 import lbm
    rng = np.random.default_rng(len(columns) * 100 + columns[0])
    exps = np.arange(400, 560, 2.5)
    A = rng.normal(size=(len(exps), 16, 16)) + 1j * rng.normal(size=(len(exps), 16, 16))
    for c in columns:
        A[:, c + 1:, c] *= 2.0 ** -exps[:, None]
    n = len(A)
    omega, radius, nf = lbm.lbm_eig16(np.tile(A, (copies, 1, 1)))
    assert nf == 0
    ref = np.linalg.eigvals(A)
    norm = np.linalg.norm(A, 2, axis=(1, 2))
    for c in {0, copies - 1}:
        for i in range(n):
            assert _match(omega[c * n + i], ref[i]) <= 1e-11 * norm[i], (c, exps[i])
            assert abs(radius[c * n + i] - np.abs(ref[i]).max()) <= 1e-11 * norm[i]
