"""GPU test of the amplification matrices written by blocks of eight: numbers of matrices
around that, several wave vectors and cases per block, an output aligned to doubles
only; every matrix the same as computed alone, bit for bit, and nothing written
beyond the last."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,nk", [(1, 1), (1, 7), (1, 8), (3, 3), (5, 5), (2, 40), (17, 1)])
def test_blocks_of_matrices(nc, nk):
    import torch
    from paper_0908_3749_gb300 import lbm
    rng = np.random.default_rng(nc * 100 + nk)
    states = np.stack([rng.uniform(0.5, 2, nc), rng.uniform(-1, 1, nc), rng.uniform(-1, 1, nc),
                       rng.uniform(0.5, 2, nc)], 1)
    cases, k = lbm.vn_cases(states, 10.0 ** rng.uniform(3, 5, (nc, 16))), rng.uniform(-800, 800, (nk, 2))
    dx, dy, dt = 2e-3, 3e-3, 1e-5
    all_ = lbm.lbm_vn_matrices(cases, k, dx, dy, dt)
    for c in range(nc):
        for q in range(nk):
            one = lbm.lbm_vn_matrices(cases[c:c + 1], k[q:q + 1], dx, dy, dt)
            np.testing.assert_array_equal(all_[c, q], one[0, 0])
    n = nc * nk * 512
    buf = torch.full((n + 4,), -7.0, device="cuda", dtype=torch.float64)
    lbm.lbm_vn_matrices(torch.tensor(cases, device="cuda"), torch.tensor(k, device="cuda"), dx, dy, dt, buf[1:n + 1])
    got = buf.cpu().numpy()
    np.testing.assert_array_equal(got[1:n + 1].view(np.complex128).reshape(all_.shape), all_)
    assert got[0] == -7 and (got[n + 1:] == -7).all()
    # the spectra are these matrices'
    radius, _, _ = lbm.lbm_vn_spectrum(cases, k, dx, dy, dt)
    want = np.abs(np.linalg.eigvals(all_)).max(-1)
    assert np.abs(radius - want).max() <= 1e-11 * np.abs(all_).sum(-1).max()
