"""GPU test of the corrector's bounded waits (test hook: the waits for copies, for
products or for both expire at once): the call reports LBM_ERR_TIMEOUT, the
parameters and the Adam state stay those before the step, also over several steps
without a report, and what follows is what a network without the incident computes,
bit for bit. Sizes: one tile, and several tiles per CTA."""
import numpy as np
import pytest

from test_gpu_corrector import _fields

pytestmark = pytest.mark.gpu


def _params(net):
    from paper_0908_3749_gb300 import lbm
    p = np.empty(lbm.CNN_NPARAMS, np.float32)
    lbm.lbm_cnn_get_params(net, p)
    return p


@pytest.mark.parametrize("which", [1, 2, 3])
@pytest.mark.parametrize("H,W", [(9, 12), (800, 640)])
def test_an_expired_wait_leaves_the_network_as_it_was(H, W, which):
    import torch
    from paper_0908_3749_gb300 import corrector, lbm
    rng = np.random.default_rng(H)
    c, t = (torch.tensor(_fields(rng, H, W), device="cuda") for _ in range(2))
    out, ref = torch.empty_like(c), torch.empty_like(c)
    nets = [lbm.lbm_cnn_create(H, W) for _ in range(2)]
    a, b = nets

    def expires(call):
        with pytest.raises(lbm.LBMError) as e:
            call()
        assert e.value.code == lbm.LBM_ERR_TIMEOUT
    try:
        for n in nets:
            lbm.lbm_cnn_set_params(n, corrector.init_params(3))
            lbm.lbm_cnn_train_step(n, c, t)
        one = _params(a)
        np.testing.assert_array_equal(one, _params(b))
        lbm.lbm_cnn_debug_give_up(a, which)
        expires(lambda: lbm.lbm_cnn_train_step(a, c, t))
        np.testing.assert_array_equal(_params(a), one)
        expires(lambda: lbm.lbm_cnn_loss_grad(a, c, t))
        expires(lambda: lbm.lbm_cnn_correct(a, c, out))
        for _ in range(3):
            lbm.lbm_cnn_train_step(a, c, t, want_loss=False)
        lbm.lbm_cnn_debug_give_up(a, 0)
        np.testing.assert_array_equal(_params(a), one)
        expires(lambda: lbm.lbm_cnn_train_step(a, c, t))    # reports the three before it
        np.testing.assert_array_equal(_params(a), one)
        for _ in range(2):
            assert lbm.lbm_cnn_train_step(a, c, t) == lbm.lbm_cnn_train_step(b, c, t)
        np.testing.assert_array_equal(_params(a), _params(b))
        assert lbm.lbm_cnn_correct(a, c, out, mass_tol=1e6) == lbm.lbm_cnn_correct(b, c, ref, mass_tol=1e6)
        assert torch.equal(out, ref)
        # new parameters forget an expired wait
        lbm.lbm_cnn_debug_give_up(a, which)
        lbm.lbm_cnn_train_step(a, c, t, want_loss=False)
        lbm.lbm_cnn_debug_give_up(a, 0)
        for n in nets:
            lbm.lbm_cnn_set_params(n, corrector.init_params(4))
        assert lbm.lbm_cnn_train_step(a, c, t) == lbm.lbm_cnn_train_step(b, c, t)
        np.testing.assert_array_equal(_params(a), _params(b))
    finally:
        for n in nets:
            lbm.lbm_cnn_destroy(n)
