"""GPU test of the corrector's buffers: networks of several sizes alive at once, created
and destroyed in turn by several threads, keep their results apart and compute what
a network alone computes, bit for bit."""
import threading

import numpy as np
import pytest

from test_gpu_corrector import _fields

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (9, 12), (17, 65), (40, 33)]


def _losses(h, w, steps):
    import torch
    from paper_0908_3749_gb300 import corrector, lbm
    rng = np.random.default_rng(h * w)
    c, t = (torch.tensor(_fields(rng, h, w), device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    net = lbm.lbm_cnn_create(h, w)
    try:
        lbm.lbm_cnn_set_params(net, corrector.init_params(2))
        out = [lbm.lbm_cnn_train_step(net, c, t) for _ in range(steps)]
        rms = lbm.lbm_cnn_residual_rms(net, c, t)
        p = np.empty(lbm.CNN_NPARAMS, np.float32)
        lbm.lbm_cnn_get_params(net, p)
        return out, rms, p
    finally:
        lbm.lbm_cnn_destroy(net)


def test_many_networks_in_several_threads():
    alone = [_losses(h, w, 3) for h, w in SIZES]
    failed = []

    def work(k):
        try:
            for r in range(12):
                i = (k + r) % len(SIZES)
                got = _losses(*SIZES[i], 3)
                assert got[0] == alone[i][0] and got[1] == alone[i][1]
                np.testing.assert_array_equal(got[2], alone[i][2])
        except BaseException as e:  # noqa: B902 - handed to the main thread
            failed.append(e)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]


def test_more_networks_than_a_page_of_results():
    from paper_0908_3749_gb300 import corrector, lbm
    import torch
    nets = [lbm.lbm_cnn_create(2, 3) for _ in range(130)]
    try:
        rng = np.random.default_rng(0)
        c, t = (torch.tensor(_fields(rng, 2, 3), device="cuda") for _ in range(2))
        losses = set()
        for n in nets:
            lbm.lbm_cnn_set_params(n, corrector.init_params(2))
            losses.add(lbm.lbm_cnn_loss_grad(n, c, t)[0])
        assert len(losses) == 1
    finally:
        for n in nets:
            lbm.lbm_cnn_destroy(n)
