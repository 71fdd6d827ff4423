"""GPU tests of the corrector's convolution and weight-gradient tiles (8 rows x
32 pixels with a halo of one) at sizes where a tile can go wrong: one pixel,
one row or column, one tile exactly, one pixel more and less, several tiles
with ragged edges.

Gradients and corrected features against the FP64 CPU reference run with the
same BF16 rounding of parameters, activations and output gradients. What is left
is the FP32 accumulation order (288 products of a dot product: relative error
below 288 x 2^-24 = 1.8e-5) and single BF16 roundings that it tips over (2^-8
of one value each): the bar is a relative L2 error of 2e-3."""
import numpy as np
import pytest

from oracle import cnn
from test_gpu_corrector import _bf16, _fields, _unpack

pytestmark = pytest.mark.gpu

BAR = 2e-3


@pytest.mark.parametrize("H,W", [(1, 1), (1, 70), (40, 1), (7, 31), (8, 32), (9, 33), (17, 65),
                                 (24, 96), (130, 100)])
def test_tile_edges_match_cpu_reference(H, W):
    import torch
    from paper_0908_3749_gb300 import corrector, lbm
    rng = np.random.default_rng(H * 1000 + W)
    params = corrector.init_params(5)
    for w, b in _unpack(params):
        b[...] = rng.standard_normal(b.shape) * 0.1
    last = _unpack(params)[-1][0]
    last[...] = rng.standard_normal(last.shape) * 0.05
    coarse, target = _fields(rng, H, W), _fields(rng, H, W)
    scale = (0.5, 2.0, 1.0, 0.25)
    dc, dt = (torch.tensor(a, device="cuda") for a in (coarse, target))
    out = torch.empty_like(dc)
    net = lbm.lbm_cnn_create(H, W)
    try:
        lbm.lbm_cnn_set_params(net, params)
        lbm.lbm_cnn_set_output_scale(net, scale)
        loss, g = lbm.lbm_cnn_loss_grad(net, dc, dt)
        fallback = lbm.lbm_cnn_correct(net, dc, out, mass_tol=1e6)
    finally:
        lbm.lbm_cnn_destroy(net)
    ref_params = [(w.astype(np.float64) if l == 0 else _bf16(w), b.astype(np.float64))
                  for l, (w, b) in enumerate(_unpack(params))]
    x = cnn.features(*coarse).astype(np.float32).astype(np.float64)
    t = cnn.features(*target).astype(np.float32).astype(np.float64)
    rloss, rgrads = cnn.loss_and_grads(x, t, ref_params, x_res=x, store=cnn.bf16, scale=scale)
    assert abs(loss - rloss) <= 1e-5 * rloss, (loss, rloss)
    for l, (gw, gb) in enumerate(_unpack(g.astype(np.float64))):
        for got, ref in ((gw, rgrads[l][0]), (gb, rgrads[l][1])):
            assert np.linalg.norm(got - ref) <= BAR * max(np.linalg.norm(ref), 1e-30), l
    rout, _ = cnn.forward(x, ref_params, x_res=x, store=cnn.bf16, scale=scale)
    got = cnn.features(*out.cpu().numpy())
    assert not fallback
    for c in range(4):  # relative to the correction, which the network computes
        assert np.linalg.norm(got[..., c] - rout[..., c]) <= BAR * np.linalg.norm(rout[..., c] - x[..., c]), c
