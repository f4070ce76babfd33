"""The network's kernels at the edges of their tiles, against the FP64 oracle: 16 x 8 x 2 tiles (sides below 64: one
tile per box edge, a row that wraps on both sides at 16), 16 x 8 x 8 tiles (64 and 80: more tiles than one wave, an odd
number per row)."""
import numpy as np
import pytest

from oracle import nn as onn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 32, 48, 64, 80])
def test_forward_and_gradients_at_tile_edges(n):
    import torch
    from paper_1506_03737_gb300 import colapm as C
    rng = np.random.default_rng(n)
    psi = (rng.standard_normal((n ** 3, 3)) * 3.0).astype(np.float32)
    tgt = (rng.standard_normal((n ** 3, 3)) * 0.4).astype(np.float32)
    net = C.colapm_nn_create(n, C.nn_default_config(s_in=4.0, s_out=0.5, seed=n),
                             torch.cuda.current_stream().cuda_stream)
    try:
        dpsi, dtgt = torch.from_numpy(psi).cuda(), torch.from_numpy(tgt).cuda()
        out = torch.empty_like(dpsi)
        C.colapm_nn_forward(net, dpsi, out)
        g, loss = C.colapm_nn_grads(net, dpsi, dtgt)
        params = [(onn.bf16_round(w), b.astype(np.float32).astype(np.float64))
                  for w, b in onn.unflatten(C.colapm_nn_get_params(net).astype(np.float64))]
    finally:
        C.colapm_nn_destroy(net)
    x = onn.bf16_round(psi.reshape(n, n, n, 3).astype(np.float64) / 4.0)
    y, _ = onn.forward(x, params, onn.bf16_round)
    lref, gref = onn.loss_and_grads(x, tgt.reshape(n, n, n, 3).astype(np.float64) / 0.5, params, store=onn.bf16_round)
    # BF16-stored hidden activations and gradients (2^-9 per value): the bars of the other network tests
    err = np.linalg.norm(out.cpu().numpy().reshape(y.shape) - 0.5 * y) / np.linalg.norm(0.5 * y)
    assert err < 2e-3
    assert abs(loss / lref - 1) < 1e-4
    for (gw, gb), (rw, rb) in zip(onn.unflatten(g.astype(np.float64)), gref):
        assert np.linalg.norm(gw - rw) < 1e-2 * np.linalg.norm(rw)
        assert np.linalg.norm(gb - rb) < 1e-2 * np.linalg.norm(rb) + 1e-12
