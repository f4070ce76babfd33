"""The network's loss over the whole range of the errors, against FP64: ordinary ones, squares beyond the range of a float on
either side, a mixture within a tile, none, and infinities; both tile shapes and the tensor-core engine.

Tolerance: the twelve squares of a lane's tile are summed with their rounding errors (36 FP32 additions of errors below
36 x 2^-25 of the sum: 2.3e-12 of it at worst), the tiles and lanes in FP64 (below 4e-11 for 3 x 48^3 terms if every
rounding went one way, a thousandth of that as they fall): 4e-12."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(n, target, zero=False, engine=0):
    import torch

    from paper_1506_03737_gb300 import colapm as C
    nn = C.colapm_nn_create(n, C.nn_default_config(engine=engine))
    try:
        if zero:   # the network's output is then 0 and the difference the target itself
            C.colapm_nn_set_params(nn, np.zeros(C.NN_PARAMS, np.float32))
        g = torch.Generator().manual_seed(5)
        psi = torch.randn((n ** 3, 3), generator=g).cuda()
        tgt = torch.from_numpy(target).cuda()
        out = torch.empty_like(psi)
        C.colapm_nn_forward(nn, psi, out, False)   # s_out = 1: the network's own output
        C.colapm_nn_sync(nn)
        d = out.cpu().numpy() - target             # rounded to FP32, as the library's difference is
        _, loss = C.colapm_nn_grads(nn, psi, tgt)
        return loss, math.fsum((d.astype(np.float64) ** 2).ravel()) / d.size
    finally:
        C.colapm_nn_destroy(nn)


@pytest.mark.parametrize("n,engine", [(16, 0), (48, 0), (128, 1)])
@pytest.mark.parametrize("case", ["ordinary", "large", "small", "mixed", "none", "inf"])
def test_loss_over_the_range_of_errors(n, engine, case):
    rng = np.random.default_rng(n)
    t = rng.standard_normal((n ** 3, 3)).astype(np.float32)
    if case == "ordinary":
        loss, want = run(n, t, False, engine)
    else:
        scale = {"large": np.float32(1e25), "small": np.float32(1e-30), "none": np.float32(0), "inf": np.float32(1)}.get(case)
        if case == "mixed":   # tiles of one size and tiles of all
            scale = (10.0 ** rng.integers(-30, 26, t.shape)).astype(np.float32)
            scale[: t.shape[0] // 2] = np.float32(1e-20)
        t = t * scale
        if case == "inf":
            t[7, 1] = np.inf
        loss, want = run(n, t, True, engine)
    if case in ("none", "inf"):
        assert loss == want
    else:
        assert math.isfinite(want) and want > 0 and abs(loss / want - 1) <= 4e-12
