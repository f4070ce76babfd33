"""Device arrays at any address: float arrays that do not start at a multiple of 4, 8 or 16 bytes give what aligned ones give,
bit for bit, in the calls that use device arrays in place and in the network's output layer (which needs multiples of 4)."""
import pytest

pytestmark = pytest.mark.gpu


def at(offset, n, values=None):
    """n floats `offset` bytes behind an aligned address, as a byte tensor."""
    import torch
    t = torch.zeros(4 * n + 64, dtype=torch.uint8, device="cuda")[offset:offset + 4 * n]
    if values is not None:
        t.copy_(values.contiguous().view(-1).view(torch.uint8))
    return t


def floats(t):
    import torch
    return t.clone().view(torch.float32)


@pytest.mark.parametrize("np_,nm", [(32, 64), (32, 32), (16, 32)])
@pytest.mark.parametrize("offset", [1, 2, 4, 8])
def test_context_arrays(np_, nm, offset):
    import torch

    from paper_1506_03737_gb300 import colapm as C
    n = 3 * np_ ** 3
    g = torch.Generator().manual_seed(1)
    psi = [torch.randn(n, generator=g).cuda() for _ in range(2)]
    ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=100.0), torch.cuda.current_stream().cuda_stream)
    try:
        got = []
        for off in (0, offset):
            C.colapm_set_displacements(ctx, *(at(off, n, p) for p in psi))
            lpt = [at(off, n) for _ in range(2)]
            C.colapm_get_lpt(ctx, *lpt)
            force = at(off, 3 * nm ** 3)
            C.colapm_get_force(ctx, force)
            got.append([floats(t) for t in (*lpt, force)])
    finally:
        C.colapm_destroy(ctx)
    assert all(float(a.abs().max()) > 0 for a in got[0])
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("n", [16, 48])
@pytest.mark.parametrize("offset", [4, 8])
def test_network_arrays(n, offset):
    import numpy as np
    import torch

    from paper_1506_03737_gb300 import colapm as C
    g = torch.Generator().manual_seed(2)
    psi, tgt = (torch.randn(3 * n ** 3, generator=g).cuda() for _ in range(2))
    nn = C.colapm_nn_create(n, C.nn_default_config(s_in=2.0, s_out=0.5), torch.cuda.current_stream().cuda_stream)
    try:
        got = []
        for po, to in ((0, 0), (offset, 0), (0, offset)):
            p, out, added, t = at(po, 3 * n ** 3, psi), at(to, 3 * n ** 3), at(po, 3 * n ** 3), at(to, 3 * n ** 3, tgt)
            C.colapm_nn_forward(nn, p, out, False)
            C.colapm_nn_forward(nn, p, added, True)
            grads, loss = C.colapm_nn_grads(nn, p, t)
            got.append((floats(out), floats(added), grads, loss))
    finally:
        C.colapm_nn_destroy(nn)
    for out, added, grads, loss in got[1:]:
        assert torch.equal(out, got[0][0]) and torch.equal(added, got[0][1])
        assert np.array_equal(grads, got[0][2])
        assert abs(loss / got[0][3] - 1) < 1e-12   # FP64 sums in the order the blocks finish
