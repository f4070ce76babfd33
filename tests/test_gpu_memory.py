"""Contexts in little memory: what fits without the force meshes of the blocked layout (12 B per cell) is still created, steps on
the plain layout, and gets its later arrays.

Tolerance between the layouts (the same transforms in another order of passes): positions to 1e-5 of a cell after a step
of at most a few cells, as FP32 forces of 1e-6 relative error leave them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NP, NM = 96, 384


def run(C, hold=None, free_after=0):
    """Displacements after a step, with all but `free_after` bytes beyond the context's own need held by `hold`."""
    rng = np.random.default_rng(3)
    q = np.arange(NP) * 2 * np.pi / NP
    psi = np.stack([np.sin(q + k)[:, None, None] * np.cos(q)[None, :, None] * np.cos(q + k)[None, None, :] for k in range(3)])
    psi = (2.0 * psi + 0.05 * rng.standard_normal(psi.shape)).astype(np.float32)
    block = hold(free_after) if hold else None
    ctx = C.colapm_create(C.default_params(np=NP, nm=NM, box=192.0))
    try:
        C.colapm_set_displacements(ctx, psi, np.zeros_like(psi))
        C.colapm_step(ctx, 1)
        out = np.empty((NP ** 3, 3), np.float32)
        C.colapm_get_displacement(ctx, out)
        k, p, n = C.colapm_power(ctx, 20)
        pos = np.empty((NP ** 3, 3), np.float32)
        C.colapm_get_particles_async(ctx, pos, None)
        C.colapm_wait_particles(ctx)
        return out, n
    finally:
        C.colapm_destroy(ctx)
        del block


def test_context_without_room_for_the_blocked_layout():
    import torch

    from paper_1506_03737_gb300 import colapm as C
    out0, n0 = run(C)   # also loads the kernels
    need = 148 * NP ** 3 + 20 * NM ** 3 + (64 << 20)   # the documented need, and the small tables

    def hold(free_after):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        return torch.empty(free - need - free_after, dtype=torch.uint8, device="cuda")

    room = 12 * NM ** 3
    out1, n1 = run(C, hold, room // 2)
    torch.cuda.empty_cache()
    assert np.abs(out1 - out0).max() <= 1e-5 * 192.0 / NM + 1e-6 * np.abs(out0).max()
    assert np.array_equal(n0, n1)
