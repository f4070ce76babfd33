"""The force meshes whose z and y passes move their tiles by boxes (z from 256 points on, y from 512), for every window power,
against the general plan on a clustered state.

Tolerance: forward and inverse transforms have up to 60 radix-2 levels together, each adding at most 2^-24 of the rms of
what it transforms, in both results: 60 x 2 x 6e-8 = 7.2e-6 of the rms force."""
import pytest

from paper_1506_03737_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nm,deconvs", [(256, (0, 1, 2)), (320, (0, 2)), (384, (0, 1, 2)), (512, (0, 1, 2)), (1024, (0, 2))])
def test_boxed_force_agrees_with_the_general_plan(nm, deconvs):
    import torch

    from paper_1506_03737_gb300 import colapm as C
    np_ = 64
    cell, off, _ = workloads.clustered_state(np_, nm, 21)
    zero = torch.zeros((3, np_, np_, np_), device="cuda")
    out = [torch.empty((3, nm, nm, nm), device="cuda") for _ in range(2)]
    for deconv in deconvs:
        ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=2.0 * nm, deconv=deconv),
                              torch.cuda.current_stream().cuda_stream)
        try:
            C.colapm_set_displacements(ctx, zero, zero)
            C.colapm_set_state(ctx, cell, off)
            for plan, o in ((C.PLAN_ALL, out[0]), (0, out[1])):
                C.colapm_set_plan(ctx, plan)
                C.colapm_get_force(ctx, o)
        finally:
            C.colapm_destroy(ctx)
        d2 = r2 = 0.0
        for j in range(3):   # one component at a time: the differences of all three would not be small at 1024^3
            d2 += float((out[0][j] - out[1][j]).pow_(2).sum(dtype=torch.float64))
            r2 += float(out[1][j].pow(2).sum(dtype=torch.float64))
        assert r2 > 0 and (d2 / r2) ** 0.5 < 7.2e-6
