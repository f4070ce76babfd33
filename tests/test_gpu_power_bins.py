"""P(k) of the small meshes with few bins (a warp's sums meet in one) and with many (two copies of the bins instead of sixteen, up
to the largest number), against the general plan and through the call without allocations.

Tolerances as for the boxed passes: up to 21 radix-2 levels, each adding 6e-8 of the rms to an amplitude and twice that to its
square in both results: 5.1e-6, taken as 1e-5 of the mean bin; mean |k|: sums in FP32, 4e-6. Counts are equal."""
import numpy as np
import pytest

from paper_1506_03737_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_,nm", [(32, 32), (32, 64), (96, 96), (64, 128), (32, 160)])
def test_few_and_many_bins(np_, nm):
    import torch

    from paper_1506_03737_gb300 import colapm as C
    box = 2.0 * nm
    cell, off, _ = workloads.random_state(np_, nm, 8)
    dev = [torch.from_numpy(a).cuda() for a in (cell, off)]
    ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=box))
    try:
        C.colapm_make_ics(ctx)
        C.colapm_set_state(ctx, cell, off)
        for nbins in (1, 2, 7, 63, 64, 4 * nm, 4 * nm + 1, 4096):
            got = []
            for plan in (C.PLAN_ALL, 0):
                C.colapm_set_plan(ctx, plan)
                got.append(C.colapm_power(ctx, nbins))
            if nm <= 128 and nbins <= 512:
                got.append(C.colapm_power_noalloc(*dev, np_ ** 3, nm, box, nbins, stream=torch.cuda.current_stream().cuda_stream))
            k0, p0, m0 = got.pop(1)
            on = m0 > 0
            for k, p, m in got:
                assert np.array_equal(m, m0)
                assert np.all(np.abs(k - k0)[on] <= 4e-6 * k0[on])
                assert np.all(np.abs(p - p0)[on] <= 1e-5 * p0[on].mean())
    finally:
        C.colapm_destroy(ctx)
