"""P(k) of the meshes whose z pass moves its tiles by boxes (256, 384, 512) and of the ones between them, against the
general plan: few and many bins, a range that leaves modes out on both sides.

Tolerances, for a state without clustering (modes of about the same size): each of the 27 radix-2 levels at most adds
6e-8 of the rms to an amplitude, twice that to its square (3.2e-6, both results 6.4e-6): 1e-5. Mean |k|: sums of at
most 32 terms in FP32, 6e-8 each: 4e-6. Counts are equal."""
import numpy as np
import pytest

from paper_1506_03737_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nm", [256, 320, 384, 512])
def test_boxed_power_agrees_with_the_general_plan(nm):
    from paper_1506_03737_gb300 import colapm as C
    np_ = 64
    ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=2.0 * nm))
    try:
        C.colapm_make_ics(ctx)
        cell, off, _ = workloads.random_state(np_, nm, 6)
        C.colapm_set_state(ctx, cell, off)
        kf = 2 * np.pi / (2.0 * nm)
        for args in ((1,), (7, 5.5 * kf, 0.3 * nm * kf), (100,), (4096,)):
            got = {}
            for plan in (C.PLAN_ALL, 0):
                C.colapm_set_plan(ctx, plan)
                got[plan] = C.colapm_power(ctx, *args)
            (k, p, m), (k0, p0, m0) = got[C.PLAN_ALL], got[0]
            assert np.array_equal(m, m0)
            on = m > 0
            assert np.all(np.abs(k - k0)[on] <= 4e-6 * k0[on])
            assert np.all(np.abs(p - p0)[on] <= 1e-5 * p0[on].mean())
    finally:
        C.colapm_destroy(ctx)
