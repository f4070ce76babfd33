"""P(k) and mean |k| of random clustered states against FP64 (the oracle's binning of a numpy transform). Nearly all of
P's error is bias, which does not vary between states (a pass takes 3 to 9e-8 of a line's power), so it is pinned per mesh:
the rms over the bins of two states with each mode divided by its own window and short lines with roots from one table,
plus 4%. Mean |k|: sums of at most 16 roots in FP32, each addition within 6e-8 and on average a third of that: 2.5e-8."""
import numpy as np
import pytest

from oracle import power as opower
from paper_1506_03737_gb300 import workloads

pytestmark = pytest.mark.gpu

LIMITS = {(32, 32): 0.945e-7, (64, 64): 1.952e-7, (96, 96): 1.312e-7, (64, 128): 1.545e-7, (160, 160): 1.796e-7,
          (96, 192): 1.680e-7, (64, 256): 2.219e-7, (96, 384): 2.413e-7}


def errors(C, np_, nm):
    """rms relative error over the bins of (P, mean |k|), two states."""
    box = 2.0 * np_
    kmin, kmax = 0.71 * 2 * np.pi / box, 0.97 * np.pi * nm / box   # no edge on a mode
    dp, dk = [], []
    for seed in (11, 12):
        cell, off, _ = workloads.clustered_state(np_, nm, seed)
        ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=box))
        try:
            zero = np.zeros((3, np_, np_, np_), np.float32)
            C.colapm_set_displacements(ctx, zero, zero)
            C.colapm_set_state(ctx, cell, off)
            k, p, cnt = C.colapm_power(ctx, 60, kmin, kmax)
        finally:
            C.colapm_destroy(ctx)
        kr, pr, nr = opower.power_from_positions((cell + off.astype(np.float64)) * (box / nm), box, np_, nm, 60, kmin, kmax,
                                                  fft="numpy")
        assert np.array_equal(cnt, nr)
        ok = nr > 0
        dp.append(p[ok] / pr[ok] - 1)
        dk.append(k[ok] / kr[ok] - 1)
    return tuple(float(np.sqrt(np.mean(np.concatenate(d) ** 2))) for d in (dp, dk))


@pytest.mark.parametrize("np_,nm", list(LIMITS))
def test_power_error_against_fp64(np_, nm):
    from paper_1506_03737_gb300 import colapm as C
    p, k = errors(C, np_, nm)
    assert p <= LIMITS[np_, nm] and k <= 2.5e-8
