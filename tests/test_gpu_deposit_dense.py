"""The deposit on meshes coarser than the particle grid (neighbouring lanes merge their weights): bit-exact against
the oracle for random states (no neighbours share a cell), lattice-like ones (almost all do, wraps and ties
included) and clustered ones; and the force meshes written into device arrays in place."""
import numpy as np
import pytest

from oracle import pm as opm
from paper_1506_03737_gb300 import workloads

pytestmark = pytest.mark.gpu


def lattice_state(np_, nm, seed):
    """Sites of the particle grid moved by up to half a mesh cell."""
    rng = np.random.default_rng(seed)
    i = np.arange(np_) * (nm / np_)
    z, y, x = np.meshgrid(i, i, i, indexing="ij")
    u = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1) + rng.uniform(-0.5, 0.5, size=(np_ ** 3, 3))
    fl = np.floor(u)
    off = np.minimum((u - fl).astype(np.float32), np.nextafter(np.float32(1), np.float32(0)))
    return (fl.astype(np.int64) % nm).astype(np.int32), off


@pytest.mark.parametrize("np_,nm", [(32, 16), (64, 32), (64, 16), (192, 96)])
@pytest.mark.parametrize("kind", ["random", "lattice", "clustered"])
def test_dense_deposit_is_bit_exact(np_, nm, kind):
    from paper_1506_03737_gb300 import colapm as C
    ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=2.0 * np_))
    try:
        C.colapm_make_ics(ctx)
        if kind == "lattice":
            cell, off = lattice_state(np_, nm, 3)
        else:
            cell, off, _ = (workloads.random_state if kind == "random" else workloads.clustered_state)(np_, nm, 4)
        C.colapm_set_state(ctx, cell, off)
        rho = np.empty(nm ** 3, np.int64)
        C.colapm_get_density(ctx, rho)
    finally:
        C.colapm_destroy(ctx)
    assert np.array_equal(rho, opm.cic_deposit(cell.astype(np.float64) + off, nm).ravel())


@pytest.mark.parametrize("np_,nm", [(16, 32), (32, 64), (96, 192), (128, 256)])
def test_arrays_in_place_give_what_copies_give(np_, nm):
    """Device arrays (used in place), misaligned device arrays and host arrays: the same forces and particles."""
    import torch
    from paper_1506_03737_gb300 import colapm as C
    ctx = C.colapm_create(C.default_params(np=np_, nm=nm, box=2.0 * np_), torch.cuda.current_stream().cuda_stream)
    try:
        C.colapm_make_ics(ctx)
        C.colapm_step(ctx, 2)
        host = np.empty(3 * nm ** 3, np.float32)
        C.colapm_get_force(ctx, host)
        buf = torch.empty(3 * nm ** 3 + 1, device="cuda")
        for start in (0, 1):
            part = buf[start:start + 3 * nm ** 3]
            C.colapm_get_force(ctx, part)
            assert np.array_equal(part.cpu().numpy(), host), start
        psi = [np.empty(3 * np_ ** 3, np.float32) for _ in range(2)]
        C.colapm_get_lpt(ctx, *psi)
        n = 3 * np_ ** 3
        b2 = torch.empty(n + 1, device="cuda")
        for start in (0, 1):
            C.colapm_get_lpt(ctx, b2[start:start + n], None)
            assert np.array_equal(b2[start:start + n].cpu().numpy(), psi[0]), start
        got = []
        for fields in (psi, [torch.from_numpy(p).cuda() for p in psi], [psi[0], torch.from_numpy(psi[1]).cuda()]):
            C.colapm_set_displacements(ctx, *fields)
            C.colapm_step(ctx, 1)
            pos, mom = np.empty((np_ ** 3, 3), np.float32), np.empty((np_ ** 3, 3), np.float32)
            C.colapm_get_particles(ctx, pos, mom)
            got.append((pos, mom))
        for pos, mom in got[1:]:
            assert np.array_equal(pos, got[0][0]) and np.array_equal(mom, got[0][1])
    finally:
        C.colapm_destroy(ctx)
