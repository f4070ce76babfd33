"""The work that a user of the library has it do, as cases that can be timed and compared.

Kinds of a case (``kind``), each one pass through the public calls of ``colapm.py``:

  spectrum   colapm_power_noalloc of device positions (called inside another framework's loop)
  step       a known displacement field placed as particles, COLA / PM steps, displacement and momenta read back
  force      the three force meshes of an evolved particle state
  power      P(k) of an evolved particle state, or its cross-correlation with a second one
  ics        2LPT initial conditions of a new seed and their displacement fields
  mock       a whole mock: initial conditions of a new seed, all steps, P(k) (in redshift space after finalize, if asked)
  batch      many mocks of uneven sizes replayed with new seeds
  nn_forward the learned correction applied to a displacement field
  nn_grads   loss and gradients of one pair
  nn_train   one Adam step on one pair, and the updated parameters

The transforms behind a P(k) run in single precision, so its values are kept in single precision here; mode counts
stay whole numbers. ``exact`` restates each single-layer case in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_1506_03737_gb300 import colapm as C

COSMO = dict(omega_m=0.3, omega_b=0.05, h=0.7, n_s=0.96, sigma8=0.8)
MESHES = (16, 32, 64, 96, 128, 160, 192, 256, 320, 384, 512, 1024)
NN_SHAPES = ((3, 16), (16, 16), (16, 16), (16, 3))


def listed():
    return [
        # latency: a spectrum of a few particles between two steps of somebody else's code
        dict(name="spectrum_64m", kind="spectrum", n=32 ** 3, nm=64, box=256.0, nbins=32),
        # latency: one step of the smallest named workload
        dict(name="step_32p_64m", kind="step", np=32, nm=64, box=256.0, steps=1, cola=True, deconv=1, stepping=0),
        # a whole mock of the smallest size of a batch, run on its own
        dict(name="mock_64p_128m", kind="mock", np=64, nm=128, box=128.0, steps=10, cola=True, stepping=0, spacing=0,
             rsd=False, nbins=100),
        # the coarse, few-step run that the learned correction starts from (mesh as fine as the particle grid)
        dict(name="mock_128p_128m", kind="mock", np=128, nm=128, box=256.0, steps=5, cola=True, stepping=0, spacing=0,
             rsd=False, nbins=24),
        # the force of a clustered state on a mixed-radix mesh (the largest size of a batch)
        dict(name="force_192p_384m", kind="force", np=192, nm=384, box=512.0, deconv=1),
        # one step of the middle named workload
        dict(name="step_256p_512m", kind="step", np=256, nm=512, box=512.0, steps=1, cola=True, deconv=1, stepping=0),
        # the measurement at the end of the middle workload
        dict(name="power_256p_512m", kind="power", np=256, nm=512, box=512.0, nbins=100, cross=False),
        # initial conditions of the middle workload
        dict(name="ics_256p", kind="ics", np=256, nm=256, box=512.0),
        # the largest named workload: one mock, initial conditions to P(k)
        dict(name="mock_512p_1024m", kind="mock", np=512, nm=1024, box=1024.0, steps=10, cola=True, stepping=0,
             spacing=0, rsd=False, nbins=100),
        # uneven mocks (64^3 to 192^3 particles, two of each size) in one graph
        dict(name="batch_10", kind="batch", mocks=10, smallest=64, sizes=5, steps=10, nbins=100),
        # the learned correction of the 128^3 workload: inference and training
        dict(name="nn_forward_128", kind="nn_forward", n=128, add=True),
        dict(name="nn_train_128", kind="nn_train", n=128),
    ]


def draw(rng):
    kind = rng.choice(("spectrum", "step", "force", "power", "ics", "mock", "mock", "batch", "nn_forward", "nn_grads",
                       "nn_train"))
    if kind == "spectrum":
        nm = rng.choice((16, 32, 64, 96, 128))
        return dict(kind=kind, n=int(math.exp(rng.uniform(math.log(1000), math.log(4e6)))), nm=nm,
                    box=round(rng.uniform(64, 1024), 1), nbins=rng.randint(8, 200))
    if kind in ("nn_forward", "nn_grads", "nn_train"):
        n = 16 * int(round(math.exp(rng.uniform(0, math.log(12)))))
        return dict(kind=kind, n=n, add=rng.random() < 0.5) if kind == "nn_forward" else dict(
            kind=kind, n=n, scale=round(rng.uniform(0.5, 2.0), 3))
    if kind == "ics":
        np_ = rng.choice(MESHES[1:-1])
        return dict(kind=kind, np=np_, nm=np_, box=round(np_ * rng.uniform(1.0, 4.0), 1))
    if kind == "batch":
        return dict(kind=kind, mocks=rng.randint(2, 12), smallest=rng.choice((32, 64, 96)), sizes=rng.randint(1, 4),
                    steps=rng.randint(3, 12), nbins=rng.randint(16, 128))
    # particles of 32^3 to 256^3 on meshes of half to four times as many cells per side, up to 512
    pairs = [(p, m) for p in MESHES[1:8] for m in (p // 2, p, 2 * p, 4 * p) if m in MESHES and 32 <= m <= 512]
    np_, nm = rng.choice(pairs)
    box = round(np_ * rng.uniform(1.0, 4.0), 1)
    if kind == "step":
        return dict(kind=kind, np=np_, nm=nm, box=box, steps=rng.randint(1, 3), cola=rng.random() < 0.75,
                    deconv=rng.randint(0, 2), stepping=rng.randint(0, 1))
    if kind == "force":
        return dict(kind=kind, np=np_, nm=nm, box=box, deconv=rng.randint(0, 2))
    if kind == "power":
        return dict(kind=kind, np=np_, nm=nm, box=box, nbins=rng.randint(8, 200), cross=rng.random() < 0.25)
    return dict(kind=kind, np=np_, nm=nm, box=box, steps=rng.randint(2, 20), cola=rng.random() < 0.75,
                stepping=rng.randint(0, 1), spacing=rng.randint(0, 1), rsd=rng.random() < 0.25,
                nbins=rng.randint(8, 200))


# --- inputs -----------------------------------------------------------------------------------

class Owned:
    """A library handle that is given back with the object."""

    def __init__(self, handle, destroy):
        self.h, self._destroy = handle, destroy

    def __del__(self):
        if self.h:
            self._destroy(self.h)
            self.h = None


def _context(**kw):
    return Owned(C.colapm_create(C.default_params(**COSMO, **kw), torch.cuda.current_stream().cuda_stream),
                 C.colapm_destroy)


def _generator(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed % (1 << 40)) + tag)
    return g


def _displacement(n, rms, seed, tag, slope=1.5):
    """Three smooth periodic fields [3][z][y][x] of the given rms: white noise filtered as 1 / k^slope."""
    g = _generator(seed, tag)
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda")
    kx = torch.fft.rfftfreq(n, 1.0 / n, device="cuda")
    k2 = k.view(-1, 1, 1) ** 2 + k.view(1, -1, 1) ** 2 + kx.view(1, 1, -1) ** 2
    filt = (k2 + 4.0) ** (-0.5 * slope) * torch.exp(-k2 / (0.35 * n) ** 2)
    filt[0, 0, 0] = 0.0
    out = torch.empty((3, n, n, n), device="cuda")
    for j in range(3):
        f = torch.fft.irfftn(torch.fft.rfftn(torch.randn((n, n, n), device="cuda", generator=g)) * filt, s=(n, n, n))
        out[j] = f * (rms / f.std())
    return out


def _evolved_state(case, seed, tag):
    """Cells and offsets of an evolved state in id order: a displaced lattice, a fifth of it fallen into clumps."""
    np_, nm = case["np"], case["nm"]
    g = _generator(seed, tag)
    cell = case["box"] / nm
    q = (torch.arange(np_, device="cuda", dtype=torch.float64) * (nm / np_) + 0.5)
    d = _displacement(np_, 5.0 / cell, seed, tag + 1)
    u = torch.stack([(q.view(1, 1, -1) + d[0]).reshape(-1), (q.view(1, -1, 1) + d[1]).reshape(-1),
                     (q.view(-1, 1, 1) + d[2]).reshape(-1)], dim=1)
    del d
    n = np_ ** 3
    centres = torch.rand((max(8, n // 400), 3), device="cuda", generator=g, dtype=torch.float64) * nm
    k = n // 5
    pick = torch.randint(0, centres.shape[0], (k,), device="cuda", generator=g)
    where = torch.randperm(n, device="cuda", generator=g)[:k]
    u[where] = centres[pick] + torch.randn((k, 3), device="cuda", generator=g, dtype=torch.float64) * (0.5 / cell)
    fl = torch.floor(u)
    off = (u - fl).float().clamp_(0.0, 1.0 - 2.0 ** -24)
    return torch.remainder(fl, nm).to(torch.int32).contiguous(), off.contiguous()


def _positions(case, seed):
    """Cells and offsets of any number of particles, half of them in clumps."""
    n, nm = case["n"], case["nm"]
    g = _generator(seed, 3)
    u = torch.rand((n, 3), device="cuda", generator=g, dtype=torch.float64) * nm
    centres = torch.rand((max(4, n // 400), 3), device="cuda", generator=g, dtype=torch.float64) * nm
    pick = torch.randint(0, centres.shape[0], (n // 2,), device="cuda", generator=g)
    u[:n // 2] = centres[pick] + torch.randn((n // 2, 3), device="cuda", generator=g, dtype=torch.float64)
    fl = torch.floor(u)
    off = (u - fl).float().clamp_(0.0, 1.0 - 2.0 ** -24)
    return torch.remainder(fl, nm).to(torch.int32).contiguous(), off.contiguous()


def _nn_inputs(case, seed):
    """A displacement field [n^3][3], a target and trained-like parameters (He-normal weights, small biases)."""
    n = case["n"]
    psi = _displacement(n, 5.0 * case.get("scale", 1.0), seed, 20).reshape(3, -1).t().contiguous()
    tgt = _displacement(n, 0.5, seed, 30, slope=0.5).reshape(3, -1).t().contiguous()
    rng = np.random.default_rng(seed % (1 << 32))
    flat = []
    for i, o in NN_SHAPES:
        flat += [rng.standard_normal(27 * o * i) * math.sqrt(2.0 / (27 * i)), rng.standard_normal(o) * 0.05]
    return psi, tgt, np.concatenate(flat).astype(np.float32)


def _step_fields(case, seed):
    n = case["np"]
    return _displacement(n, 5.0, seed, 40), _displacement(n, 1.5, seed, 50)


def _run_kw(case):
    return dict(np=case["np"], nm=case["nm"], box=case["box"])


def _mock_seed(seed, k):
    return (seed * 7919 + k) % (1 << 62)


def _batch_params(case):
    ps = []
    for r in range(case["mocks"]):
        k = r % case["sizes"]
        np_ = case["smallest"] + 32 * k
        ps.append(C.default_params(**COSMO, np=np_, nm=2 * np_, box=2.0 * np_ + 32.0 * k, n_steps=case["steps"]))
    return ps


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "spectrum":
        s["cell"], s["off"] = _positions(case, seed)
    elif kind == "step":
        s["ctx"] = _context(**_run_kw(case), cola=int(case["cola"]), deconv=case["deconv"], stepping=case["stepping"])
        s["psi1"], s["psi2"] = _step_fields(case, seed)
        n = case["np"] ** 3
        s["out"] = [torch.empty((n, 3), device="cuda") for _ in range(2)]
    elif kind in ("force", "power"):
        names = ("ctx", "ctx2") if case.get("cross") else ("ctx",)
        for i, name in enumerate(names):
            s[name] = _context(**_run_kw(case), deconv=case.get("deconv", 1))
            cell, off = _evolved_state(case, seed, 60 + 10 * i)
            zero = torch.zeros((3, case["np"], case["np"], case["np"]), device="cuda")
            C.colapm_set_displacements(s[name].h, zero, zero)
            C.colapm_set_state(s[name].h, cell, off)
        if kind == "force":
            s["out"] = torch.empty((3,) + (case["nm"],) * 3, device="cuda")
    elif kind == "ics":
        s["ctx"] = _context(**_run_kw(case))
        s["out"] = [torch.empty((3,) + (case["np"],) * 3, device="cuda") for _ in range(2)]
    elif kind == "mock":
        s["ctx"] = _context(**_run_kw(case), n_steps=case["steps"], cola=int(case["cola"]), stepping=case["stepping"],
                            spacing=case["spacing"])
    elif kind == "batch":
        b = C.colapm_batch_create(_batch_params(case), 0, torch.cuda.current_stream().cuda_stream)
        s["batch"] = Owned(b, C.colapm_batch_destroy)
        # the first run tunes and captures; a user's program replays the batch many times after it
        C.colapm_batch_run(b, case["mocks"], case["nbins"], seeds=[1 + i for i in range(case["mocks"])])
    else:
        s["psi"], s["target"], params = _nn_inputs(case, seed)
        s["nn"] = Owned(C.colapm_nn_create(case["n"], C.nn_default_config(s_in=4.0, s_out=0.5),
                                           torch.cuda.current_stream().cuda_stream), C.colapm_nn_destroy)
        C.colapm_nn_set_params(s["nn"].h, params)
        s["out"] = torch.empty_like(s["psi"])
    torch.cuda.synchronize()
    return s


# --- one pass ---------------------------------------------------------------------------------

def _spectrum(kpn):
    k, p, n = kpn
    return dict(k=k.astype(np.float32), p=p.astype(np.float32), modes=n)


def run(s):
    case, kind, seed = s["case"], s["case"]["kind"], s["seed"]
    if kind == "spectrum":
        return _spectrum(C.colapm_power_noalloc(s["cell"], s["off"], case["n"], case["nm"], case["box"], case["nbins"],
                                                stream=torch.cuda.current_stream().cuda_stream))
    if kind == "step":
        ctx = s["ctx"].h
        C.colapm_set_displacements(ctx, s["psi1"], s["psi2"])
        C.colapm_step(ctx, case["steps"])
        C.colapm_get_displacement(ctx, s["out"][0])
        C.colapm_get_particles(ctx, None, s["out"][1])
        return dict(displacement=s["out"][0], momentum=s["out"][1])
    if kind == "force":
        return C.colapm_get_force(s["ctx"].h, s["out"])
    if kind == "power":
        if case["cross"]:
            return _spectrum(C.colapm_cross_correlation(s["ctx"].h, s["ctx2"].h, case["nbins"]))
        return _spectrum(C.colapm_power(s["ctx"].h, case["nbins"]))
    if kind == "ics":
        ctx = s["ctx"].h
        C.colapm_reseed(ctx, _mock_seed(seed, 0))
        C.colapm_make_ics(ctx)
        C.colapm_get_lpt(ctx, *s["out"])
        return dict(psi1=s["out"][0], psi2=s["out"][1])
    if kind == "mock":
        ctx = s["ctx"].h
        C.colapm_reseed(ctx, _mock_seed(seed, 0))
        C.colapm_make_ics(ctx)
        C.colapm_step(ctx, -1)
        if case["rsd"]:
            C.colapm_finalize(ctx)
            return _spectrum(C.colapm_power_rsd(ctx, -1, case["nbins"]))
        return _spectrum(C.colapm_power(ctx, case["nbins"]))
    if kind == "batch":
        n = case["mocks"]
        return _spectrum(C.colapm_batch_run(s["batch"].h, n, case["nbins"],
                                            seeds=[_mock_seed(seed, i) for i in range(n)]))
    nn = s["nn"].h
    if kind == "nn_forward":
        return C.colapm_nn_forward(nn, s["psi"], s["out"], case["add"])
    if kind == "nn_grads":
        g, loss = C.colapm_nn_grads(nn, s["psi"], s["target"])
        return dict(grads=g, loss=np.float32(loss))
    C.colapm_nn_train_step(nn, s["psi"], s["target"], want_loss=False)
    return C.colapm_nn_get_params(nn)


# --- what a pass cannot do without ------------------------------------------------------------

def _fft_flops(n, transforms):
    return transforms * 2.5 * n ** 3 * math.log2(n ** 3)


def _force_work(np_, nm):
    """Deposit, four transforms and three force meshes: 16 B of a position; per cell the int64 density written and
    read (16 B), the half spectrum written and read twice (an out-of-core 3-D transform passes twice over its data,
    24 B) and the three force meshes written (12 B). """
    return 16 * np_ ** 3 + 52 * nm ** 3, _fft_flops(nm, 4) + 50 * np_ ** 3 + 20 * nm ** 3


def _step_work(np_, nm):
    """One step: 96 B per particle (position, momentum and both displacements read, position and momentum written,
    the position read once more by the deposit) and 80 B per cell."""
    return 96 * np_ ** 3 + 80 * nm ** 3, _fft_flops(nm, 4) + 200 * np_ ** 3 + 20 * nm ** 3


def _power_work(np_, nm):
    return 16 * np_ ** 3 + 28 * nm ** 3, _fft_flops(nm, 1) + 50 * np_ ** 3 + 10 * nm ** 3


def _ics_work(np_):
    """One spectrum out, nine fields transformed to real space, the source back, three more fields: 13 transforms,
    each field written and read once per pass of two."""
    return 8 * 14 * np_ ** 3 + 40 * np_ ** 3, _fft_flops(np_, 13) + 150 * np_ ** 3


def work(case):
    kind = case["kind"]
    if kind == "spectrum":
        b, f = 24 * case["n"] + 28 * case["nm"] ** 3, _fft_flops(case["nm"], 1) + 50 * case["n"] + 10 * case["nm"] ** 3
    elif kind == "step":
        np_, nm = case["np"], case["nm"]
        b, f = _step_work(np_, nm)
        b, f = case["steps"] * b + (24 + 40 + 24) * np_ ** 3, case["steps"] * f
    elif kind == "force":
        b, f = _force_work(case["np"], case["nm"])
    elif kind == "power":
        b, f = _power_work(case["np"], case["nm"])
        if case["cross"]:
            b, f = 2 * b, 2 * f
    elif kind == "ics":
        b, f = _ics_work(case["np"])
        b += 48 * case["np"] ** 3
    elif kind in ("mock", "batch"):
        b = f = 0
        if kind == "mock":
            sizes = [(case["np"], case["nm"], case["steps"] + int(case["rsd"]))]
        else:
            sizes = [(p.np, p.nm, p.n_steps) for p in _batch_params(case)]
        for np_, nm, steps in sizes:
            for k, (x, y) in ((1, _ics_work(np_)), (steps, _step_work(np_, nm)), (1, _power_work(np_, nm))):
                b, f = b + k * x, f + k * y
    else:
        n3 = case["n"] ** 3
        mults = 27 * sum(i * o for i, o in NN_SHAPES)
        if kind == "nn_forward":
            b, f = 24 * n3, 2 * mults * n3
        else:   # forward, gradients of the activations (all layers but the first) and of the weights
            back = 27 * sum(i * o for i, o in NN_SHAPES[1:])
            # the three hidden activations written and read once in 16 bits
            b, f = 24 * n3 + 3 * 2 * 32 * n3, 2 * (2 * mults + back) * n3
    return {"bytes": float(b), "flops": float(f)}


# --- the same in 64 bits ----------------------------------------------------------------------

def _cic(u, nm):
    """Base cell and weights per axis of mesh coordinates u [P, 3] (fractions in steps of 2^-15, the path's definition)."""
    c = torch.floor(u)
    f = torch.round((u - c) * 32768.0) / 32768.0
    return torch.remainder(c, nm).long(), f


def _corners(c, f, nm):
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                i = (((c[:, 2] + dz) % nm) * nm + (c[:, 1] + dy) % nm) * nm + (c[:, 0] + dx) % nm
                w = (f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (f[:, 2] if dz else 1 - f[:, 2])
                yield i, w


def _delta(u, nm):
    rho = torch.zeros(nm ** 3, dtype=torch.float64, device="cuda")
    c, f = _cic(u, nm)
    for i, w in _corners(c, f, nm):
        rho.index_add_(0, i, w)
    return (rho * (nm ** 3 / u.shape[0]) - 1.0).view(nm, nm, nm)


def _axes(n):
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    kx = torch.fft.rfftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    return k.view(-1, 1, 1), k.view(1, -1, 1), kx.view(1, 1, -1)


def _window(n):
    out = 1.0
    for k in _axes(n):
        out = out * torch.sinc(k / n) ** 2
    return out


def _inverse_k2(n):
    """1 / k^2 on the half grid in units of the grid spacing; 0 at k = 0 and on the Nyquist planes."""
    kz, ky, kx = _axes(n)
    n2 = kz ** 2 + ky ** 2 + kx ** 2
    ok = (n2 > 0) & (kz.abs() != n // 2) & (ky.abs() != n // 2) & (kx.abs() != n // 2)
    return torch.where(ok, (n / (2 * math.pi)) ** 2 / n2.clamp(min=1.0), torch.zeros_like(n2))


def _force(u, nm, deconv):
    g = torch.fft.rfftn(_delta(u, nm)) * _inverse_k2(nm)
    if deconv:
        g = g / _window(nm) ** deconv
    w = 2 * math.pi / nm
    return torch.stack([torch.fft.irfftn(g * (1j * w * k), s=(nm,) * 3) for k in reversed(_axes(nm))])


def _state_u(cell, off):
    return cell.double() + off.double()


def _bins(nm, box, nbins):
    kz, ky, kx = _axes(nm)
    kf = 2 * math.pi / box
    k = kf * torch.sqrt(kz ** 2 + ky ** 2 + kx ** 2)
    kmin, kmax = kf, math.pi * nm / box
    edges = torch.tensor([kmin * (kmax / kmin) ** (b / nbins) for b in range(nbins + 1)], dtype=torch.float64,
                         device="cuda")
    b = torch.bucketize(k, edges, right=True) - 1
    ok = (b >= 0) & (b < nbins) & (kz.abs() != nm // 2) & (ky.abs() != nm // 2) & (kx != nm // 2)
    mult = torch.where(kx == 0, 1.0, 2.0).expand_as(k)   # both halves of the grid
    return k, torch.where(ok, b, torch.full_like(b, nbins)).reshape(-1), mult


def _binned(v, b, mult, nbins):
    out = torch.zeros(nbins + 1, dtype=torch.float64, device="cuda")
    out.index_add_(0, b, (v * mult).reshape(-1))
    return out[:nbins]


def _power(u, nm, box, nbins, u2=None):
    k, b, mult = _bins(nm, box, nbins)
    cnt = _binned(torch.ones_like(k), b, mult, nbins)
    d = torch.fft.rfftn(_delta(u, nm))
    if u2 is None:
        p = _binned(d.abs() ** 2 / _window(nm) ** 2, b, mult, nbins) * (box ** 3 / nm ** 6) / cnt
    else:
        e = torch.fft.rfftn(_delta(u2, nm))
        p = _binned((d * e.conj()).real, b, mult, nbins) / torch.sqrt(
            _binned(d.abs() ** 2, b, mult, nbins) * _binned(e.abs() ** 2, b, mult, nbins))
    return dict(k=(_binned(k, b, mult, nbins) / cnt).cpu().numpy(), p=p.cpu().numpy(), modes=None)


def _growth(om, a_list):
    """(D1, D2, P1, P2) at each a: the first- and second-order growth equations in ln a by classical RK4."""
    def rhs(lna, y):
        a = math.exp(lna)
        e = math.sqrt(om / a ** 3 + 1 - om)
        return np.array([y[1] / (a * a * e), 1.5 * om * y[0] / (a * e), y[3] / (a * a * e),
                         1.5 * om * (y[2] - y[0] ** 2) / (a * e)])

    def to(a, steps=3000):
        a0 = 1e-5
        e0 = math.sqrt(om / a0 ** 3 + 1 - om)
        y, l0 = np.array([a0, a0 ** 3 * e0, -3 / 7 * a0 ** 2, -6 / 7 * a0 ** 4 * e0]), math.log(a0)
        h = (math.log(a) - l0) / steps
        for i in range(steps):
            x = l0 + i * h
            k1 = rhs(x, y)
            k2 = rhs(x + h / 2, y + h / 2 * k1)
            k3 = rhs(x + h / 2, y + h / 2 * k2)
            k4 = rhs(x + h, y + h * k3)
            y = y + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        return y

    n = to(1.0)[0]
    return [(lambda y: (y[0] / n, y[2] / n ** 2, y[1] / n, y[3] / n ** 2))(to(a)) for a in a_list]


def _integral(f, lo, hi):
    x, w = np.polynomial.legendre.leggauss(64)
    return float(np.sum(w * f(0.5 * (hi - lo) * x + 0.5 * (hi + lo))) * 0.5 * (hi - lo))


def _exact_step(case, seed):
    np_, nm, box, om = case["np"], case["nm"], case["box"], COSMO["omega_m"]
    cell = box / nm
    e = lambda a: np.sqrt(om / a ** 3 + 1 - om)  # noqa: E731
    a = [0.1 + 0.9 * i / 10 for i in range(11)]
    g = _growth(om, a[:case["steps"] + 1])
    psi1, psi2 = ([f.reshape(3, -1).t().double() / cell for f in _step_fields(case, seed)])
    q = torch.arange(np_, device="cuda", dtype=torch.float64) * (nm / np_) + 0.5
    ones = torch.ones((np_,) * 3, dtype=torch.float64, device="cuda")
    q = torch.stack([(q.view(1, 1, -1) * ones).reshape(-1), (q.view(1, -1, 1) * ones).reshape(-1),
                     (q.view(-1, 1, 1) * ones).reshape(-1)], dim=1)
    d = g[0][0] * psi1 + g[0][1] * psi2
    p = torch.zeros_like(d) if case["cola"] else g[0][2] * psi1 + g[0][3] * psi2
    n = -2.5
    for i in range(case["steps"]):
        u = torch.remainder(q + d, nm)
        f = _force(u, nm, case["deconv"]).reshape(3, -1)
        c, w = _cic(u, nm)
        acc = torch.zeros_like(d)
        for idx, wt in _corners(c, w, nm):
            for j in range(3):
                acc[:, j] += wt * f[j][idx]
        if case["cola"]:
            acc -= g[i][0] * psi1 + (g[i][1] - g[i][0] ** 2) * psi2
        lo, hi = (a[0] if i == 0 else 0.5 * (a[i - 1] + a[i])), 0.5 * (a[i] + a[i + 1])
        if case["stepping"]:
            kick = 1.5 * om * _integral(lambda x: 1 / (x * x * e(x)), lo, hi)
            drift = _integral(lambda x: 1 / (x ** 3 * e(x)), a[i], a[i + 1])
        else:
            kick = 1.5 * om * (hi ** n - lo ** n) / (n * a[i] ** (n - 1)) / (a[i] ** 2 * e(a[i]))
            drift = hi ** -n * _integral(lambda x: x ** (n - 3) / e(x), a[i], a[i + 1])
        p = p + kick * acc
        d = d + drift * p
        if case["cola"]:
            d = d + (g[i + 1][0] - g[i][0]) * psi1 + (g[i + 1][1] - g[i][1]) * psi2
    return dict(displacement=torch.remainder(d + nm / 2, nm).sub_(nm / 2) * cell, momentum=p * cell)


def _philox(m, seed):
    """The first two words of Philox4x32-10 (Salmon et al. 2011) for counters m and a 64-bit key."""
    mask, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    c = [m & mask, m >> sh, np.zeros_like(m), np.zeros_like(m)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        x, y = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(y >> sh) ^ c[1] ^ np.uint64(k0), y & mask, (x >> sh) ^ c[3] ^ np.uint64(k1), x & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[0], c[1]


def _linear_pk(k):
    """BBKS spectrum of the cosmology above, normalised to sigma_8 with an 8 Mpc/h top-hat."""
    def shape(k):
        x = k / (COSMO["omega_m"] * COSMO["h"])
        t = np.log1p(2.34 * x) / (2.34 * x) * (1 + 3.89 * x + (16.1 * x) ** 2 + (5.46 * x) ** 3 + (6.71 * x) ** 4) ** -0.25
        return k ** COSMO["n_s"] * t * t
    lk = np.linspace(math.log(1e-5), math.log(1e2), 65537)
    kk = np.exp(lk)
    x = 8 * kk
    w = np.where(x < 1e-3, 1 - x * x / 10, 3 * (np.sin(x) - x * np.cos(x)) / x ** 3)
    f = kk ** 3 * shape(kk) * w * w / (2 * math.pi ** 2)
    simpson = (lk[1] - lk[0]) / 3 * (f[0] + f[-1] + 4 * f[1:-1:2].sum() + 2 * f[2:-1:2].sum())
    return COSMO["sigma8"] ** 2 / simpson * shape(k)


def _exact_ics(case, seed):
    n, box = case["np"], case["box"]
    h = n // 2
    i = np.arange(n, dtype=np.uint64)
    m = (i.reshape(-1, 1, 1) * np.uint64(n) + i.reshape(1, -1, 1)) * np.uint64(n) + i[:h].reshape(1, 1, -1)
    r0, r1 = _philox(m, _mock_seed(seed, 0))
    u1, u2 = (torch.from_numpy((2.0 * (r >> np.uint64(9)).astype(np.float64) + 1.0) * 2.0 ** -24).cuda() for r in (r0, r1))
    s = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64).round().long()
    n2 = (s.view(-1, 1, 1) ** 2 + s.view(1, -1, 1) ** 2 + s[:h].view(1, 1, -1) ** 2)
    amp = np.zeros(3 * h * h + 1)
    amp[1:] = n ** 3 * np.sqrt(_linear_pk(2 * math.pi / box * np.sqrt(np.arange(1, amp.size))) / box ** 3)
    dk = torch.from_numpy(amp).cuda()[n2] * torch.sqrt(-torch.log(u1)) * torch.exp(2j * math.pi * u2)
    plane = dk[:, :, 0].clone()   # on k_x = 0 the larger index of each conjugate pair mirrors its partner
    j = torch.arange(n, device="cuda")
    part = (n - j) % n
    mine, other = j.view(-1, 1) * n + j.view(1, -1), part.view(-1, 1) * n + part.view(1, -1)
    mirrored = plane[part][:, part].conj()
    dk[:, :, 0] = torch.where(mine > other, mirrored, plane)
    full = torch.zeros((n, n, h + 1), dtype=torch.complex128, device="cuda")
    full[:, :, :h] = dk
    g, w = _inverse_k2(n), 2 * math.pi / n
    k = [w * x for x in reversed(_axes(n))]
    inv = lambda x: torch.fft.irfftn(x, s=(n,) * 3)  # noqa: E731
    a = full * g
    psi1 = torch.stack([inv(1j * k[c] * a) for c in range(3)])
    phi = {(c, d): inv(k[c] * k[d] * a) for c in range(3) for d in range(c, 3)}
    src = (phi[0, 0] * phi[1, 1] + phi[0, 0] * phi[2, 2] + phi[1, 1] * phi[2, 2] - phi[0, 1] ** 2 - phi[0, 2] ** 2
           - phi[1, 2] ** 2)
    b = torch.fft.rfftn(src) * g
    psi2 = torch.stack([inv(-1j * k[c] * b) for c in range(3)])
    return dict(psi1=psi1 * (box / n), psi2=psi2 * (box / n))


def _nn_params(flat):
    out, at = [], 0
    for i, o in NN_SHAPES:
        w = torch.from_numpy(flat[at:at + 27 * o * i].astype(np.float64)).cuda().view(27, o, i)
        at += 27 * o * i
        out.append((w, torch.from_numpy(flat[at:at + o].astype(np.float64)).cuda()))
        at += o
    return out


_TAPS = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _roll(v, d, sign):
    return torch.roll(v, tuple(-sign * x for x in d), (0, 1, 2))


def _exact_nn(case, seed):
    n = case["n"]
    psi, tgt, flat = _nn_inputs(case, seed)
    params = _nn_params(flat)
    acts = [psi.double().view(n, n, n, 3) / 4.0]
    for l, (w, b) in enumerate(params):
        z = b + sum(_roll(acts[-1], d, 1) @ w[t].t() for t, d in enumerate(_TAPS))
        acts.append(torch.relu(z) if l < 3 else z)
    if case["kind"] == "nn_forward":
        out = 0.5 * acts[-1].reshape(-1, 3)
        return out + psi.double() if case["add"] else out
    diff = acts[-1] - tgt.double().view(n, n, n, 3) / 0.5
    dz, grads = 2.0 * diff / diff.numel(), []
    for l in range(3, -1, -1):
        w, _ = params[l]
        f = dz.reshape(-1, dz.shape[-1])
        dw = torch.stack([f.t() @ _roll(acts[l], d, 1).reshape(-1, w.shape[2]) for d in _TAPS])
        grads = [dw.reshape(-1), f.sum(0)] + grads
        if l:
            dz = sum(_roll(dz, d, -1) @ w[t] for t, d in enumerate(_TAPS)) * (acts[l] > 0)
    grads = torch.cat(grads).cpu().numpy()
    if case["kind"] == "nn_grads":
        return dict(grads=grads, loss=float((diff ** 2).mean()))
    return flat.astype(np.float64) - 1e-3 * grads / (np.abs(grads) + 1e-8)   # the first Adam step


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return _power(_state_u(*_positions(case, seed)), case["nm"], case["box"], case["nbins"])
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "force":
        return _force(_state_u(*_evolved_state(case, seed, 60)), case["nm"], case["deconv"])
    if kind == "power":
        u = _state_u(*_evolved_state(case, seed, 60))
        u2 = _state_u(*_evolved_state(case, seed, 70)) if case["cross"] else None
        return _power(u, case["nm"], case["box"], case["nbins"], u2)
    if kind == "ics" and case["np"] <= 256:   # larger fields take too long to draw on the host
        return _exact_ics(case, seed)
    if kind.startswith("nn_"):
        return _exact_nn(case, seed)
    return None   # whole runs: the steps amplify the last digits of the first ones
