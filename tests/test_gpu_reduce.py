"""Mass and free energy against sums in extended precision: the row ends (one to nine columns
past a multiple of four, rows of one to several warps), row blocks that end early, single planes,
both sides of the FP64 form's size limit, the value ranges of the error-free pairs and those
beyond them, and a caller's field whose pitch and address allow no vector loads.

Tolerance: sums of N terms whose own rounding is 2^-53, in trees at most 40 additions deep:
40 x 2^-53 = 4.5e-15 of the sum of the terms' magnitudes."""
import ctypes

import numpy as np
import pytest

from paper_2109_02598_gb300 import _lib

pytestmark = pytest.mark.gpu
TOL = 4.5e-15
L = np.longdouble


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def energy_terms(fields, c, h):
    p = fields[0]
    t = [L(0.5) * ((np.roll(x, -1, d) - x) / L(h)) ** 2 for x in fields for d in range(x.ndim)]
    t += [-L(0.5) * L(c[0]) * p * p, L(0.25) * L(c[1]) * p ** 4]
    if len(fields) == 2:
        m = fields[1]
        t += [-L(0.5) * L(c[2]) * m * m, L(0.25) * L(c[3]) * m ** 4, -L(c[4]) * p * p * m]
    return t


def values(kind, shape, seed):
    r = np.random.RandomState(seed)
    x = r.uniform(-1, 1, size=(2,) + shape)
    if kind == "wide":  # magnitudes on both sides of every limit of the pairs
        x *= 10.0 ** r.uniform(-12, 8, size=x.shape)
    if kind == "blocks":  # whole chunks zero, tiny or large
        x *= np.repeat(10.0 ** r.choice([-9.0, 0.0, 7.0], size=(2,) + shape[:-1] + (1,)),
                       shape[-1], axis=-1)
        x[..., : shape[-1] // 3] = 0
    return x.astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (9, 5), (128, 128), (33, 127), (7, 1030),
                                   (1, 1, 4), (3, 2, 6), (9, 30, 70), (40, 40, 41), (41, 40, 40),
                                   (37, 64, 65)])
@pytest.mark.parametrize("kind", ["noise", "wide", "blocks"])
def test_mass_and_energy(pf, shape, kind):
    x = values(kind, shape, 31)
    f = [a.astype(L) for a in x]
    h, vol = 0.7, L(0.7) ** len(shape)
    for model, c in (("ac", (0.9, 1.1)), ("c", (1.0, 0.9, 1.1, 0.8, 0.7))):
        nf = 1 if model == "ac" else 2
        g = pf.Grid(shape, nf, h).set_model(model, c, 1e-6, force=True).write_fields(x[:nf])
        for k in range(nf):
            got = g.mass(k)
            assert abs(L(got) - f[k].sum() * vol) <= TOL * np.abs(f[k]).sum() * vol
        t = energy_terms(f[:nf], c, h)
        want, size = sum(a.sum() for a in t) * vol, sum(np.abs(a).sum() for a in t) * vol
        assert abs(L(g.energy()) - want) <= TOL * size
        g.close()


@pytest.mark.parametrize("nx,pitch,offset", [(61, 61, 0), (64, 64, 1), (30, 35, 2), (8, 12, 0)])
def test_noalloc_takes_any_pitch_and_address(pf, nx, pitch, offset):
    import torch
    lib, ny = _lib.load(), 45
    buf = torch.full((offset + ny * pitch,), float("nan"), device="cuda")
    x = values("noise", (ny, nx), 5)[0]
    view = buf[offset:].view(ny, pitch)
    view[:, :nx] = torch.from_numpy(x).cuda()
    # the last row ends with its last value
    ptr = buf.data_ptr() + 4 * offset
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    n = (ctypes.c_int64 * 3)(nx, ny, 1)
    s = torch.cuda.current_stream().cuda_stream
    for i, what in enumerate((_lib.PF_REDUCE_MASS, _lib.PF_REDUCE_ENERGY)):
        _lib.check(lib.pf_reduce_noalloc(what, 2, n, pitch, ctypes.c_void_p(ptr), 1.0, 0.9, 1.1,
                                         ctypes.c_void_p(out.data_ptr() + 8 * i),
                                         ctypes.c_void_p(s)))
    mass, energy = out.cpu().numpy()
    f = x.astype(L)
    t = energy_terms([f], (0.9, 1.1), 1.0)
    assert abs(L(mass) - f.sum()) <= TOL * np.abs(f).sum()
    assert abs(L(energy) - sum(a.sum() for a in t)) <= TOL * sum(np.abs(a).sum() for a in t)
