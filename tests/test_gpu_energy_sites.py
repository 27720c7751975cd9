"""Free energy of large grids (2^16 sites and more) where it lies in a few sites of a flat field, and
in 2D with rows of several pieces, every remainder of nx by 4 and row blocks that end early.

Tolerance of the few sites, of the sum of the terms' magnitudes, h = 1 (so that h rounds nothing): a
term passes at most 2 roundings to 2^-53 as its thread's words become a double, 1 by its coefficient,
2 (Model C: 5) in its thread's sum, and one addition per further thread with a term: the sites' own,
their neighbours' to the left, in the row and in the plane before, at most 4 threads for one site and 7
for two. So 8 (11) and 11 (14) times 2^-53."""
import ctypes

import numpy as np
import pytest

from paper_2109_02598_gb300 import _lib
from test_gpu_reduce import L, TOL, energy_terms, values

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def few(x, c):
    """Energy and its terms' magnitudes of a field that is zero but at the middle of x's box."""
    t = energy_terms([a.astype(L) for a in x], c, 1.0)
    return sum(a.sum() for a in t), sum(np.abs(a).sum() for a in t)


@pytest.mark.parametrize("shape", [(300, 259), (41, 40, 40)])
@pytest.mark.parametrize("sites", [1, 2])
@pytest.mark.parametrize("model,c", [("ac", (0.9, 1.1)), ("ac", (0.0, 0.0)),
                                     ("c", (1.0, 0.9, 1.1, 0.8, 0.7))])
def test_energy_in_few_sites(pf, shape, sites, model, c):
    r = np.random.RandomState(5)
    nf = 1 if model == "ac" else 2
    bound = (8 if sites == 1 else 11) + (3 if nf == 2 else 0)
    g = pf.Grid(shape, nf).set_model(model, c, 1e-6, force=True)
    box = (5,) * len(shape)
    for _ in range(64):
        at = tuple(r.randint(2, s - 3) for s in shape)
        v = r.uniform(50, 150, size=(nf, sites)) * r.choice([-1, 1], size=(nf, sites))
        x = np.zeros((nf,) + shape, np.float32)
        b = np.zeros((nf,) + box, np.float32)
        x[(slice(None),) + at[:-1] + (slice(at[-1], at[-1] + sites),)] = v
        b[(slice(None),) + (2,) * (len(shape) - 1) + (slice(2, 2 + sites),)] = v
        g.write_fields(x)
        want, size = few(b, c)
        assert abs(L(g.energy()) - want) <= bound * L(2.0) ** -53 * size, (at, v)
    g.close()


@pytest.mark.parametrize("shape", [(257, 256), (300, 259), (67, 1030), (33, 2049), (131, 514)])
@pytest.mark.parametrize("kind", ["noise", "wide", "blocks"])
def test_large_2d(pf, shape, kind):
    x = values(kind, shape, 37)
    f = [a.astype(L) for a in x]
    for model, c in (("ac", (0.9, 1.1)), ("c", (1.0, 0.9, 1.1, 0.8, 0.7))):
        nf = 1 if model == "ac" else 2
        g = pf.Grid(shape, nf, 0.7).set_model(model, c, 1e-6, force=True).write_fields(x[:nf])
        for k in range(nf):
            assert abs(L(g.mass(k)) - f[k].sum() * L(0.7) ** 2) <= TOL * np.abs(f[k]).sum() * L(0.7) ** 2
        t = energy_terms(f[:nf], c, 0.7)
        want, size = sum(a.sum() for a in t) * L(0.7) ** 2, sum(np.abs(a).sum() for a in t) * L(0.7) ** 2
        assert abs(L(g.energy()) - want) <= TOL * size
        g.close()


def test_large_field_of_odd_pitch_and_address(pf):
    import torch
    lib, nx, ny, pitch, offset = _lib.load(), 261, 260, 263, 3
    buf = torch.full((offset + ny * pitch,), float("nan"), device="cuda")
    x = values("noise", (ny, nx), 6)[0]
    buf[offset:].view(ny, pitch)[:, :nx] = torch.from_numpy(x).cuda()
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    n = (ctypes.c_int64 * 3)(nx, ny, 1)
    for i, what in enumerate((_lib.PF_REDUCE_MASS, _lib.PF_REDUCE_ENERGY)):
        _lib.check(lib.pf_reduce_noalloc(what, 2, n, pitch, ctypes.c_void_p(buf.data_ptr() + 4 * offset),
                                         1.0, 0.9, 1.1, ctypes.c_void_p(out.data_ptr() + 8 * i),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    mass, energy = out.cpu().numpy()
    f = x.astype(L)
    t = energy_terms([f], (0.9, 1.1), 1.0)
    assert abs(L(mass) - f.sum()) <= TOL * np.abs(f).sum()
    assert abs(L(energy) - sum(a.sum() for a in t)) <= TOL * sum(np.abs(a).sum() for a in t)
