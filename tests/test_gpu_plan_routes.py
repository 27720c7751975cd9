"""Untuned grids that leave the usual kernels: few rows, few planes, and single steps of large grids. The
same bits as a tuning of the caller's, for a single step, the library's depth and what it leaves over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SETUP = {"ac": ((1.0, 1.0), 0.05), "ch": ((1.0, 1.0, 1.0), 0.01), "gs": ((0.2, 0.1, 0.04, 0.06), 0.5),
         "c": ((1.0,) * 5, 0.005)}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


@pytest.mark.parametrize("model,shape", [
    # few rows: strips where the sites alone would call for tiles
    ("ac", (1, 65537)), ("ch", (4, 65536)), ("gs", (11, 30002)), ("c", (33, 12301)),
    # single steps beyond the L2 cache
    ("gs", (2561, 2562)), ("ac", (3601, 3600)), ("c", (2600, 2601)), ("ch", (3500, 3602)),
    ("gs", (260, 256, 256)), ("ac", (128, 320, 320)), ("gs", (101, 384, 330)),
    # few large planes
    ("ac", (1, 1024, 1024)), ("gs", (2, 752, 768)), ("ch", (4, 1024, 640)), ("ac", (3, 733, 745)),
    ("ac", (9, 1600, 1536)), ("gs", (5, 1600, 1664))])
def test_untuned_equals_explicit(pf, model, shape):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    coeffs, dt = SETUP[model]
    x = [torch.rand(shape, generator=gen, device="cuda") * 0.2 + s
         for s in ((0.7, 0.1) if model in ("gs", "c") else (-0.1,))]
    tuning = (64, 16, 1) if len(shape) == 2 else (32, 16, 1)
    grids = [pf.Grid(shape, len(x)).set_model(model, coeffs, dt) for _ in range(2)]
    grids[1].set_tuning(*tuning)
    for n in (1, 3, 7, 30):  # (30: a graph)
        out = []
        for g in grids:
            g.write_fields(x).step(n)
            out.append(g.read_fields(device=True))
        assert all(torch.equal(a, b) for a, b in zip(*out)), n
    for g in grids:
        g.close()
