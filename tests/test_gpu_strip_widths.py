"""Widths of the 2D strip kernel: rows shorter than a strip, of a length that is and is not a multiple
of a lane's columns, and strips that end at, before and after the row's end, in grids and as
instances of a batch; and the sizes at which an untuned grid changes kernels. The tiled kernel's
bits (which the parity tests hold to the oracle)."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

COEFFS = {"ac": (1.0, 1.0), "ch": (1.0, 1.0, 1.0), "gs": (0.2, 0.1, 0.04, 0.06),
          "c": (1.0, 1.0, 1.0, 1.0, 1.0)}
DT = {"ac": 0.05, "ch": 0.01, "gs": 0.5, "c": 0.005}
WIDTHS = [1, 2, 3, 4, 5, 6, 8, 31, 52, 55, 56, 57, 58, 62, 64, 65, 113, 114, 119, 120, 121, 122, 124,
          126, 127, 128, 130, 224, 225, 240, 242, 244]


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def fields(model, shape):
    n = 2 if model in ("gs", "c") else 1
    return tuple(synthetic.uniform(9, 80 + i, int(np.prod(shape)), 0.05, 0.6).reshape(shape)
                 .astype(np.float32) for i in range(n))


def run(pf, model, x0, tuning, steps=(5, 8)):
    g = pf.Grid(x0[0].shape, len(x0)).set_model(model, COEFFS[model], DT[model]).write_fields(x0)
    if tuning:
        g.set_tuning(*tuning)
    for n in steps:
        g.step(n)
    out = g.read_fields()
    g.close()
    return out


@pytest.mark.parametrize("model", ["ac", "gs", "ch", "c"])
@pytest.mark.parametrize("nx", WIDTHS)
def test_strip_widths_are_bitwise_the_tiles(pf, model, nx):
    x0 = fields(model, (21, nx))
    ref = run(pf, model, x0, (128, 16, 1))
    for width in (64, 128):
        for k in ((1, 2, 4) if model in ("ac", "gs") else (1, 2)):
            for a, b in zip(run(pf, model, x0, (width, pf.PF_TILE_STRIPS, k)), ref):
                assert np.array_equal(a, b), (width, k)


def test_batch_of_all_widths_is_bitwise_the_tiled_batch(pf):
    def batch(tuning):
        b = pf.Batch([dict(nx=nx, ny=13 + i, Du=0.2, Dv=0.1, F=0.04, k=0.06)
                      for i, nx in enumerate(WIDTHS)], 0.5)
        for i, nx in enumerate(WIDTHS):
            for f, a in enumerate(fields("gs", (13 + i, nx))):
                b.write(i, f, a)
        if tuning:
            b.set_tuning(*tuning)
        else:  # the probes leave the state as it was
            b.autotune()
        b.run(13)
        out = [b.read(i, f) for i in range(len(WIDTHS)) for f in (0, 1)]
        b.close()
        return out

    ref = batch((64, 16, 1))
    for tuning in [(w, pf.PF_TILE_STRIPS, k) for w in (64, 128) for k in (1, 2, 4)] + [None]:
        assert all(np.array_equal(a, b) for a, b in zip(batch(tuning), ref)), tuning


@pytest.mark.parametrize("model,shape", [("gs", (1024, 768)), ("gs", (769, 1024)), ("ac", (1023, 771)),
                                         ("ch", (770, 1023)), ("c", (769, 1025)),
                                         ("c", (2048, 3072)), ("c", (2047, 3077))])
def test_untuned_grids_are_bitwise_the_tiles(pf, model, shape):
    x0 = fields(model, shape)
    for a, b in zip(run(pf, model, x0, None, (7,)), run(pf, model, x0, (128, 16, 1), (7,))):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("calls", [(13,), (1, 2, 3, 7), (4, 9)])
def test_untuned_batch_is_bitwise_depth_one(pf, calls):
    def batch(tuning):
        b = pf.Batch([dict(nx=nx, ny=13 + i, Du=0.2, Dv=0.1, F=0.04, k=0.06)
                      for i, nx in enumerate(WIDTHS)], 0.5)
        for i, nx in enumerate(WIDTHS):
            for f, a in enumerate(fields("gs", (13 + i, nx))):
                b.write(i, f, a)
        if tuning:
            b.set_tuning(*tuning)
        for n in calls:
            b.run(n)
        out = [b.read(i, f) for i in range(len(WIDTHS)) for f in (0, 1)]
        b.close()
        return out

    assert all(np.array_equal(a, b) for a, b in zip(batch(None), batch((64, 16, 1))))
