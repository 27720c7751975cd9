"""Task heights of the 2D strip kernel: grids whose rows make one short task, several tasks of the
least height with a short last one, and more strips than a wave of warps holds. The tiled
kernel's bits (which the parity tests hold to the oracle)."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

COEFFS = {"ac": (1.0, 1.0), "ch": (1.0, 1.0, 1.0), "gs": (0.2, 0.1, 0.04, 0.06),
          "c": (1.0, 1.0, 1.0, 1.0, 1.0)}
DT = {"ac": 0.05, "ch": 0.01, "gs": 0.5, "c": 0.005}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


@pytest.mark.parametrize("model", ["ac", "gs", "ch", "c"])
@pytest.mark.parametrize("shape", [(1, 300), (3, 70), (5, 130), (13, 64), (61, 517), (7, 30011),
                                   (3, 400003), (1111, 90)])
def test_strip_heights_are_bitwise_the_tiles(pf, model, shape):
    n = 2 if model in ("gs", "c") else 1
    x0 = tuple(synthetic.uniform(7, 60 + i, int(np.prod(shape)), 0.05, 0.6).reshape(shape)
               .astype(np.float32) for i in range(n))

    def run(tuning):
        g = pf.Grid(shape, n).set_model(model, COEFFS[model], DT[model]).write_fields(x0)
        g.set_tuning(*tuning)
        g.step(5)
        g.step(8)
        out = g.read_fields()
        g.close()
        return out

    ref = run((128, 16, 1))
    for width in (64, 128):
        for k in ((1, 2, 4) if model in ("ac", "gs") else (1, 2)):
            for a, b in zip(run((width, pf.PF_TILE_STRIPS, k)), ref):
                assert np.array_equal(a, b), (width, k)
