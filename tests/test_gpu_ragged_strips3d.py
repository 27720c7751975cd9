"""3D streaming kernels on rows too long for one tile whose length is no multiple of four: strips with a
wrapping halo, remainders of one to three columns, two to four strips, and many of which the last has
one to three columns. Bars as in the kernels' own tests."""
import numpy as np
import pytest

import oracle
from test_gpu_one_level3d import COEFFS as COEFFS1, DT as DT1, check, uniform
from test_gpu_two_level3d import COEFFS, DT, fields_for

pytestmark = pytest.mark.gpu

SHAPES = [(3, 4, nx) for nx in (257, 258, 259, 263, 497, 498, 499, 503, 745, 746, 747)]
SHAPES += [(2, 3, nx) for nx in (15129, 15130, 15131)]  # 61 strips of 248 columns and the rest


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
@pytest.mark.parametrize("shape", SHAPES)
def test_two_levels(pf, model, shape):
    x0 = fields_for(model, shape)
    g = pf.Grid(shape, len(x0)).set_model(model, COEFFS[model], DT[model]).set_tuning(32, 16, 1)
    out = []
    for calls in ((1,) * 7, (7,), (2, 5)):
        g.write_fields(x0)
        for n in calls:
            g.step(n)
        out.append(g.read_fields())
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(o, out[0]))
    two = g.write_fields(x0).step(2).read_fields()
    g.close()
    want = oracle.run(model, x0, COEFFS[model], DT[model], 2)
    scale = max(np.abs(b).max() for b in want)
    assert max(np.abs(a.astype(np.float64) - b).max() for a, b in zip(two, want)) <= 2e-6 * scale


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("stencil", ["std", "iso", "iso27"])
@pytest.mark.parametrize("model", ["ac", "gs"])
def test_stencils(pf, model, stencil, shape):
    check(pf, model, uniform(shape, 1 if model == "ac" else 2, 71), COEFFS1[model], DT1[model], stencil)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1, 3, 4])
def test_species(pf, n, shape):
    E = [[0] * n, [1] + [0] * (n - 1), [0] * (n - 1) + [1], [1] * n, [2] + [0] * (n - 1)]
    K = np.random.RandomState(n).uniform(-0.2, 0.2, size=(n, len(E)))
    check(pf, "rd", uniform(shape, n, 72), oracle.rd_pack((0.2, 0.05, 0.12, 0.07)[:n], E, K), 0.2)
