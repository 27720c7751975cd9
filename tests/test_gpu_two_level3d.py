"""The two-level 3D kernel behind the general tiles (two steps a launch for Allen-Cahn and
Gray-Scott, chemical potential and step for Models B and C; 7-point stencil, any size): against
the oracle, and for the models that have one, bit for bit against the single-step kernel that
also takes any size. Shapes at the edges of its cases: full rows (nx % 4 == 0, nx <= 256), one
strip of ragged rows with every remainder, two and three strips (one of them a column wide),
row counts around a tile, grids thinner than the halo, and single planes."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

COEFFS = {"ac": (1.0, 1.0), "ch": (1.0, 1.0, 1.0), "gs": (0.2, 0.1, 0.04, 0.06),
          "c": (1.0, 1.0, 1.0, 1.0, 1.0)}
DT = {"ac": 0.05, "ch": 0.01, "gs": 0.5, "c": 0.005}
SHAPES = [(6, 9, 256), (5, 11, 248), (4, 7, 249), (5, 6, 250), (4, 9, 251), (3, 5, 260),
          (3, 4, 497), (33, 35, 30), (18, 41, 64), (2, 3, 1), (1, 1, 4), (1, 2, 7), (64, 5, 12),
          (3, 330, 9)]


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def fields_for(model, shape):
    if model == "gs":
        return synthetic.gray_scott_init(shape, seed=700, n_seeds=3, side=4, noise=0.05)
    x = synthetic.allen_cahn_init(shape, seed=701, lo=-0.5, hi=0.5)
    if model == "c":
        return (x, synthetic.cahn_hilliard_init(shape, seed=702, amp=0.4))
    return (x,)


@pytest.mark.parametrize("model", ["ac", "gs", "ch", "c"])
@pytest.mark.parametrize("shape", SHAPES)
def test_two_level_kernel(pf, model, shape):
    x0 = fields_for(model, shape)

    def run(calls, tuning=(32, 16, 1)):
        g = pf.Grid(shape, len(x0)).set_model(model, COEFFS[model], DT[model])
        if tuning is not None:
            g.set_tuning(*tuning)
            assert g.tuning == tuning
        g.write_fields(x0)
        for n in calls:
            g.step(n)
        out = g.read_fields()
        g.close()
        return out

    # one call of six steps, an odd call, calls of two (direct launches), and the library's
    # default: the same bits as single steps, and within the parity bars of the oracle
    # (1e-6 per step for these few steps)
    ref = run([1] * 18)
    for calls, tuning in (((18,), (32, 16, 1)), ((7, 11), (64, 8, 1)), ((2,) * 9, None)):
        for a, b in zip(run(calls, tuning), ref):
            assert np.array_equal(a, b), (calls, tuning)
    two = run((2,))
    want = oracle.run(model, x0, COEFFS[model], DT[model], 2)
    scale = max(np.abs(b).max() for b in want)
    assert max(np.abs(a.astype(np.float64) - b).max() for a, b in zip(two, want)) <= 2e-6 * scale
