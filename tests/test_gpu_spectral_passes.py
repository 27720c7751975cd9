"""The fused spectral engine's pass plans that the other sizes do not reach: every last radix (2, 4,
8) with none, one or more radix-8 passes beside it, along x, y and z, against the FP64 oracle with
the bar of the other fused sizes (2e-5 after 20 steps), and a call of several steps equal to as
many calls of one, bit for bit."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

COEFFS = {"ac": (1.0, 1.0), "c": (1.0, 1.0, 1.0, 1.0, 1.0)}
DT = {"ac": 0.05, "c": 0.005}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def run(pf, model, x0, calls):
    s = pf.Spectral(x0[0].shape, model, COEFFS[model], DT[model])
    s.set_engine("fused")
    for f, x in enumerate(x0):
        s.write_field(f, x)
    for n in calls:
        s.step(n)
    out = s.read_fields()
    s.close()
    return out


@pytest.mark.parametrize("model", ["ac", "c"])
@pytest.mark.parametrize("shape", [(4, 32), (8, 512), (512, 32), (1024, 16), (32, 4, 8),
                                   (2, 8, 512), (8, 128, 4), (128, 4, 8)])
def test_pass_plans(pf, model, shape):
    x0 = [synthetic.allen_cahn_init(shape, seed=17 + f, lo=-0.5, hi=0.5)
          for f in range(len(COEFFS[model]) // 2)]
    got = run(pf, model, x0, [20])
    ref = oracle.spectral_run(model, x0, COEFFS[model], DT[model], 20)
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 2e-5 * np.abs(r).max()
    for g, one in zip(got, run(pf, model, x0, [1] * 20)):
        assert np.array_equal(g, one)
