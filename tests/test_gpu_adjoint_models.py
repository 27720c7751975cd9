"""One grid whose model changes between adjoint passes: the buffers of the recorded pass are those of
its model's blocks (four steps of Model A, two of Model B), so the next forward pass has to size
them anew, and a reverse pass belongs to a forward pass of the same model. Gradients equal a fresh
handle's bit for bit."""
import ctypes

import numpy as np
import pytest

from paper_2109_02598_gb300 import _lib

pytestmark = pytest.mark.gpu

SETUP = {"ac": ((1.0, 1.0), 0.1), "ch": ((1.0, 1.0, 0.5), 0.02)}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def one_pass(g, model, x, lam, n, ckpt):
    coeffs, dt = SETUP[model]
    g.set_model(model, coeffs, dt).write_field(0, x)
    _lib.check(g._lib.pf_adj_forward(g.handle, n, ckpt))
    return backward(g, lam)


def backward(g, lam):
    out, dth = np.empty_like(lam), (ctypes.c_double * 4)()
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (lam, out)]
    _lib.check(g._lib.pf_adj_backward(g.handle, p[0], None, 0, p[1], None, dth))
    return out, np.array(list(dth)[:len(g.coeffs)])


@pytest.mark.parametrize("order", [("ac", "ch", "ac"), ("ch", "ac", "ch")])
@pytest.mark.parametrize("n,ckpt", [(4, 4), (9, 8), (12, 0), (13, 13), (30, 6)])
def test_gradients_after_a_change_of_model(pf, order, n, ckpt):
    rng = np.random.default_rng(11)
    x = (0.2 + 0.5 * rng.random((37, 66))).astype(np.float32)
    lam = (rng.random(x.shape) - 0.3).astype(np.float32)
    g = pf.Grid(x.shape, 1)
    for model in order:
        got, dth = one_pass(g, model, x, lam, n, ckpt)
        fresh = pf.Grid(x.shape, 1)
        want, want_dth = one_pass(fresh, model, x, lam, n, ckpt)
        fresh.close()
        assert np.array_equal(got, want) and np.array_equal(dth, want_dth), model
    g.close()


def test_a_reverse_pass_needs_a_forward_pass_of_its_model(pf):
    x = np.full((16, 64), 0.3, np.float32)
    g = pf.Grid(x.shape, 1)
    want, want_dth = one_pass(g, "ac", x, x, 6, 0)
    g.set_model("ch", *SETUP["ch"])
    with pytest.raises(pf.PfError, match="another model"):
        backward(g, x)
    # back to the recorded model, with other coefficients: the recorded ones count
    g.set_model("ac", (0.5, 0.7), 0.05)
    got, dth = backward(g, x)
    assert np.array_equal(got, want) and np.array_equal(dth, want_dth)
    g.close()
