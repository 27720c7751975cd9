"""Blocks of adjoint steps (several reverse steps in one launch, their states recomputed on chip):
tile edges, ragged widths, grids below a tile and its halo, every remainder of the block length.
Gradients equal those of one-step blocks bit for bit, and the initial state's those of the FP64
oracle to 1e-4 relative L2: up to 9 steps of a dozen FP32 roundings (2^-24) on terms of at most
four times lambda, 9 * 12 * 4 * 6e-8 = 2.6e-5 of lambda^N's size, of which diffusion leaves at
least a third in these runs."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SETUP = {"gs": ((0.2, 0.1, 0.04, 0.06), 0.5), "ac": ((1.0, 1.0), 0.1),
         "ch": ((1.0, 1.0, 0.5), 0.02)}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def inputs(model, shape):
    rng = np.random.default_rng(7)
    nf = 2 if model == "gs" else 1
    x = [(0.2 + 0.5 * rng.random(shape)).astype(np.float32) for _ in range(nf)]
    return x, [(rng.random(shape) - 0.3).astype(np.float32) for _ in range(nf)]


def gradients(pf, model, x, lam, n, ckpt, passes=1):
    from paper_2109_02598_gb300 import _lib
    coeffs, dt = SETUP[model]
    g = pf.Grid(x[0].shape, len(x)).set_model(model, coeffs, dt)
    ptr = [a.ctypes.data_as(ctypes.c_void_p) for a in lam] + [None]
    for _ in range(passes):
        for f, a in enumerate(x):
            g.write_field(f, a)
        _lib.check(g._lib.pf_adj_forward(g.handle, n, ckpt))
        out = [np.empty_like(a) for a in x]
        po = [a.ctypes.data_as(ctypes.c_void_p) for a in out] + [None]
        dth = (ctypes.c_double * 4)()
        _lib.check(g._lib.pf_adj_backward(g.handle, ptr[0], ptr[1], 0, po[0], po[1], dth))
    g.close()
    return out, np.array(list(dth)[:len(coeffs)])


@pytest.mark.parametrize("model", ["gs", "ac", "ch"])
@pytest.mark.parametrize("shape", [(16, 64), (17, 65), (3, 5), (33, 127), (50, 202)])
@pytest.mark.parametrize("n,ckpt", [(5, 0), (6, 0), (7, 0), (8, 0), (9, 7), (9, 9)])
def test_blocks(pf, model, shape, n, ckpt):
    x, lam = inputs(model, shape)
    g0, dth = gradients(pf, model, x, lam, n, ckpt, passes=3)
    one, one_th = gradients(pf, model, x, lam, n, 1)
    assert all(np.array_equal(a, b) for a, b in zip(g0, one)) and np.array_equal(dth, one_th)
    coeffs, dt = SETUP[model]
    if model == "gs":
        ref = oracle.gray_scott_adjoint(*x, coeffs, dt, n, *[a.astype(np.float64) for a in lam])[:2]
    else:
        ref = oracle.phase_field_adjoint(model, x[0], coeffs, dt, n, lam[0].astype(np.float64))[:1]
    err = sum(((a - r) ** 2).sum() for a, r in zip(g0, ref))
    assert err <= 1e-8 * sum((r ** 2).sum() for r in ref)


@pytest.mark.parametrize("model", ["gs", "ac", "ch"])
def test_states_recomputed_by_strips(pf, model):
    # above 2^21 sites the states between blocks are recomputed by the strip kernel
    x, lam = inputs(model, (1100, 1950))
    g0, dth = gradients(pf, model, x, lam, 9, 9)
    one, one_th = gradients(pf, model, x, lam, 9, 1)
    assert all(np.array_equal(a, b) for a, b in zip(g0, one)) and np.array_equal(dth, one_th)
