"""The reverse pass at an interval of the caller's: segments recomputed on a branch of their own into two
buffers while the ones before go back. Many segments (buffers reused, a short last one, one block and
several), launched directly, recorded and replayed; gradients equal those of one-step segments, which
recompute nothing, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SETUP = {"gs": ((0.2, 0.1, 0.04, 0.06), 0.5), "ac": ((1.0, 1.0), 0.1), "ch": ((1.0, 1.0, 0.5), 0.02)}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


@pytest.mark.parametrize("model", ["gs", "ac", "ch"])
@pytest.mark.parametrize("shape", [(40, 66), (388, 516), (900, 1000)])
@pytest.mark.parametrize("n,ckpt", [(47, 5), (40, 9), (33, 3), (24, 12)])
def test_two_branches(pf, model, shape, n, ckpt):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(12)
    nf = 2 if model == "gs" else 1
    x = [torch.rand(shape, generator=gen, device="cuda") * 0.5 + 0.2 for _ in range(nf)]
    lam = [torch.rand(shape, generator=gen, device="cuda") - 0.3 for _ in range(nf)]
    side = torch.cuda.Stream()  # the grid's stream: the default one, and another
    out = []
    for c, stream, passes in ((1, None, 1), (ckpt, None, 3), (ckpt, side, 2)):
        torch.cuda.synchronize()
        g = pf.Grid(shape, nf, stream=stream).set_model(model, *SETUP[model])
        for _ in range(passes):
            g.write_fields(x)
            pf.adjoint_forward(g, n, c)
            d = pf.adjoint_backward(g, *lam)
            g.synchronize()
            out.append([np.asarray(d[2])] + [t.cpu().numpy() for t in d[:2] if t is not None])
        g.close()
    assert all(np.array_equal(a, b) for o in out[1:] for a, b in zip(out[0], o))
