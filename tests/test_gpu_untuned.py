"""A grid or batch without a tuning of the caller's stays so: through a checkpoint, where a restored run
is to take the kernels (and bits) of the one it resumes, and through a call that keeps the present
values."""
import numpy as np
import pytest

from paper_2109_02598_gb300 import checkpoint

pytestmark = pytest.mark.gpu

SETUP = {"gs": ((0.2, 0.1, 0.04, 0.06), 0.5), "ch": ((1.0, 1.0, 1.0), 0.01)}


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def untuned(g):
    import ctypes
    v = ctypes.c_int(-1)
    assert g._lib.pf_is_untuned(g.handle, ctypes.byref(v)) == 0
    return bool(v.value)


@pytest.mark.parametrize("model,shape,tuning", [("gs", (70, 90), (64, 16, 1)), ("ch", (96, 128), (128, 16, 2)),
                                                ("gs", (16, 32, 128), (128, 16, 1))])
def test_checkpoints_keep_a_grid_untuned(pf, tmp_path, model, shape, tuning):
    rng = np.random.default_rng(5)
    coeffs, dt = SETUP[model]
    x = [(0.2 + 0.3 * rng.random(shape)).astype(np.float32) for _ in range(2 if model == "gs" else 1)]
    path = str(tmp_path / "c.npz")
    g = pf.Grid(shape, len(x)).set_model(model, coeffs, dt).write_fields(x)
    assert untuned(g)
    g.step(7).save(path)
    g.step(9)
    want = g.read_fields()
    assert checkpoint.load_state(path)[0]["tuning"] == [0, 0, 0]
    h = pf.Grid.load(path)
    assert untuned(h) and h.tuning == g.tuning
    h.step(9)
    assert all(np.array_equal(a, b) for a, b in zip(want, h.read_fields()))
    h.set_tuning(*tuning).save(path)  # a tuning of the caller's, the default tile's among them
    h.close()
    h = pf.Grid.load(path)
    assert not untuned(h) and h.tuning == tuning
    h.set_tuning(0, 0, 0)
    assert untuned(h)
    h.set_tuning(0, 0, 1)
    assert not untuned(h)
    h.set_stencil("iso")  # which resets the tuning
    assert untuned(h)
    h.close()
    g.close()
