"""A grid or batch without a tuning of the caller's stays so: through a checkpoint, where a restored run
is to take the kernels (and bits) of the one it resumes, and through a call that keeps the present
values."""
import ctypes

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
    v = ctypes.c_int(-1)
    ask = g._lib.pf_batch_is_untuned if hasattr(g, "shapes") else g._lib.pf_is_untuned
    assert ask(g._h, ctypes.byref(v)) == 0
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


def test_batch_keeps_its_values(pf):
    rng = np.random.default_rng(6)
    shapes = [(40, 52), (33, 70)]
    x = [[(0.2 + 0.3 * rng.random(s)).astype(np.float32) for _ in range(2)] for s in shapes]

    def run(b):
        for i in range(2):
            for f in range(2):
                b.write(i, f, x[i][f])
        b.run(11)
        return [b.read(i, f) for i in range(2) for f in range(2)]

    specs = [dict(nx=s[1], ny=s[0], Du=0.2, Dv=0.1, F=0.04, k=0.06) for s in shapes]
    b = pf.Batch(specs, 0.5)
    assert untuned(b)
    want, named = run(b), b.tuning
    b.set_tuning(0, 0, 0)
    assert untuned(b) and b.tuning == named
    assert all(np.array_equal(p, q) for p, q in zip(want, run(b)))
    b.set_tuning(*named)  # asked for: runs what it names
    assert not untuned(b)
    b.set_tuning(0, 0, 0)
    assert not untuned(b) and b.tuning == named
    assert all(np.array_equal(p, q) for p, q in zip(want, run(b)))
    b.close()
