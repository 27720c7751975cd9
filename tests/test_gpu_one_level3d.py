"""The one-level streaming 3D kernel (one step of Allen-Cahn and Gray-Scott with the 7-, 19- and
27-point Laplacians, and of N species), at the edges of its tiles: full rows, ragged rows with
every remainder (wide and short ones, whose ends take several copies a thread), two and three
strips, one-row and one-plane grids. And every monomial of degree three or less in up to four
species, with some of higher degree, on both dimensions' kernels.

Against the oracle after one step and after three: rel L-inf <= 1e-6 per step, the single-step
bar of the other kernels."""
import itertools

import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

COEFFS = {"ac": (1.0, 1.0), "gs": (0.2, 0.1, 0.04, 0.06)}
DT = {"ac": 0.05, "gs": 0.5}
ORACLE_ST = {"std": "std", "iso": "19iso", "iso27": "27iso"}
SHAPES = [(5, 9, 256), (4, 7, 249), (4, 6, 250), (3, 5, 251), (3, 4, 260), (3, 3, 497),
          (21, 23, 40), (9, 70, 73), (2, 3, 1), (1, 1, 4), (1, 2, 7), (5, 1, 50), (40, 5, 9)]


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def uniform(shape, n, seed):
    return tuple(synthetic.uniform(seed, 60 + i, int(np.prod(shape)), 0.05, 0.9)
                 .reshape(shape).astype(np.float32) for i in range(n))


def check(pf, model, x0, coeffs, dt, stencil="std"):
    ref = x0
    g = pf.Grid(x0[0].shape, len(x0)).set_model(model, coeffs, dt)
    if stencil != "std":
        g.set_stencil(stencil)
    g.write_fields(x0)
    for steps in (1, 2):  # single launches
        for _ in range(steps):
            g.step(1)
            ref = oracle.euler_step(model, ref, coeffs, dt, stencil=ORACLE_ST[stencil])
        got = g.read_fields()
        scale = max(np.abs(b).max() for b in ref)
        err = max(np.abs(a.astype(np.float64) - b).max() for a, b in zip(got, ref))
        assert err <= (1e-6 if steps == 1 else 3e-6) * scale
    g.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("stencil", ["std", "iso", "iso27"])
@pytest.mark.parametrize("model", ["ac", "gs"])
def test_stencils(pf, model, stencil, shape):
    check(pf, model, uniform(shape, 1 if model == "ac" else 2, 71), COEFFS[model], DT[model],
          stencil)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1, 2, 3, 4])
def test_species(pf, n, shape):
    E = [[0] * n, [1] + [0] * (n - 1), [0] * (n - 1) + [1], [1] * n, [2] + [0] * (n - 1)]
    K = np.random.RandomState(n).uniform(-0.2, 0.2, size=(n, len(E)))
    check(pf, "rd", uniform(shape, n, 72), oracle.rd_pack((0.2, 0.05, 0.12, 0.07)[:n], E, K), 0.2)


@pytest.mark.parametrize("shape", [(6, 5, 12), (17, 20)])
@pytest.mark.parametrize("n", [1, 2, 3, 4])
def test_every_monomial(pf, n, shape):
    exps = [e for e in itertools.product(range(4), repeat=n) if sum(e) <= 3]
    exps += [e for e in itertools.product(range(4), repeat=n) if sum(e) in (4, 7, 3 * n)][:6]
    order = np.random.RandomState(9 + n).permutation(len(exps))
    x0 = uniform(shape, n, 73)
    for at in range(0, len(exps), 8):
        E = [list(exps[i]) for i in order[at:at + 8]]
        K = np.random.RandomState(at).uniform(-0.2, 0.2, size=(n, len(E)))
        check(pf, "rd", x0, oracle.rd_pack((0.2, 0.05, 0.12, 0.07)[:n], E, K), 0.2)
