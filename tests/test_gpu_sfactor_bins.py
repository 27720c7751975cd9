"""Binning of the structure factor at the edges of its walk along ky: half spectra of one to
several chunks of kx with and without a Nyquist column, row counts around the load-ahead and the
segments, one bin and the most bins, and spacings at which squared wavenumbers under- or
overflow. Against the oracle: counts and centres exactly, means to 1e-10 of the largest (the bar
of the other structure-factor tests)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


@pytest.mark.parametrize("shape", [(1, 2), (7, 3), (9, 62), (65, 64), (130, 131), (64, 66),
                                   (2, 3, 4), (5, 8, 63), (3, 33, 128), (17, 16, 2)])
@pytest.mark.parametrize("bins", [1, 2, 31, 1024])
@pytest.mark.parametrize("h", [1.0, 0.37, 1e-170, 1e170])
def test_bins_against_the_oracle(pf, shape, bins, h):
    psi = np.random.RandomState(len(shape) + bins).uniform(-1, 1, shape).astype(np.float32)
    with np.errstate(all="ignore"):
        c0, m0, n0 = oracle.structure_factor(psi, h, bins)
    c, m, n = pf.structure_factor(psi, h, bins)
    assert np.array_equal(c, c0) and np.array_equal(n, n0)
    assert np.abs(m - m0).max() <= 1e-10 * max(1.0, m0.max())
