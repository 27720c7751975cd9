"""States that the adjoint's forward pass stores by the library's choice: bounded over all the handles of
a device (4 GiB), given back with the handle, and without influence on the gradients."""
import gc

import pytest

pytestmark = pytest.mark.gpu

N, STEPS = 2048, 400  # 100 states of 33.5 MB by blocks of four steps, 20 + 4 by sqrt(N) checkpoints
STATE = 2 * 4 * N * N


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    import paper_2109_02598_gb300 as pf
    return pf


def forward(pf, g, x, steps=STEPS):
    """Device memory that the forward pass took."""
    import torch
    g.write_fields(x)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    pf.adjoint_forward(g, steps)
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


def setup(pf):
    import torch
    gc.collect()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    x = [torch.rand((N, N), generator=gen, device="cuda") * 0.3 + s for s in (0.5, 0.0)]
    lam = [torch.rand((N, N), generator=gen, device="cuda") - 0.3 for _ in range(2)]
    grids = [pf.Grid((N, N), 2).set_model("gs", (0.2, 0.1, 0.04, 0.06), 0.5) for _ in range(3)]
    return x, lam, grids


def test_stored_states_are_bounded_over_handles(pf):
    import torch
    x, lam, (a, b, c) = setup(pf)
    assert forward(pf, a, x) >= 100 * STATE  # fits alone
    took = forward(pf, b, x)                 # the two together do not
    assert 24 * STATE <= took <= 30 * STATE
    ga, gb = (pf.adjoint_backward(g, *lam) for g in (a, b))
    assert torch.equal(ga[0], gb[0]) and torch.equal(ga[1], gb[1]) and ga[2] == gb[2]
    a.close()                                # given back
    assert forward(pf, c, x) >= 100 * STATE
    b.close()
    c.close()


def test_a_repeated_request_keeps_its_schedule(pf):
    x, lam, (a, b, c) = setup(pf)
    forward(pf, a, x)
    assert forward(pf, b, x) <= 30 * STATE
    a.close()  # there would be room for b's now
    for _ in range(3):
        assert forward(pf, b, x) == 0
        pf.adjoint_backward(b, *lam)
    assert forward(pf, b, x, STEPS - 100) > 40 * STATE  # another request: chosen anew
    assert forward(pf, b, x, STEPS - 100) == 0
    b.close()
    c.close()
