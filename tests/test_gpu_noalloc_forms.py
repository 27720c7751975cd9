"""pf_reduce_noalloc after one warm-up call: a call that takes another of the reduction's kernels than
the warm-up did (by quantity, size or alignment) allocates nothing and can be captured into a graph.
In a process of its own, where no other call has loaded any of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import ctypes
import torch
from paper_2109_02598_gb300 import _lib
lib = _lib.load()
out = torch.zeros(8, dtype=torch.float64, device="cuda")
field = torch.full((400 * 404 + 8,), 0.5, device="cuda")

def call(i, what, nx, ny, pitch, offset, stream):
    n = (ctypes.c_int64 * 3)(nx, ny, 1)
    _lib.check(lib.pf_reduce_noalloc(what, 2, n, pitch, ctypes.c_void_p(field.data_ptr() + 4 * offset),
                                     1.0, 0.9, 1.1, ctypes.c_void_p(out.data_ptr() + 8 * i),
                                     ctypes.c_void_p(stream.cuda_stream)))

M, E = _lib.PF_REDUCE_MASS, _lib.PF_REDUCE_ENERGY
s = torch.cuda.Stream()
g = torch.cuda.CUDAGraph()
call(0, M, 8, 8, 8, 0, s)  # the warm-up: one block, vector loads
torch.cuda.synchronize()
forms = [(M, 8, 8, 8, 0), (M, 400, 400, 404, 0), (M, 400, 400, 403, 1), (E, 30, 40, 32, 0),
         (E, 30, 40, 31, 3), (E, 400, 400, 404, 0), (E, 400, 400, 403, 2)]
with torch.cuda.stream(s):
    g.capture_begin()
    for i, f in enumerate(forms):
        call(i + 1, *f, s)
    g.capture_end()
g.replay()
torch.cuda.synchronize()
want = [0.5 * nx * ny if w == M else (-0.5 * 0.9 * 0.25 + 0.25 * 1.1 * 0.0625) * nx * ny
        for w, nx, ny, _, _ in forms]
got = out.cpu().tolist()[1:]
assert all(abs(a - b) <= 1e-12 * abs(b) for a, b in zip(got, want)), (got, want)
for i, f in enumerate(forms):  # and uncaptured
    free = torch.cuda.mem_get_info()[0]
    call(i + 1, *f, s)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free, f
print("captured", len(forms))
"""


def test_every_form_after_one_warm_up(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_02598_gb300.build import build
    build()
    env = dict(os.environ, CUDA_MODULE_LOADING="LAZY")
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "captured 7" in r.stdout, r.stdout + r.stderr
