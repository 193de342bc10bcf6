"""The first computation of a process may be inside a stream capture: setting a context up
leaves nothing for the calls to set up."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1406_4350_gb300 import build
    build.build()


FIRST_CALL = """
import numpy as np, torch, sys
sys.path.insert(0, %r)
from synth import make_cell
from paper_1406_4350_gb300.chebfi import ChebFI, _block, _stream, fortran
import ctypes
n = %d
L = 0.42 * n
cell = make_cell(L, n, 0.5 * (2.0 * np.pi / L * 0.23 * n) ** 2, 1, 8, 3, True, 41)
g = ChebFI.from_cell(cell)
Y = fortran(cell.Y0)
out = torch.zeros_like(Y)
f = g.lib.chebfi_apply_H_noalloc
f.restype = ctypes.c_int
f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int64] * 2 + [ctypes.c_void_p]
handle = ctypes.c_void_p()
assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(handle))) == 0
side = torch.cuda.ExternalStream(handle.value)  # a stream that the default stream orders itself with
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, stream=side):
    y, nb, ld = _block(Y)
    rc = f(g.h, y, _block(out)[0], nb, ld, _stream())
    assert rc == 0, g.lib.chebfi_last_error(g.h).decode()
graph.replay()
torch.cuda.synchronize()
ref = g.apply_H(Y)
assert torch.equal(out, ref) or (out - ref).abs().max() <= 1e-11 * ref.abs().max()
print("captured")
"""


# the first computation of a process, inside a stream capture: nothing may be left to set up
# (a general grid, fixed-point planes between FP64 and between double-float z passes, and the
# compiled FP64 passes)
@pytest.mark.parametrize("n", [18, 20, 24, 90])
def test_first_call_inside_a_capture(n):
    r = subprocess.run([sys.executable, "-c", FIRST_CALL % (ROOT, n)], capture_output=True, text=True, cwd=ROOT,
                       timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]
