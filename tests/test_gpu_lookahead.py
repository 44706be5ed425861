"""Look-ahead (the next panel's factorization beside the rest of the trailing
update) against plain stream order, which calls get beyond the library's 64
helper streams.  In a process of its own: the helpers are never given back."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCRIPT = r"""
import ctypes, sys
import numpy as np, torch
import paper_1303_5837_gb300 as ca
from paper_1303_5837_gb300 import inputs

lib = ca.load()

def new_stream():
    s = ctypes.c_void_p()
    assert lib.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0
    return torch.cuda.ExternalStream(s.value)

def dev(A):
    return torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()

def factor(st, what, m, n, b, L, lv):
    A = dev(inputs.gaussian(m, n, m + n + b))
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        out = (ca.calu_factor if what == "lu" else ca.caqr_factor)(A, b, ca.make_tree(L, lv))
    st.synchronize()
    return [A.cpu().numpy()] + [t.cpu().numpy() for t in out]

torch.cuda.init()
streams = [new_stream() for _ in range(65)]
for st in streams:                       # the first 64 get a helper each, the last none
    factor(st, "lu", 48, 48, 16, 48, [(0, 0)])
for what, m, n, b, L, lv in eval(sys.argv[1]):
    ahead = factor(streams[0], what, m, n, b, L, lv)
    plain = factor(streams[64], what, m, n, b, L, lv)
    if what == "lu":
        assert all(np.array_equal(x, y) for x, y in zip(ahead, plain)), (what, m, n, b)
    else:
        scale = np.linalg.norm(np.triu(plain[0][:n]), axis=0)
        assert (np.abs(np.triu(ahead[0][:n]) - np.triu(plain[0][:n])) <= 1e-12 * scale).all(), (what, m, n, b)
print("same")
"""


def test_look_ahead_gives_the_result_of_the_serial_order():
    """CALU bit for bit (the digit form and the FP64 pipe, panels narrower and
    wider than the digit form's smallest tile); CAQR, whose next-panel columns
    may take a kernel with another order of sums, to rounding."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cases = [("lu", 700, 700, b, 128, [(0, 0)]) for b in (8, 16, 32, 48, 64, 100, 128)]
    cases += [("lu", 900, 500, 32, 128, [(0, 1)]), ("lu", 300, 800, 64, 64, [(0, 0)]),
              ("qr", 900, 600, 32, 128, [(0, 0)]), ("qr", 2000, 1500, 64, 128, [(0, 0)])]
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT, repr(cases)], cwd=root, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stdout[-2000:] + r.stderr[-4000:]
