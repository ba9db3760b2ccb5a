"""A CUDA error is reported by the call that met it, and not again by the next one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Synchronising a stream that is being captured is an error that CUDA returns (and ends the
# capture). In a process of its own and without torch, which clears pending errors itself.
PROGRAM = """
import ctypes
from paper_2201_10132_gb300 import build, tfkt as T
build.build()
T.lib()
rt = ctypes.CDLL("libcudart.so.13")
st, graph = ctypes.c_void_p(), ctypes.c_void_p()
assert rt.cudaStreamCreateWithFlags(ctypes.byref(st), 1) == 0
p = T.Params(64, 32, 6, 3.0, 5.0, 0.5, 0.2, 0.05, 1, 0.0, 0.0, 1, T.FP32)
a = T.Solver(p, stream=st.value)
a.sync()
assert rt.cudaStreamBeginCapture(st, 1) == 0
try:
    a.sync()
    status = 0
except T.TfktError as e:
    status = e.status
pending = rt.cudaPeekAtLastError()
rt.cudaStreamEndCapture(st, ctypes.byref(graph))
rt.cudaGetLastError()                 # this program's own call
assert status == 3, status            # TFKT_ECUDA
assert pending == 0, pending
with T.Solver(p) as b:                # another context is untouched
    b.step(2)
    b.sync()
print("done")
"""


def test_the_next_context_is_usable():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr
