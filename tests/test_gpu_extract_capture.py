"""plhr_tharm_extract under stream capture: as the process's first call, after the last
operator has gone (when the workspace pool changes its state), while an operator lives,
and with an operator destroyed during the capture; each in a process of its own.  The
replayed graph gives what the plain call gives."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes, sys, torch
import paper_1408_0042_gb300 as plhr
mode = sys.argv[1]
lib, m, kp = plhr.load_library(), 12, 4
d = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")
G = [torch.eye(m, dtype=torch.float64, device="cuda") for _ in range(3)]
G[1] = torch.diag(torch.arange(1.0, m + 1, dtype=torch.float64, device="cuda"))
cs, outs = d(m) + 1.0, [d(m, kp), d(kp, kp), d(kp), d(kp), d(2 * kp), d(4)]
ptr = lambda t: ctypes.c_void_p(t.data_ptr())

def extract():
    return lib.plhr_tharm_extract(m, kp, kp, *[ptr(t) for t in G], ptr(cs), *[ptr(t) for t in outs], None,
                                  torch.cuda.current_stream().cuda_stream)

if mode != "first":
    op = plhr.Operator.laplacian((8, 8), 0.1)
    assert extract() == 0
    torch.cuda.synchronize()
    if mode == "gone":
        del op
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    if mode == "destroyed":
        del op
    assert extract() == 0
for t in outs:
    t.zero_()
graph.replay()
torch.cuda.synchronize()
got = [t.cpu() for t in outs]
for t in outs:
    t.zero_()
assert extract() == 0
torch.cuda.synchronize()
bits = lambda t: t.cpu().view(torch.int64)     # two of the outputs hold ints
assert all(torch.equal(bits(a), bits(b)) for a, b in zip(got, outs))
assert [round(x, 12) for x in got[4][::2].tolist()] == [1.0, 2.0, 3.0, 4.0]
"""


@pytest.mark.parametrize("mode", ["first", "gone", "lives", "destroyed"])
def test_capture(mode):
    import __graft_entry__
    __graft_entry__.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT, mode], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
