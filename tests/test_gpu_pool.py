"""The workspace pool is given back: with the last operator, also when a release is
still queued on a stream at that time, and by a program that holds no operator when it
creates and destroys one.  In a process of its own, where no other object lives."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes, torch
import paper_1408_0042_gb300 as plhr
lib, m, kp = plhr.load_library(), 12, 4
d = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")
G = [torch.diag(torch.arange(1.0, m + 1, dtype=torch.float64, device="cuda")) for _ in range(3)]
outs = [d(m), d(m, kp), d(kp, kp), d(kp), d(kp), d(2 * kp), d(4)]
outs[0] += 1.0
ptr = lambda t: ctypes.c_void_p(t.data_ptr())
Z = torch.randn(100000, 32, dtype=torch.float64, device="cuda")
s = torch.cuda.current_stream()

def operator():
    return plhr.Operator.laplacian((8, 8), 0.1)

def extract():
    assert lib.plhr_tharm_extract(m, kp, kp, *[ptr(g) for g in G], *[ptr(t) for t in outs], None, s.cuda_stream) == 0

def free():
    torch.cuda.synchronize()
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]

out = torch.empty((3, 32, 32), dtype=torch.float64, device="cuda")
def gram():
    nc, z, ld, cs = (ctypes.c_int * 1)(32), (ctypes.c_void_p * 1)(Z.data_ptr()), (ctypes.c_int64 * 1)(32), outs_cs
    assert lib.plhr_gram(plhr.GRAM_F64, Z.shape[0], 1, nc, z, ld, z, ld, None, None, 0.5, ptr(cs), ptr(out), s.cuda_stream) == 0
outs_cs = torch.ones(32, dtype=torch.float64, device="cuda")

op = operator()
extract()
gram()
torch.cuda.synchronize()
del op
base = free()
op = operator()
torch.cuda._sleep(400_000_000)
extract()
del op
assert not s.query()
queued = free()
gram()
extract()
held = free()
op = operator()
del op
after = free()
print(base - queued, base - held, base - after)
"""


def test_pool_is_given_back():
    import __graft_entry__
    __graft_entry__.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    queued, held, after = map(int, r.stdout.split())
    assert queued <= 0 and after <= 0
    assert held <= 64 << 20
