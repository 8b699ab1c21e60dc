"""plhr_eigvec_adjoint returns with its stream idle: grad may be read from any stream, or
V and G reused, right after the call, converged or not."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plhr():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1408_0042_gb300 as p
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return p


@pytest.mark.parametrize("tol,maxit,status", [(1e-3, 500, "PLHR_OK"), (1e-12, 1, "PLHR_ENOTCONV")])
def test_stream_is_idle_on_return(plhr, tol, maxit, status):
    dims, k = (96, 96, 96), 16
    n = int(np.prod(dims))
    pot = torch.zeros(n, dtype=torch.float64, device="cuda")
    op = plhr.Operator.hamiltonian(dims, 1.0, pot)
    V = torch.zeros((n, k), dtype=torch.float64, device="cuda")
    V[torch.arange(k) * 1000, torch.arange(k)] = 1.0
    G = torch.from_numpy(np.random.default_rng(1).standard_normal((n, k))).cuda()
    lam = np.full(k, -1.0) + 0.01 * np.arange(k)      # below the spectrum: a definite system
    g = torch.empty(n, dtype=torch.float64, device="cuda")
    s, its = torch.cuda.Stream(), ctypes.c_int(0)
    torch.cuda.synchronize()
    st = plhr.load_library().plhr_eigvec_adjoint(
        op._h, None, k, lam.ctypes.data, ctypes.c_void_p(V.data_ptr()), k, ctypes.c_void_p(G.data_ptr()), k, tol,
        maxit, ctypes.c_void_p(g.data_ptr()), ctypes.byref(its), s.cuda_stream)
    assert s.query()
    assert st == getattr(plhr, status)
