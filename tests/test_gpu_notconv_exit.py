"""What a solve that stops at maxit returns when its block has dependent columns: the
final Rayleigh-Ritz has no Cholesky factor to work with, and the outputs are the
block's own columns, normalised and in order, with their Rayleigh quotients."""
import numpy as np
import pytest

from oracle import operators as oops

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


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_dependent_columns_come_back_as_they_are(plhr, precision):
    """Two equal columns of norm 1 and a third one of norm 2: every product of the
    Gram is exact, so its second pivot is exactly zero."""
    n, h, sigma = 256, 1 / 17, 300.0
    V = np.zeros((n, 3))
    V[[3, 50, 77, 200], 0] = V[[3, 50, 77, 200], 1] = 0.5
    V[[9, 120, 121, 240], 2] = 1.0
    A = oops.laplacian_dirichlet((16, 16), h).toarray()
    unit = V / np.linalg.norm(V, axis=0)
    rq = np.einsum("ij,ij->j", unit, A @ unit)
    order = sorted(range(3), key=lambda j: abs(rq[j] - sigma))
    op = plhr.Operator.laplacian((16, 16), h)
    vals, vecs, info = plhr.solve(op, sigma, 3, tol=1e-10, maxit=0, guard=0, v_init=torch.from_numpy(V).cuda(),
                                  precision=plhr.PRECISION_F64 if precision == "f64" else plhr.PRECISION_MIXED)
    assert info["status"] == plhr.PLHR_ENOTCONV
    # a few units of the largest of five terms of about 4 / h^2 each
    assert np.abs(vals - rq[order]).max() <= 1e-14 * 8 / h ** 2
    assert np.array_equal(vecs.cpu().numpy(), unit[:, order])
    R = A @ unit - unit * rq
    rel = np.linalg.norm(R, axis=0) / np.maximum(np.abs(rq), 1.0)
    assert abs(info["max_rel_residual"] - rel.max()) <= 1e-12 * rel.max()
