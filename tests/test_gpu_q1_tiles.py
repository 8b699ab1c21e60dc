"""The Q1 stiffness and mass products at the edges of their tiles: node counts
on both sides of a tile's extent and of a z segment, column counts that leave
part of a chunk or of a warp, padded blocks, unequal axes and a coefficient of
high contrast, against the element matrices summed in extended precision."""
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


def _products(dims, h, coeff, X):
    """Stiffness and mass products, element matrix by element matrix, in
    extended precision; X is n x nc with x fastest."""
    L = np.longdouble
    nx, ny, nz = dims
    nc = X.shape[1]
    P = np.zeros((nz + 2, ny + 2, nx + 2, nc), dtype=L)
    P[1:-1, 1:-1, 1:-1] = X.reshape(nz, ny, nx, nc)
    h = L(h)
    k = np.array([[1, -1], [-1, 1]], dtype=L) / h
    m = np.array([[2, 1], [1, 2]], dtype=L) * (h / 6)
    c = coeff.astype(L).reshape(nz + 1, ny + 1, nx + 1, 1)
    A, B = np.zeros_like(P), np.zeros_like(P)
    S = [slice(0, -1), slice(1, None)]
    for a in np.ndindex(2, 2, 2):
        for b in np.ndindex(2, 2, 2):
            kk = [k[a[i], b[i]] for i in range(3)]
            mm = [m[a[i], b[i]] for i in range(3)]
            src = P[S[b[0]], S[b[1]], S[b[2]]]
            A[S[a[0]], S[a[1]], S[a[2]]] += c * (kk[0] * mm[1] * mm[2] + mm[0] * kk[1] * mm[2]
                                                 + mm[0] * mm[1] * kk[2]) * src
            B[S[a[0]], S[a[1]], S[a[2]]] += mm[0] * mm[1] * mm[2] * src
    flat = lambda Y: Y[1:-1, 1:-1, 1:-1].reshape(-1, nc).astype(np.float64)
    return flat(A), flat(B)


# A row sums 8 elements x 8 corners of terms no larger than the largest result's
# scale: 64 x 2^-53 = 7.1e-15 of it, stated as 1e-14
@pytest.mark.parametrize("dims,nc,pad", [((1, 1, 1), 1, 0), ((2, 1, 3), 2, 1), ((15, 16, 17), 3, 0),
                                         ((31, 8, 2), 4, 3), ((7, 46, 5), 5, 0), ((3, 2, 257), 7, 1),
                                         ((18, 18, 18), 9, 0), ((49, 33, 20), 12, 4), ((9, 10, 11), 64, 0)])
def test_q1_products_at_tile_edges(plhr, dims, nc, pad):
    rng = np.random.default_rng(sum(dims) * 131 + nc)
    n, h = int(np.prod(dims)), 0.037
    X = rng.standard_normal((n, nc + pad))
    coeff = 10.0 ** rng.uniform(-3, 3, int(np.prod([d + 1 for d in dims])))
    Xt = torch.from_numpy(X).cuda()[:, :nc]
    for c in (None, coeff):
        ct = None if c is None else torch.from_numpy(c).cuda()
        opA = plhr.Operator._stencil(plhr.Q1_STIFF27, dims, h, field=ct)
        opB = plhr.Operator._stencil(plhr.Q1_MASS27, dims, h)
        ra, rb = _products(dims, h, np.ones_like(coeff) if c is None else c, X[:, :nc])
        pa, pb = opA.apply_pair(opB, Xt)
        for got, ref in ((opA.apply(Xt), ra), (opB.apply(Xt), rb), (pa, ra), (pb, rb)):
            assert np.abs(got.cpu().numpy() - ref).max() <= 1e-14 * np.abs(ref).max()
