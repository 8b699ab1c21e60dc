"""The Grams of FP64 blocks whose columns lie at the ends of the number range, where the
fixed-point form (csrc/gram_fx.cu) hands the launch to the FP64 kernel: columns whose
scale in colscale undoes it, and products of a column near the upper end with one near the lower."""
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


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


# the columns of all families times 2^power and colscale times 2^-power, exactly: the
# Grams are those of power 0 to the rounding of sums of n / 304 products per block and 304
# blocks, below 2^-46 |x| |y|
@pytest.mark.parametrize("power", [-896, -950, -1000, 1008])
@pytest.mark.parametrize("n,with_q", [(3000, True), (40001, False)])
def test_column_scales_undo_the_range(plhr, power, n, with_q):
    rng = np.random.default_rng(power + n)
    m, j = 19, 11
    Z, A = rng.uniform(0.5, 1.0, (n, m)), 50.0 * rng.uniform(0.5, 1.0, (n, m))
    Q = rng.uniform(0.5, 1.5, n)[:, None] * (A - 3.0 * Z)
    cs = 1.0 / np.linalg.norm(Z, axis=0)
    z, u = Z.astype(np.longdouble) * cs, (A.astype(np.longdouble) - 3.0 * Z) * cs
    q = Q.astype(np.longdouble) * cs if with_q else u
    for X in (Z, A, Q):
        X[:, j] *= 2.0 ** power
    cs[j] *= 2.0 ** -power
    for form in (plhr.GRAM_F64, plhr.GRAM_DW):
        G = plhr.gram(form, _dev(Z), _dev(A), _dev(Q) if with_q else None, sigma=3.0, colscale=_dev(cs)).cpu().numpy()
        for k, (g, x, y) in enumerate(zip(G, (z, u, q), (z, q, z))):
            ref = x.T @ y
            if k == 1:             # the upper triangle of U^T Q, mirrored
                ref = np.triu(ref) + np.triu(ref, 1).T
            norm = np.outer(np.sqrt((x * x).sum(0)), np.sqrt((y * y).sum(0)))
            assert float(np.max(np.abs(g - ref) / norm)) <= 2.0 ** -46


def test_products_across_the_range(plhr):
    """Without column scales: the squares leave the range, the products across do not."""
    rng = np.random.default_rng(2)
    n = 2000
    Z = rng.uniform(0.5, 1.0, (n, 2))
    ref = float(Z[:, 0].astype(np.longdouble) @ Z[:, 1].astype(np.longdouble))
    Z = Z * np.array([2.0 ** 1021, 2.0 ** -1000])
    G = plhr.gram(plhr.GRAM_F64, _dev(Z), _dev(0.5 * Z), sigma=3.0).cpu().numpy()
    for g, f in zip(G, (1.0, 6.25, -2.5)):
        assert abs(g[0, 1] / (f * ref * 2.0 ** 21) - 1.0) <= 2.0 ** -46
        assert np.isinf(g[0, 0]) and abs(g[1, 1]) < 2.0 ** -1000


def test_large_column_scales_of_null_columns(plhr):
    """Columns of zeros with the column scale 1e300 (one over a floored norm), their images not zero:
    only the products of two such images leave the range."""
    rng = np.random.default_rng(4)
    n, m, null = 500, 18, [3, 4, 17]
    Z, A = rng.uniform(0.5, 1.0, (n, m)), rng.uniform(0.5, 1.0, (n, m))
    Z[:, null] = 0.0
    A[:250, 3] = A[250:, 4] = 0.0                        # the images of 3 and 4 share no row
    cs = 1.0 / np.maximum(np.linalg.norm(Z, axis=0), 1e-300)
    G = plhr.gram(plhr.GRAM_F64, _dev(Z), _dev(A), sigma=3.0, colscale=_dev(cs)).cpu().numpy()
    z, u = Z.astype(np.longdouble) * cs, (A.astype(np.longdouble) - 3.0 * Z) * cs
    for g, x, y in zip(G, (z, u, u), (z, u, z)):
        ref = x.T @ y
        out = np.abs(ref) > np.longdouble(2.0) ** 1023
        norm = np.outer(np.sqrt((x * x).sum(0)), np.sqrt((y * y).sum(0)))
        assert np.isinf(g[out]).all() and np.isfinite(g[~out]).all()
        assert (np.abs(g - ref)[~out] <= 2.0 ** -46 * norm[~out]).all()
    assert G[1, 3, 4] == 0.0
