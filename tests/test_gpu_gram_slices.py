"""The fixed-point tensor-core Gram of FP64 blocks (csrc/gram_fx.cu) at the
edges of its tiles, periods and number range, through plhr_gram, against
extended-precision products of the same inputs.

Bound: a dropped digit product is at most 2^16 2^-54 of a leading digit
product (five of them per row, which is at least 2^14 of those units for the
row of the largest entries), and the accumulator of levels 4 and 5 (with
levels 2 and 3 for columns of constant magnitude) rounds to 2^-24 of a sum
2^-27 below the leading one: 2^-46 |x| |y| covers a single row; the sums of
more rows are nearer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2.0 ** -46


@pytest.fixture(scope="module")
def plhr():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1408_0042_gb300 as p
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return p


def _families(n, m, seed, rows=None):
    """Z, AZ and Q = T U for a positive diagonal T (U^T Q symmetric); rows
    scales the rows of Z and AZ."""
    rng = np.random.default_rng(seed)
    Z, A = rng.standard_normal((n, m)), 50.0 * rng.standard_normal((n, m))
    if rows is not None:
        Z, A = Z * rows[:, None], A * rows[:, None]
    return Z, A, rng.uniform(0.5, 1.5, n)[:, None] * (A - 3.0 * Z)


def _error(plhr, Z, A, Q, form=0):
    cs = 1.0 / np.linalg.norm(Z, axis=0)
    t = lambda X: torch.from_numpy(np.ascontiguousarray(X)).cuda()
    G = plhr.gram(form, t(Z), t(A), None if Q is None else t(Q), sigma=3.0, colscale=t(cs)).cpu().numpy()
    z, a = Z.astype(np.longdouble) * cs, A.astype(np.longdouble) * cs
    u = a - 3.0 * z
    q = u if Q is None else Q.astype(np.longdouble) * cs
    ref = np.stack([z.T @ z, u.T @ q, q.T @ z])
    up = np.triu_indices(Z.shape[1])
    ref[1].T[up] = ref[1][up]          # the upper triangle of U^T Q, mirrored
    nz, nu, nq = (np.sqrt((x * x).sum(0)) for x in (z, u, q))
    scale = np.stack([np.outer(nz, nz), np.outer(nu, nq), np.outer(nq, nz)])
    return float(np.max(np.abs(G - ref) / scale))


@pytest.mark.parametrize("n,m,with_q", [(1, 1, True), (31, 16, True), (32, 17, False), (33, 64, True), (129, 15, True),
                                        (4864, 49, True), (4865, 48, False), (19457, 33, True)])
def test_tile_and_period_edges(plhr, n, m, with_q):
    """Rows around a step (32), one step or period per SM and one more; columns
    around the tile widths (multiples of 16)."""
    Z, A, Q = _families(n, m, n + m)
    assert _error(plhr, Z, A, Q if with_q else None) <= TOL
    assert _error(plhr, Z, A, Q if with_q else None, form=plhr.GRAM_DW) <= TOL


@pytest.mark.parametrize("rows", ["grow", "decay", "outlier"])
def test_exponents_follow_the_columns(plhr, rows):
    """Columns that grow by 2^60 from row to row of a CTA, that decay, and one
    with a single large entry: the integers are shifted to the new exponents."""
    n, m = 40000, 9
    x = np.linspace(-30.0, 30.0, n)
    scale = {"grow": np.exp2(x), "decay": np.exp2(-x), "outlier": np.where(np.arange(n) == 31007, 1e12, 1.0)}[rows]
    assert _error(plhr, *_families(n, m, 5, scale)) <= TOL


def test_constant_columns_over_many_periods(plhr):
    """Entries just below a power of two in every row: the largest sums the
    accumulators and the 64-bit integers meet (read back by the conversion
    instruction, written out in several rounds).  All entries are equal, so the
    Grams are n times one product."""
    n, m = 700001, 3
    c = np.array([1.0 - 2.0 ** -53, 1.9990234375, 3.999999])
    Z = torch.from_numpy(c).cuda().expand(n, m).contiguous()
    G = plhr.gram(plhr.GRAM_F64, Z, 5.0 * Z, sigma=3.0, colscale=torch.full((m,), n ** -0.5, dtype=torch.float64).cuda())
    want = np.outer(c, c)
    assert np.max(np.abs(G.cpu().numpy() / np.stack([want, 4.0 * want, 2.0 * want]) - 1.0)) <= TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_columns_stay_in_their_rows(plhr, bad):
    """A NaN or Inf in one column of Z makes the entries of that column
    non-finite, as in the plain FP64 form, and no others."""
    n, m, j = 5000, 20, 7
    Z, A, Q = _families(n, m, 3)
    Z[1234, j] = bad
    t = lambda X: torch.from_numpy(X).cuda()
    G = plhr.gram(plhr.GRAM_F64, t(Z), t(A), t(Q), sigma=3.0).cpu().numpy()
    hit = np.zeros((3, m, m), dtype=bool)
    hit[0, j, :] = hit[0, :, j] = hit[1, j, j:] = hit[1, j:, j] = hit[2, :, j] = True
    # in the 4 x 4 tiles on the diagonal the plain form keeps U_j^T Q_i of the two
    # entries (i, j), (j, i) of U^T Q, not the upper one: either may be the bad one
    free = np.zeros((3, m, m), dtype=bool)
    free[1, j - j % 4:j, j] = free[1, j, j - j % 4:j] = True
    assert np.array_equal(~np.isfinite(G) & ~free, hit & ~free)
    Z[1234, j] = 0.0
    ref = np.stack([Z.T @ Z, (A - 3.0 * Z).T @ Q, Q.T @ Z])
    ok = ~hit & ~free
    ok[1] &= np.triu(np.ones((m, m), dtype=bool))
    assert np.allclose(G[ok], ref[ok], rtol=1e-12, atol=1e-9)
