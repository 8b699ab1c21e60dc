"""Stencil products whose neighbour sums run on the integer pipes (blocks of at
least 500,000 elements): every entry against extended precision with a bound
from the seven terms it is made of, over values of any size mixed, zeros of both
signs, subnormals and values whose sums would leave the integer form, infinities
and NaN; and the FP64 V-cycle on such a block against the same columns one by one."""
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


def _terms(dims, X, periodic):
    """(2d x_c - neighbours, largest term) with X of shape dims reversed + columns."""
    L = X.astype(np.longdouble)
    d = len(dims)
    s, top = 2 * d * L, np.abs(X)
    for ax in range(d):
        for k in (1, -1):
            nb = np.roll(L, k, axis=ax)
            if not periodic:
                edge = [slice(None)] * L.ndim
                edge[ax] = 0 if k == 1 else -1
                nb[tuple(edge)] = 0
            s = s - nb
            top = np.maximum(top, np.abs(nb).astype(np.float64))
    return s, top


def _values(kind, shape, rng):
    v = rng.standard_normal(shape)
    if kind == "plain":
        return v
    if kind == "wide":       # neighbours of any relative size, beyond the 64 bits of the sum
        return v * 2.0 ** rng.integers(-90, 90, shape)
    if kind == "smooth":     # cancellation: neighbours agree to about 2^-20
        return 1.0 + v * 1e-6
    if kind == "small":      # below the range of the integer form, down to subnormals
        return v * 2.0 ** rng.integers(-1070, -380, shape).astype(np.float64)
    v *= 2.0 ** rng.integers(-460, 460, shape)   # around the upper end, zeros of both signs
    v[rng.uniform(size=shape) < 0.4] = 0.0
    v[rng.uniform(size=shape) < 0.2] = -0.0
    return v


# Truncation: 12 units (6 neighbours and 6 x_c) of 2^-6 of the largest term's last
# place, 2^-52 of it: 0.375 x 2^-53; rounding of a sum of at most 12 times the
# largest term, and of its product with 1/h^2 = 4: 12 x 2^-53 each.  In FP64 (values
# outside the integer form's range) the partial sums are at most 2, 2, 4, 2, 6, 12
# times the term: with the product 40 x 2^-53, the bound; and 2^-1072 for
# subnormal results.
@pytest.mark.parametrize("kind", ["plain", "wide", "smooth", "small", "zeros"])
@pytest.mark.parametrize("dims,nc,pad,periodic", [((67, 43, 29), 7, 0, False), ((131, 1, 3), 1300, 1, False),
                                                  ((23, 2, 5000), 3, 2, True), ((1021, 517), 1, 0, False),
                                                  ((300, 301), 8, 3, True)])
def test_products_entry_by_entry(plhr, kind, dims, nc, pad, periodic):
    rng = np.random.default_rng(len(kind) * 1000 + sum(dims) + nc)
    X = _values(kind, tuple(reversed(dims)) + (nc + pad,), rng)
    op = plhr.Operator.laplacian(dims, 0.5, periodic=periodic)
    Y = op.apply(torch.from_numpy(X.reshape(-1, nc + pad)).cuda()[:, :nc]).cpu().numpy()
    s, top = _terms(dims, X[..., :nc], periodic)
    err = np.abs(Y.reshape(s.shape).astype(np.longdouble) - 4 * s)
    assert (err <= 4 * 40 * 2.0**-53 * top.astype(np.longdouble) + 2.0**-1072).all()


def test_infinities_and_nan_reach_their_neighbours_only(plhr):
    dims, nc = (40, 33, 25), 16
    X = np.random.default_rng(3).standard_normal((25, 33, 40, nc))
    X[7, 9, 11, 3] = np.inf
    X[20, 0, 39, 5] = np.nan
    Y = plhr.Operator.laplacian(dims, 1.0).apply(torch.from_numpy(X.reshape(-1, nc)).cuda()).cpu().numpy()
    with np.errstate(invalid="ignore"):
        s, _ = _terms(dims, X, False)
    Y = Y.reshape(s.shape)
    bad = ~np.isfinite(s.astype(np.float64))
    assert (np.isfinite(Y) == ~bad).all()
    assert Y[7, 9, 11, 3] == np.inf and Y[7, 9, 12, 3] == -np.inf and np.isnan(Y[20, 0, 39, 5])


# each sweep's rounding is a few 2^-53 of the iterate; about 20 kernels follow one
# another: 1e-13 of the largest entry
@pytest.mark.parametrize("kw", [{}, {"indefinite": True}])
@pytest.mark.parametrize("dims,levels,nc,sigma", [((64, 48, 32), 3, 6, 150.0), ((512, 256), 3, 5, 2000.0)])
def test_vcycle_equals_its_columns(plhr, dims, levels, nc, sigma, kw):
    T = plhr.AVMG(plhr.Operator.laplacian(dims, 1.0 / (max(dims) + 1)), sigma, levels=levels, transfer=1, coarse=1, **kw)
    n = int(np.prod(dims))
    R = torch.from_numpy(np.random.default_rng(11).standard_normal((n, nc))).cuda()
    W = T.apply(R)
    for c in range(nc):
        w = T.apply(R[:, c:c + 1].contiguous())
        assert float((W[:, c:c + 1] - w).abs().max()) <= 1e-13 * float(w.abs().max())
