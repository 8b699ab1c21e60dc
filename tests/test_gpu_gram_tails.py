"""The fixed-point tensor-core Gram (csrc/gram_fx.cu) where the low digits of a
column's entries repeat, so that what is dropped or rounded adds up with one sign:
columns with one large entry and a tail below it, and columns of nearly constant
magnitude, against extended-precision products.

Units: an entry scaled by its column's 2^E in an SM's share has digits d_k of weight
2^-9(k+1), |d_k| <= 256; with a binade of room the largest entry is at least 2^-3, so an
absolute error counts 2^6 times as much against the product of the largest entries."""
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


def _error(plhr, Z):
    """Largest error of the three Grams of Z, U = Q = 2 Z over |x| |y|."""
    t = torch.from_numpy(Z).cuda()
    z = Z.astype(np.longdouble)
    G0 = z.T @ z
    norm = np.sqrt(np.diag(G0))
    worst = 0.0
    for form in (plhr.GRAM_F64, plhr.GRAM_DW):
        G = plhr.gram(form, t, 5.0 * t, sigma=3.0).cpu().numpy()
        for g, f in zip(G, (1, 4, 2)):
            worst = max(worst, float(np.max(np.abs(g / f - G0) / np.outer(norm, norm))))
    return worst


def test_products_of_outer_digits_are_kept(plhr):
    """A tail with the digits 1 and 5 only, both 255: its products are of levels 2, 6 and
    10, and those of level 6, 2^17 2^-72 a row, all have one sign.  Level 6 sums exactly
    (255 256 2 128 < 2^24); left are a rounding of half a unit of 2^-53 at the end of
    each of the 32 periods of 128 rows, 2^-43 of the largest entries and 2^-43.3 of the norms, and the few of the result."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    periods = 32
    Z = np.zeros((sms * 128 * periods, 2))
    share = Z.reshape(periods, sms, 128, 2)[:, 7]      # one SM's rows, in runs of 128
    share[...] = 255.0 * 2.0 ** -15 + 255.0 * 2.0 ** -51
    share[periods // 2, 0, 0] = share[periods // 2, 1, 1] = 1.0
    assert _error(plhr, Z) <= 2.0 ** -43


@pytest.mark.parametrize("tail", [1.9e-3, 1e-4, 1e-6])
def test_long_tails_stay_within_the_stated_bound(plhr, tail):
    """The stated bound: 2^-40 of the product of the largest entries for every 128 rows
    of an SM.  With tails below 2^-9 of the largest entry the levels above 4 are exact
    and the sum of levels 4 to 6 stays below 2^24 units of 2^-54; each of the 128 MMAs
    of a period may lose one unit, and the read-back half of one of 2^-53: 129 2^-54 2^6."""
    n = 300000
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(5)
    Z = np.full((n, 3), tail) * np.array([1.0, 0.73, 1.0])
    Z[:, 2] *= 0.8 + 0.2 * rng.uniform(size=n)
    Z[[7, 11, 7], [0, 1, 2]] = 1.0
    periods = -(-n // (128 * sms))
    assert _error(plhr, Z) <= periods * 2.0 ** -40


def test_nearly_constant_columns(plhr):
    """Entries whose leading three digits are large and of one sign, with low digits that
    differ: 2 d_0 d_2 + d_1^2 over 128 rows would pass 2^24 with a leading digit above
    2^7.  Below it level 2 is exact; level 3 passes 2^24 by at most 0.6 of it, in the last
    12 of its 32 MMAs of a period, which lose up to 2 units of 2^-45 each, and the sums are
    at least 128 2^-4: 3 2^-45."""
    rng = np.random.default_rng(9)
    n = 70000
    d = [np.full((n, 2), 255), np.array([250, 244]) + np.zeros((n, 2), dtype=int)]
    d += [rng.integers(249, 256, (n, 2))] + [rng.integers(-256, 256, (n, 2)) for _ in range(2)]
    X = sum(v.astype(np.int64) << (45 - 9 * k) for k, v in enumerate(d))
    assert _error(plhr, X * 2.0 ** -53) <= 2.0 ** -43
