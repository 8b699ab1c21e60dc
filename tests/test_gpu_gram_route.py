"""Which kernel formed the Grams of an FP64 block: for the columns (1, 0, e, e, ..) and
(0, 1, e, e, ..) with e = 2^-70 the fixed-point form holds e as 0 and their product is 0,
the FP64 kernel gives 30 e^2 (32 rows: one share).  Finite columns take the fixed-point
form; a column of the same call with Inf, NaN or nothing but tiny values sends it to the
FP64 kernel."""
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


@pytest.mark.parametrize("other,fixed", [(1.0, True), (0.0, True), (-2.0 ** 600, True), (2.0 ** -890, True),
                                         (np.inf, False), (np.nan, False), (2.0 ** -950, False), (5e-324, False)])
@pytest.mark.parametrize("m", [3, 40])
def test_route(plhr, other, fixed, m):
    n, e = 32, 2.0 ** -70
    Z = np.ones((n, m))
    Z[:, 0] = Z[:, 1] = e
    Z[0, 0], Z[1, 0], Z[0, 1], Z[1, 1] = 1.0, 0.0, 0.0, 1.0
    Z[:, m - 1] = 0.0
    Z[17, m - 1] = other
    t = torch.from_numpy(Z).cuda()
    for form in (plhr.GRAM_F64, plhr.GRAM_DW):
        G = plhr.gram(form, t, 2.0 * t, sigma=1.0).cpu().numpy()
        assert (G[:, 0, 1] == (0.0 if fixed else 30.0 * e * e)).all()
