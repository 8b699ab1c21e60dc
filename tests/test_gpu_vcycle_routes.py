"""Routes of the FP64 V-cycle that are taken by size only: polynomial levels whose
neighbour sums run on the integer pipes (a level of at least 500,000 elements), and line
transfers cut into several segments and column groups (more than 63 coarse points,
more than 32 columns), against the same V-cycle column by column, which is below those
sizes."""
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


def _equal(T, n, nc):
    R = torch.from_numpy(np.random.default_rng(n + nc).standard_normal((n, nc))).cuda()
    W = T.apply(R)
    for c in range(0, nc, max(1, nc // 8)):
        w = T.apply(R[:, c:c + 1].contiguous())
        # about 20 kernels after one another, each with a few 2^-53 of the iterate
        assert float((W[:, c:c + 1] - w).abs().max()) <= 1e-13 * float(w.abs().max())


@pytest.mark.parametrize("nu", [1, 2])
@pytest.mark.parametrize("dims,nc", [((64, 48, 32), 6), ((512, 256), 5)])
def test_polynomial_levels(plhr, dims, nc, nu):
    """sqrt(sigma) h = 0.7 on the finest level, above the 0.63 from which it is polynomial."""
    h = 1.0 / (max(dims) + 1)
    T = plhr.AVMG(plhr.Operator.laplacian(dims, h), 0.49 / h ** 2, levels=3, nu=nu, transfer=1, coarse=1)
    _equal(T, int(np.prod(dims)), nc)


@pytest.mark.parametrize("transfer", [0, 1])
@pytest.mark.parametrize("dims,nc", [((256, 24), 33), ((256, 24), 70), ((160, 8, 12), 33), ((128, 8, 8), 32)])
def test_transfers_in_segments_and_column_groups(plhr, dims, nc, transfer):
    h = 1.0 / (max(dims) + 1)
    T = plhr.AVMG(plhr.Operator.laplacian(dims, h), 150.0, levels=2, transfer=transfer, coarse=1)
    _equal(T, int(np.prod(dims)), nc)
