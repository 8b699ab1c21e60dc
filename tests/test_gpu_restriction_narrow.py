"""The restriction that forms four coarse lines per CTA, in FP32 and in double-word
arithmetic, on lines of few values (short lines, few columns), against the FP64 V-cycle
of the same operator, which has transfers of its own."""
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


# the tolerances of the FP32 and double-word V-cycles against the FP64 oracle
@pytest.mark.parametrize("dims", [(16, 64, 64), (4, 52, 56), (20, 60, 52), (32, 12, 20), (8, 4, 4)])
@pytest.mark.parametrize("nc", [1, 3, 4, 8])
def test_narrow_lines(plhr, dims, nc):
    T = plhr.AVMG(plhr.Operator.laplacian(dims, 1.0 / 65), 200.0, levels=3, transfer=1, coarse=1)
    R = torch.from_numpy(np.random.default_rng(nc).standard_normal((int(np.prod(dims)), nc))).cuda()
    W = T.apply(R)
    top = float(W.abs().max())
    assert float((T.apply_dw(R) - W).abs().max()) <= 1e-12 * top
    assert float((T.apply_f32(R.float()).double() - W).abs().max()) <= 2e-5 * top
