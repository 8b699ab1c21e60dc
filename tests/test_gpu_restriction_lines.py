"""The restriction that forms four coarse lines per CTA (large 3D levels, linear
transfers), in FP32 and in double-word arithmetic: coarse line counts that leave
half a group, column counts with and without 16-byte alignment, against the same
V-cycle column by column, which is below the size that takes it."""
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


# A V-cycle is about 20 sums after one another, each correct to a few units of its
# arithmetic (2^-24, 2^-46): 64 units of the largest entry
@pytest.mark.parametrize("dims,levels", [((32, 52, 50), 2), ((36, 60, 60), 3), ((30, 54, 46), 2)])
@pytest.mark.parametrize("nc", [20, 17])
def test_vcycle_equals_its_columns(plhr, dims, levels, nc):
    T = plhr.AVMG(plhr.Operator.laplacian(dims, 1.0 / (max(dims) + 1)), 200.0, levels=levels, transfer=1, coarse=1)
    R = torch.from_numpy(np.random.default_rng(7).standard_normal((int(np.prod(dims)), nc))).cuda()
    for apply, block, unit in ((T.apply_f32, R.float(), 2.0**-24), (T.apply_dw, R, 2.0**-46)):
        W = apply(block)
        for c in range(0, nc, 3):
            w = apply(block[:, c:c + 1].contiguous())
            assert float((W[:, c:c + 1] - w).abs().max()) <= 64 * unit * float(w.abs().max())
