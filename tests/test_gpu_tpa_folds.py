"""The folded axis transforms of the TPA preconditioner (csrc/spectral.cu) at
axis sizes where the parity classes are empty, of one point, odd or padded, at
the largest size, and at column counts around the tile of 32 elements, against
the oracle's FFT / sine-transform form."""
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


# double-word multiply-adds: about 2^-46 of the sum of |terms| per product, at
# most 144 terms of orthonormal rows and 6 products: 6 sqrt(144) 2^-46 = 1e-12
TOL = 1e-12


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("dims,cols", [((1, 2, 3), 1), ((4, 5, 6), 31), ((7, 8, 9), 33), ((10, 12, 14), 3),
                                       ((64, 2, 17), 10), ((144, 3, 4), 2), ((3, 144, 2), 5), ((2, 3, 144), 1),
                                       ((144, 143), 3), ((2, 96), 32), ((1, 1), 4)])
def test_tpa_matches_the_oracle(plhr, dims, cols, periodic):
    from oracle import spectral
    rng = np.random.default_rng(sum(dims) + cols)
    n = int(np.prod(dims))
    R = rng.standard_normal((n, cols))
    pot = torch.from_numpy(rng.uniform(-2.0, 0.0, n)).cuda()
    A = plhr.Operator.hamiltonian(dims, 0.7, pot, periodic)
    T = plhr.TPA(A, -0.5, 1.3)
    got = T.apply(torch.from_numpy(R).cuda()).cpu().numpy()
    ref = spectral.TPA(dims, 0.7, 1.3, periodic)(R)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()
