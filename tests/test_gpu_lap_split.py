"""The FP32-class Laplacian product with some features on the integer pipe (gram_f32_sym.cu): feature counts
around the split, tile edges, and data whose fixed-point grid is too coarse for it (an outlier; the FP32 form
then), against the FP64 oracle.  Bound: that of the existing tests of the product, 1e-5 of max |K v|, and the
grid's, 2^-20 ln 2 of each entry."""
import numpy as np
import pytest

from oracle import kqr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 127, 129, 300, 1500])
@pytest.mark.parametrize("p,gamma,outlier", [(1, 1.0, 0.0), (11, 0.1, 0.0), (12, 0.1, 0.0), (13, 0.2, 0.0), (14, 1.0, 0.0),
                                             (16, 0.1, 0.0), (17, 0.05, 300.0), (50, 0.02, 0.0), (64, 0.02, 50.0)])
def test_split_laplacian_matches_fp64(n, p, gamma, outlier):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((n, p))
    X[0] += outlier
    v = rng.standard_normal(n)
    with kqr.Problem(X, np.zeros(n), "laplacian", gamma, gram_store=0, rank0=2) as prob:
        u = prob.kmatvec(v, kqr.PREC_FP32)
    K = O.gram(X, X, "laplacian", gamma)
    ref = K @ v
    assert np.all(np.abs(u - ref) <= 1e-5 * np.max(np.abs(ref)) + 2.0 ** -20 * np.log(2.0) * (K @ np.abs(v)))
