"""FP64-class RBF products of data with few values per feature (binary, or steps of a grid), up to the feature and norm
limits of the tensor-core form: the digits of such coordinates are the same in whole columns, so that the sums over
the features add up instead of averaging out.  Bound: 1e-12 of sum_j |K_ij v_j| per row, the one every FP64-class
product has to meet; the digit products' worst case (32 features, digits of magnitude 256) leaves errors of about
1e-13 in an exponent."""
import numpy as np
import pytest

from oracle import kqr_oracle as O
from paper_2510_07929_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DIGITS = 512.0 / 511.0 / 64.0   # 2^-6 (1 + 2^-9 + 2^-18 + ...): digits of -256 below the first


def data(kind, n, p, rng):
    if kind == "binary":
        x = rng.integers(0, 2, (n, p)) * 2.0 - 1.0
    elif kind == "digits":          # |x| = 29/32 - DIGITS, largest digits throughout, with both signs
        x = (29.0 / 32.0 - DIGITS) * (rng.integers(0, 2, (n, p)) * 2.0 - 1.0)
    elif kind == "equal":           # all features of a point the same
        x = np.repeat(rng.integers(-3, 4, (n, 1)) / 3.0, p, axis=1)
    else:                           # thirds of a grid
        x = rng.integers(-3, 4, (n, p)) / 3.0
    x[n // 2:] = -x[:n - n // 2]    # mean zero
    return x


@pytest.mark.parametrize("kind", ["binary", "digits", "equal", "grid"])
@pytest.mark.parametrize("p,reach", [(32, 27.9), (32, 3.0), (16, 27.9), (7, 12.0)])
def test_few_valued_features(kind, p, reach):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    n = 600
    X = data(kind, n, p, np.random.default_rng(p))
    scale = 1.0 if kind == "digits" and reach > 20 and p == 32 else np.sqrt(reach / np.max(np.sum(X * X, axis=1)))
    X = X * scale                   # log2(e) gamma |x|^2 up to reach with gamma = ln 2
    gamma = np.log(2.0)
    K = O.gram(X, X, "rbf", gamma)
    with kqr.Problem(X, np.zeros(n), "rbf", gamma, gram_store=0, rank0=2) as prob:
        for m in (1, 4):
            V = W.random_vectors(n, m, seed=m) if m > 1 else W.random_vectors(n, seed=1)
            U = prob.kmatvec(V, kqr.PREC_HIGH)
            err = np.abs(U - K @ V) / (K @ np.abs(V))
            assert err.max() <= 1e-12, (kind, p, reach, m, err.max())
