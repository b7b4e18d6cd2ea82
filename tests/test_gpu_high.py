"""FP64-class RBF products on the tensor cores (gram_high_tc.cu) against the FP64 oracle, at the edges of its
128 x 64 tiles, of its digit layouts (p = 16 | 17, 32 | 33) and of the norms it accepts.  Bound: 1e-12 of
sum_j |K_ij v_j| per row, the one every FP64-class product has to meet."""
import numpy as np
import pytest

from oracle import kqr_oracle as O
from paper_2510_07929_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K_():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    return kqr


def check(K_, X, gamma, ms, seed=0, **opts):
    n = X.shape[0]
    K = O.gram(X, X, "rbf", gamma)
    with K_.Problem(X, np.zeros(n), "rbf", gamma, gram_store=0, **opts) as prob:
        for m in ms:
            V = W.random_vectors(n, m, seed=seed + m) if m > 1 else W.random_vectors(n, seed=seed + 1)
            U = prob.kmatvec(V, K_.PREC_HIGH)
            err = np.abs(U - K @ V) / (np.abs(K) @ np.abs(V))
            assert err.max() <= 1e-12, (n, X.shape[1], m, err.max())


@pytest.mark.parametrize("n,p", [(2, 1), (63, 2), (64, 16), (65, 17), (127, 8), (128, 32), (129, 31), (500, 15),
                                 (1000, 20), (1291, 5)])
def test_high_products_match_oracle(K_, n, p):
    X = np.random.default_rng(n).standard_normal((n, p))
    check(K_, X, 1.0 / p, (1, 2, 3, 8), seed=n)


@pytest.mark.parametrize("p,reach", [(1, 26.9), (3, 26.9), (32, 26.9), (3, 40.0), (33, 5.0)])
def test_high_products_at_the_norm_limit(K_, p, reach):
    """Largest log2(e) gamma |x - mean|^2 just inside the tensor path's limit, and beyond it (other kernels);
    repeated and nearly repeated points, whose exponent is zero up to rounding."""
    rng = np.random.default_rng(p)
    X = rng.standard_normal((400, p))
    X[1], X[2] = X[0], X[0] + 1e-9
    X[200:] = -X[:200]                       # mean zero
    X *= np.sqrt(reach / (np.max(np.sum(X * X, axis=1)) / np.log(2.0)))
    check(K_, X, 1.0, (1, 4))


def test_high_multi_vector_products_are_reproducible(K_):
    wl = W.rbf_small(n=3001, p=8)
    V = W.random_vectors(wl.n, 8, seed=3)
    with K_.Problem(wl.X, wl.y, "rbf", wl.gamma) as prob:
        a = prob.kmatvec(V, K_.PREC_HIGH)
        b = prob.kmatvec(V, K_.PREC_HIGH)
    np.testing.assert_array_equal(a, b)
