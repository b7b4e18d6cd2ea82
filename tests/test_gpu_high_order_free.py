"""One-vector FP64-class RBF products: the same bits in every run with default options, and sums that lose nothing by
it, also for rows far below the largest ones.  Bound: 1e-12 of sum_j |K_ij v_j| per row, the one every FP64-class
product has to meet."""
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


@pytest.mark.parametrize("n,p", [(129, 3), (2000, 10), (9001, 20), (20011, 32)])
def test_one_vector_products_are_reproducible(K_, n, p):
    wl = W.rbf_mid(n=n, p=p, seed=n)
    with K_.Problem(wl.X, wl.y, "rbf", wl.gamma, rank0=2, gram_store=0) as prob:
        for v in (W.random_vectors(n, seed=1), np.exp(12 * W.random_vectors(n, seed=2))):
            a = prob.kmatvec(v, K_.PREC_HIGH)
            for _ in range(6):
                np.testing.assert_array_equal(a, prob.kmatvec(v, K_.PREC_HIGH))


# Two clusters whose entries across are 2^-reach, vectors that are zero on one of them (whole rows are then sums of
# such entries) or spread over 2^+-spread, and scaled as a whole.
@pytest.mark.parametrize("reach,spread,scale", [(40.0, 0, 1.0), (90.0, 0, 1.0), (90.0, 30, 1.0), (60.0, 0, 1e-25),
                                                (60.0, 10, 1e30), (5.0, 60, 1.0)])
def test_small_rows_keep_their_precision(K_, reach, spread, scale):
    rng = np.random.default_rng(int(reach))
    n, p = 700, 4
    X = 0.02 * rng.standard_normal((n, p))
    X[::2, 0] += 0.5 * np.sqrt(reach * np.log(2.0))
    X[1::2, 0] -= 0.5 * np.sqrt(reach * np.log(2.0))
    K = O.gram(X, X, "rbf", 1.0)
    v = scale * rng.standard_normal(n) * 2.0 ** rng.uniform(-spread, spread, n)
    if spread == 0:
        v[::2] = 0.0
    with K_.Problem(X, np.zeros(n), "rbf", 1.0, rank0=2, gram_store=0) as prob:
        u = prob.kmatvec(v, K_.PREC_HIGH)
    assert np.all(np.abs(u - K @ v) <= 1e-12 * (K @ np.abs(v)))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_vectors_give_nan(K_, bad):
    X = np.random.default_rng(0).standard_normal((300, 5))
    v = np.ones(300)
    with K_.Problem(X, np.zeros(300), "rbf", 0.1, rank0=2, gram_store=0) as prob:
        v[17] = bad
        assert not np.isfinite(prob.kmatvec(v, K_.PREC_HIGH)).any()
        v[17] = 0.0
        u = prob.kmatvec(v, K_.PREC_HIGH)      # nothing is left over from the product before
        K = O.gram(X, X, "rbf", 0.1)
        assert np.all(np.abs(u - K @ v) <= 1e-12 * (K @ np.abs(v)))
