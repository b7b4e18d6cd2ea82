"""The persistent RBF tiles of gram_rbf_tc.cu (symmetric for one vector, row sums for several): shares of
the tile order that start, end or change row tile anywhere, for one to a few hundred row tiles, in each
operand form (fp16 parts, TF32 parts with one and two atoms per row, one TF32 term), against the FP64
oracle.  Bounds: those of the existing tests of the same products (FP32 class 1e-5 of max |K v|; TF32:
2^-9 of the cross terms, entrywise below)."""
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


@pytest.mark.parametrize("n", [2, 127, 128, 129, 256, 257, 300, 385, 1100, 2177, 2300, 2431, 5000])
@pytest.mark.parametrize("p,spread", [(3, 1.0), (20, 1.0), (30, 1.0), (45, 1.0), (20, 9.0), (60, 9.0)])
def test_symmetric_tiles_cover_every_pair(K_, n, p, spread):
    """spread = 9: norms beyond 60, so the row factors do not fold and the TF32 parts are used."""
    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((n, p))
    X[0] *= spread
    gamma = 1.0 / p
    v = rng.standard_normal(n)
    with K_.Problem(X, np.zeros(n), "rbf", gamma, gram_store=0, rank0=2) as prob:
        u = prob.kmatvec(v, K_.PREC_FP32)
        t = prob.kmatvec(v, K_.PREC_TF32)
    ref = O.kmatvec(X, v, "rbf", gamma)
    # the exponent 2 g - n_i - n_j is rounded at 2^-24 of its parts once per MMA step (at most 24) and three
    # times outside: below 2^-19 (n_i + n_j) ln 2 of the entry
    Xc = (X - X.mean(0)) * np.sqrt(gamma / np.log(2.0))
    nr = np.linalg.norm(Xc, axis=1)
    K = O.gram(X, X, "rbf", gamma)
    far = (K * (np.add.outer(nr ** 2, nr ** 2) * (np.log(2.0) * 2.0 ** -19))) @ np.abs(v)
    assert np.all(np.abs(u - ref) <= 1e-5 * np.max(np.abs(ref)) + far)
    # one TF32 term: the exponent 2 xs_i . xs_j errs by at most 2 * 2^-11 * 2 |xs_i||xs_j|
    bound = (K * np.expm1(np.log(2.0) * 2.0 ** -9 * np.outer(nr, nr) * 1.1 + 1e-6)) @ np.abs(v) + 1e-5 * np.max(np.abs(ref)) + far
    assert np.all(np.abs(t - ref) <= bound)


@pytest.mark.parametrize("n", [2, 257, 1000, 1409, 1500, 1536, 1537, 1700, 2600])
@pytest.mark.parametrize("p,spread", [(1, 1.0), (8, 1.0), (9, 1.0), (32, 1.0), (20, 9.0)])
def test_multi_vector_tiles_cover_every_pair(K_, n, p, spread):
    """Two to eight vectors: row pairs of 256 rows shared out over the CTAs anywhere, partial sums per CTA;
    bound as above, and repeated products are bit-identical."""
    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((n, p))
    X[0] *= spread
    gamma = 1.0 / p
    K = O.gram(X, X, "rbf", gamma)
    Xc = (X - X.mean(0)) * np.sqrt(gamma / np.log(2.0))
    nr = np.linalg.norm(Xc, axis=1)
    with K_.Problem(X, np.zeros(n), "rbf", gamma, gram_store=0, rank0=2) as prob:
        for m in (2, 3, 5, 8):
            V = rng.standard_normal((n, m))
            U = prob.kmatvec(V, K_.PREC_FP32)
            ref = K @ V
            far = (K * (np.add.outer(nr ** 2, nr ** 2) * (np.log(2.0) * 2.0 ** -19))) @ np.abs(V)
            assert np.all(np.abs(U - ref) <= 1e-5 * np.max(np.abs(ref)) + far)
            np.testing.assert_array_equal(U, prob.kmatvec(V, K_.PREC_FP32))
