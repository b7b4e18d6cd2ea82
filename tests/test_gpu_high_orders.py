"""FP64-class RBF products of one and of several vectors in turn on one handle, against the FP64 oracle: the two
kinds keep work lists and partial sums of their own, in whichever order they are first asked for.  Bound: 1e-12 of
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


@pytest.mark.parametrize("order", [(8, 1, 8), (2, 1, 8, 1, 2), (3, 1, 5), (1, 2, 8, 1, 4), (4, 1, 1, 7)])
@pytest.mark.parametrize("n", [300, 2000])
def test_products_in_any_order(K_, n, order):
    p = 6
    X = np.random.default_rng(n).standard_normal((n, p))
    K = O.gram(X, X, "rbf", 0.2)
    with K_.Problem(X, np.zeros(n), "rbf", 0.2, gram_store=0, rank0=2) as prob:
        for k, m in enumerate(order):
            V = W.random_vectors(n, m, seed=7 * k + m) if m > 1 else W.random_vectors(n, seed=7 * k + 1)
            U = prob.kmatvec(V, K_.PREC_HIGH)
            err = np.abs(U - K @ V) / (np.abs(K) @ np.abs(V))
            assert err.max() <= 1e-12, (order, k, m, err.max())


def test_grid_with_fp32_cg(K_):
    """A grid whose CG runs in FP32: its first FP64-class products are the columns' gradients, several or one at a
    time.  Nine columns, so that a full round of products has a group of eight and one alone."""
    wl = W.rbf_small(n=700, p=8, seed=5)
    gamma = 2.0
    K = O.gram(wl.X, wl.X, "rbf", gamma)
    taus = np.array([0.1, 0.5, 0.9] * 3)
    lams = np.repeat([1e-2, 3e-2, 1e-1], 3)
    with K_.Problem(wl.X, wl.y, "rbf", gamma, cg_high=0, time_limit_s=120.0) as prob:
        for _ in range(2):      # the second time both work lists are there
            alpha, beta, kkt, status, _ = prob.solve_grid(taus, lams, tol=1e-6)
            assert np.all(status == K_.OK), status
            for c in range(len(taus)):
                a = O.project_feasible(alpha[:, c], taus[c])
                ref = O.solve_dense(K, wl.y, taus[c], lams[c], tol=1e-9)
                d, d_ref = (O.dual_objective(v, K @ v, wl.y, lams[c]) for v in (a, ref["alpha"]))
                assert abs(d - d_ref) <= 1e-6 * (1 + abs(d_ref)), (taus[c], lams[c], d, d_ref)
