"""Batched products of finite data whose squared norms leave the FP32 range: exponents that are inf - inf are NaN, and
a NaN has to reach the result rather than turn into a number.  The default form and the one that passes the Gram tile
through shared memory (which rounds with cvt.rna.tf32) agree on where; ordinary data beside it is right."""
import numpy as np
import pytest

from oracle import kqr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big", [1e19, 3e20, 1e60, 1e200])
@pytest.mark.parametrize("sizes,p,m", [((200, 130, 300), 8, 16), ((64, 500), 3, 5)])
def test_overflowing_norms_give_nan(big, sizes, p, m):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    rng = np.random.default_rng(p)
    Xs = [rng.random((n, p)) for n in sizes]
    Xs[1] = Xs[1] * big
    V = rng.standard_normal((sum(sizes), m))
    with kqr.Batch(Xs, 1.0 / p) as bt:
        U = bt.kmatmul(V)
    with kqr.Batch(Xs, 1.0 / p, p_in_smem=True) as bt:
        R = bt.kmatmul(V)
    np.testing.assert_array_equal(np.isnan(U), np.isnan(R))
    lo, hi = sizes[0], sizes[0] + sizes[1]
    if big >= 3e20:
        assert np.isnan(U[lo:hi]).any()
    assert np.isfinite(U[:lo]).all() and np.isfinite(U[hi:]).all()
    K = O.gram(Xs[0], Xs[0], "rbf", 1.0 / p)
    assert np.all(np.abs(U[:lo] - K @ V[:lo]) <= 2.0 ** -8 * (K @ np.abs(V[:lo])) + 1e-30)
