"""The batched product's 128-column steps: items of one, two and more steps in any order on a CTA (more items
than CTAs), result columns around the 16-column steps of its second contraction, against FP64.  Bound: the one
of the batched products, 2^-8 of sum_j K_ij |V_jc| entrywise (TF32 coordinates, Gram entries and vectors)."""
import numpy as np
import pytest

from oracle import kqr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,p,m", [([1, 127, 128, 129, 255, 256, 257, 384, 385], 8, 16),
                                       ([100, 200, 300] * 120, 5, 17), ([40] * 400, 2, 1), ([700, 60] * 80, 31, 48),
                                       ([130] * 153 + [1000], 8, 64)])
def test_batch_steps_match_fp64(sizes, p, m):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    rng = np.random.default_rng(len(sizes) + p)
    Xs = [rng.random((n, p)) for n in sizes]
    V = rng.standard_normal((sum(sizes), m))
    with kqr.Batch(Xs, 1.0 / p) as bt:
        U = bt.kmatmul(V)
        np.testing.assert_array_equal(U, bt.kmatmul(V))
    at = 0
    for X in Xs:
        v = V[at:at + len(X)]
        K = O.gram(X, X, "rbf", 1.0 / p)
        assert np.all(np.abs(U[at:at + len(X)] - K @ v) <= 2.0 ** -8 * (K @ np.abs(v)) + 1e-30)
        at += len(X)
