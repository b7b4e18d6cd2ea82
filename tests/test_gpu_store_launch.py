"""The one-launch product of a stored K (gram_stored.cu): sizes up to its line of 5120 rows and beyond it,
ragged last tiles, products one after another (the sums it leaves zero), in place and at odd offsets,
against the FP64 oracle at the bound of the existing FP32-class tests, 1e-5 of max |K v|."""
import numpy as np
import pytest

from oracle import kqr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["rbf", "laplacian"])
@pytest.mark.parametrize("n", [2, 127, 128, 129, 1000, 2001, 5119, 5120, 5121])
def test_products_one_after_another(n, kind):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 5))
    with kqr.Problem(X, np.zeros(n), kind, 0.2, gram_store=1, rank0=2) as prob:
        buf = torch.zeros(2 * n + 3, dtype=torch.float64, device="cuda")
        for rep in range(3):
            v = rng.standard_normal(n)
            ref = O.kmatvec(X, v, kind, 0.2)
            bound = 1e-5 * np.max(np.abs(ref))
            assert np.max(np.abs(prob.kmatvec(v, kqr.PREC_FP32) - ref)) <= bound
            V, U = buf[1:1 + n], buf[n + 2:2 * n + 2]   # 8-byte aligned only
            V.copy_(torch.as_tensor(v))
            torch.cuda.synchronize()
            prob.kmatvec_dev(V, U, kqr.PREC_FP32)
            torch.cuda.synchronize()
            assert np.max(np.abs(U.cpu().numpy() - ref)) <= bound
            prob.kmatvec_dev(V, V, kqr.PREC_FP32)
            torch.cuda.synchronize()
            assert np.max(np.abs(V.cpu().numpy() - ref)) <= bound
            assert float(buf[0]) == 0.0 and float(buf[n + 1]) == 0.0 and float(buf[-1]) == 0.0
