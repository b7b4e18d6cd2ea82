"""FP64-class RBF products where memory is short: the tensor-core form's layout (256 bytes a row and more) or its
partial sums cannot be had, the CUDA-core kernels' smaller buffers can.  The product has to come out all the same.
Bound: 1e-12 of sum_j |K_ij v_j| per row, the one every FP64-class product has to meet."""
import ctypes

import numpy as np
import pytest

from oracle import kqr_oracle as O
from paper_2510_07929_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class Budget:
    """Allocator callbacks that refuse a request above `limit` bytes."""

    def __init__(self, lib):
        import torch

        self.limit, self.refused = None, 0

        def alloc(nbytes, _):
            if self.limit is not None and nbytes > self.limit:
                self.refused += 1
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes))

        def free(ptr, _):
            if ptr:
                torch.cuda.caching_allocator_delete(ptr)

        self.refs = (ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(alloc),
                     ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(free))
        lib.kqr_set_allocator(ctypes.cast(self.refs[0], ctypes.c_void_p), ctypes.cast(self.refs[1], ctypes.c_void_p),
                              None)


# n = 2000 (2048 padded rows), p = 8: digits 2048 x 256 bytes, partial sums of eight vectors 8 x 2048 x 64 bytes;
# the CUDA-core product's partial sums 16 x 2048 x 8 bytes
@pytest.mark.parametrize("limit,calls", [(300_000, (1, 8, 1)), (600_000, (8, 1, 8))])
def test_products_fall_back_when_memory_is_short(limit, calls):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    n, p = 2000, 8
    X = np.random.default_rng(1).standard_normal((n, p))
    K = O.gram(X, X, "rbf", 0.2)
    budget = Budget(kqr.lib())
    try:
        with kqr.Problem(X, np.zeros(n), "rbf", 0.2, gram_store=0, rank0=2) as prob:
            for k, m in enumerate(calls + (8,)):
                budget.limit = limit if k < len(calls) else None
                V = W.random_vectors(n, m, seed=k + 3) if m > 1 else W.random_vectors(n, seed=k + 3)
                U = prob.kmatvec(V, kqr.PREC_HIGH)
                err = np.abs(U - K @ V) / (np.abs(K) @ np.abs(V))
                assert err.max() <= 1e-12, (k, m, err.max())
            assert budget.refused > 0
    finally:
        kqr.use_cuda_allocator()
