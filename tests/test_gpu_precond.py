"""The Woodbury core's blocked inverse through kqr_precond_apply_dev (Lemma 1), at ranks around
the edges of its 32 x 32 blocks and of its doubling steps, against the FP64 oracle."""
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


def woodbury_error(K_, n, rank, L, gam, seed):
    import torch

    wl = W.lap_large(n=n, p=20, seed=seed)
    with K_.Problem(wl.X, wl.y, wl.kind, wl.gamma, rank0=rank, adaptive_rank=0,
                    pivot_uniforms=W.pivot_uniforms(max(rank, 2))) as prob:
        F, _, r, _ = prob.factor()
        assert r == rank
        rv = np.random.default_rng(seed).standard_normal(n)
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        prob.precond_apply_dev(torch.from_numpy(L).cuda(), gam, torch.from_numpy(rv).cuda(), out)
    ref = O.woodbury_apply(F.astype(np.float64), L, gam, rv)
    return np.max(np.abs(out.cpu().numpy() - ref)) / np.max(np.abs(ref))


# The core is I + U^T L^{-1} U with L in [0.5, 1.5]: condition at most ~4 n (the constant mode), so
# both sides' FP64 errors stay below 4 n N 2^-53 = 4e-10 at n = 1200, N = 700.
@pytest.mark.parametrize("rank", [1, 2, 30, 31, 32, 33, 62, 63, 64, 95, 96, 130, 255, 256, 700])
def test_core_inverse_at_block_edges(K_, rank):
    n = 1200
    L = np.random.default_rng(rank).uniform(0.5, 1.5, n)
    assert woodbury_error(K_, n, rank, L, 0.3, seed=rank) <= 4e-10


# Weights from 1e-30 to 1e12 (their products leave the FP32 range without the power-of-two scaling), ranks
# at the edges of the 64 x 64 tiles, rows at the edges of the 64-row sums.  Bound: the one of the Lemma 1
# test (both sides solve with a core whose condition is at most that of L^-1 times that of U^T U).
@pytest.mark.parametrize("n,rank", [(64, 5), (65, 63), (127, 64), (1000, 65), (1537, 128), (4099, 129)])
@pytest.mark.parametrize("low", [1e-12, 1e-2, 1e30])
def test_core_gram_at_tile_edges(K_, n, rank, low):
    rng = np.random.default_rng(rank)
    L = low * rng.uniform(1.0, 10.0, n)
    assert woodbury_error(K_, n, rank, L, 0.3, seed=rank) <= 1e-8


@pytest.mark.parametrize("kind,n,r0", [("laplacian", 2, 2), ("rbf", 63, 9), ("laplacian", 64, 20), ("rbf", 129, 30),
                                       ("laplacian", 9728, 24), ("rbf", 9729, 24), ("laplacian", 13001, 16)])
def test_rpcholesky_pivots_at_chunk_edges(K_, kind, n, r0):
    """Pivot draws against the oracle (same uniforms) where the rows per CTA change and where chunks are ragged."""
    wl = W.lap_large(n=n, p=7, seed=n) if kind == "laplacian" else W.rbf_mid(n=n, p=7, seed=n)
    u = W.pivot_uniforms(r0, seed=5)
    with K_.Problem(wl.X, wl.y, kind, wl.gamma, rank0=r0, adaptive_rank=0, pivot_uniforms=u, gram_store=0) as prob:
        F, piv, r, _ = prob.factor()
    F0, piv_o = O.rpcholesky(lambda s: O.gram(wl.X, wl.X[s:s + 1], kind, wl.gamma)[:, 0], np.ones(n), r0, u)
    np.testing.assert_array_equal(piv, piv_o)
    np.testing.assert_allclose(F, F0[:, :r], atol=2e-6 * np.max(np.abs(F0)))


# The apply's passes over F at the edges of their tiles (32 columns, 128 rows) and with r and L far outside the
# FP32 range (the double-float parts are scaled by powers of two): relative to the same apply at scale 1 the result
# only picks up the power of two, exactly, where all scale factors are powers of two.
@pytest.mark.parametrize("n,rank", [(127, 7), (129, 8), (1025, 31), (3000, 63)])
def test_apply_scales_exactly(K_, n, rank):
    import torch

    wl = W.lap_large(n=n, p=6, seed=n)
    rng = np.random.default_rng(n)
    L = rng.uniform(0.5, 2.0, n)
    rv = rng.standard_normal(n)
    with K_.Problem(wl.X, wl.y, wl.kind, wl.gamma, rank0=rank, adaptive_rank=0) as prob:
        F, _, _, _ = prob.factor()

        def apply(r):
            out = torch.empty(n, dtype=torch.float64, device="cuda")
            prob.precond_apply_dev(torch.from_numpy(L).cuda(), 0.5, torch.from_numpy(r).cuda(), out)
            return out.cpu().numpy()

        base = apply(rv)
        ref = O.woodbury_apply(F.astype(np.float64), L, 0.5, rv)
        # condition of the core at most ~10 n: both sides' FP64 errors below 10 n N 2^-53
        assert np.max(np.abs(base - ref)) <= 2e-9 * np.max(np.abs(ref))
        for e in (-800, -150, 40, 400):
            # the sums into U^T L^-1 r arrive in any order: FP64 rounding differs between calls
            np.testing.assert_allclose(apply(np.ldexp(rv, e)), np.ldexp(base, e), rtol=0,
                                       atol=2e-9 * np.ldexp(np.max(np.abs(base)), e))
