"""Precision of the Woodbury core and apply (kqr_precond_apply_dev): no further from the exact Lemma 1 result than the
same steps in FP64 with plain running sums.  Both errors are geometric means over right-hand sides; the factor 1.5 is
the spread of such a mean of eight (a single error varies by a factor of about 2.5 either way)."""
import numpy as np
import pytest

from oracle import kqr_oracle as O
from paper_2510_07929_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def K_():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_07929_gb300 import build

    build.build()
    from paper_2510_07929_gb300 import kqr

    return kqr


def diagonals(n, F, rng):
    dres = np.maximum(1.0 - np.sum(F.astype(float) ** 2, axis=1), 0.0)
    dres = np.maximum(dres, 0.1 * dres.mean())
    return {"flat": (rng.random(n) + 0.3, 1.0), "phase1": (1e-2 + dres, 1e-2),
            "newton": (np.where(rng.random(n) < 0.33, 1e-5, 1.0) + dres, 1.0)}


def exact(U, L, C, R):
    Ul, Ll = U.astype(LD), L.astype(LD)[:, None]
    G = (Ul / Ll).T @ Ul + C
    Gi = np.linalg.inv(G.astype(float))
    T = Ul.T @ (R / Ll)
    X = (Gi @ T.astype(float)).astype(LD)
    for _ in range(5):
        X = X + (Gi @ (T - G @ X).astype(float)).astype(LD)
    return (R - Ul @ X) / Ll


def in_fp64(U, L, C, R):
    """Running FP64 sums, row after row and column after column."""
    Li = 1.0 / L
    G = np.zeros((U.shape[1],) * 2)
    for u, w in zip(U, Li):
        G += np.outer(u * w, u)
    c = np.linalg.cholesky(G + C)
    Wi = np.linalg.inv(c)
    T = np.stack([np.cumsum(U * (Li * r)[:, None], axis=0)[-1] for r in R.T], axis=1)
    T2 = (Wi.T @ Wi) @ T
    S = np.stack([np.cumsum(U * t, axis=1)[:, -1] for t in T2.T], axis=1)
    return Li[:, None] * (R - S)


@pytest.mark.parametrize("n,rank", [(700, 120), (1100, 60), (500, 250)])
def test_apply_errs_no_more_than_fp64(K_, n, rank):
    import torch

    wl = W.rbf_mid(n=n, p=16, seed=n)
    rng = np.random.default_rng(rank)
    R = rng.standard_normal((n, 8))
    with K_.Problem(wl.X, wl.y, wl.kind, wl.gamma, rank0=rank, adaptive_rank=0, gram_store=0,
                    pivot_uniforms=W.pivot_uniforms(rank)) as prob:
        F, _, r, _ = prob.factor()
        assert r == rank
        U = np.concatenate([F.astype(float), np.ones((n, 1))], axis=1)
        for name, (L, gam) in diagonals(n, F, rng).items():
            C = np.eye(r + 1)
            C[r, r] = 1.0 / gam
            ref = exact(U, L, C, R)
            got = []
            for c in range(R.shape[1]):
                out = torch.empty(n, dtype=torch.float64, device="cuda")
                prob.precond_apply_dev(torch.from_numpy(L).cuda(), gam, torch.from_numpy(R[:, c].copy()).cuda(), out)
                got.append(out.cpu().numpy())
            host = in_fp64(U, L, C, R)

            def error(x):
                e = np.linalg.norm((x - ref).astype(float), axis=0) / np.linalg.norm(ref.astype(float), axis=0)
                return np.exp(np.mean(np.log(e)))

            e_gpu, e_host = error(np.stack(got, axis=1)), error(host)
            assert e_gpu <= 1.5 * e_host, (name, n, rank, e_gpu, e_host)
