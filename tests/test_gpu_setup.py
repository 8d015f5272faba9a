"""The FP64 offline stage (relu_qp_setup's layer bank) against a direct FP64
evaluation of the factored layer in NumPy, at the sizes where its blocks can go
wrong: around the Cholesky block (32), the product tiles (16, 32, 64) and the
doubling levels of the triangular inverse (64, 128, 256), with ragged last
blocks, without constraint rows, with equality rows, and with more bank entries
than one group of the scratch holds.

Bound: both sides form K^{-1} with errors of a few n u kappa(K) relative to
|K^{-1}| (u = 2^-53, kappa the 2-norm condition number), and the products add n u;
the difference is held to 16 (n + m) u kappa(K) of the matrix's largest entry.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIGMA = 1e-6
BANK = (0.1, 1.0, 10.0)
U = 2.0 ** -53


@pytest.fixture(scope="module")
def rq():
    import paper_2311_18056_gb300 as rq
    from paper_2311_18056_gb300 import build
    build.build()
    return rq


def problem(n, m, eq, seed=0):
    rng = np.random.default_rng([12, n, m, seed])
    M = rng.standard_normal((n, n))
    P = M @ M.T / n + 0.1 * np.eye(n)
    A = rng.standard_normal((m, n)) / np.sqrt(n)
    l, u = -np.ones(m), np.ones(m)
    l[:eq] = u[:eq]
    return P, A, l, u


@pytest.mark.parametrize("n,m,eq", [(1, 0, 0), (1, 1, 0), (15, 17, 3), (31, 33, 0), (32, 32, 32), (33, 1, 0), (63, 65, 2),
                                    (64, 0, 0), (65, 129, 0), (97, 40, 8), (128, 96, 0), (130, 70, 7), (257, 31, 0),
                                    (300, 450, 20)])
def test_bank_at_block_edges(rq, n, m, eq):
    P, A, l, u = problem(n, m, eq)
    h = rq.ReluQP(P, A if m else None, l, u, sigma=SIGMA, rho_bank=BANK, keep_fp64=True)
    try:
        for r, rho in enumerate(BANK):
            s = np.where(l == u, 1000.0, 1.0)
            C = A.T @ ((rho * s)[:, None] * A)
            K = P + SIGMA * np.eye(n) + C
            D = np.linalg.inv(K)
            X = D @ (SIGMA * np.eye(n) - C)
            Wt = np.block([[X, D @ A.T], [A @ X, A @ D @ A.T]])
            Bop = -np.vstack([D, A @ D])
            got_W, got_B = h.get_layer(r)
            tol = 16 * (n + m) * U * np.linalg.cond(K)
            assert np.max(np.abs(got_W - Wt)) <= tol * np.max(np.abs(Wt)), (r, tol)
            assert np.max(np.abs(got_B - Bop)) <= tol * np.max(np.abs(Bop)), (r, tol)
    finally:
        h.close()


def test_bank_in_several_groups(rq):
    """16 entries of n = 3000 take more than one group of the stage's scratch: without
    constraint rows every entry is the same layer, sigma D with D K = I."""
    n = 3000
    rng = np.random.default_rng(5)
    d = rng.uniform(1.0, 2.0, n)
    v = rng.standard_normal(n) / np.sqrt(n)
    h = rq.ReluQP(np.diag(d) + np.outer(v, v), None, np.zeros(0), np.zeros(0), sigma=SIGMA,
                  rho_bank=tuple(0.1 * 1.5 ** k for k in range(16)), keep_fp64=True)
    try:
        a = 1.0 / (d + SIGMA)          # Sherman-Morrison for K = diag(d + sigma) + v v'
        D = np.diag(a) - np.outer(a * v, a * v) / (1.0 + v @ (a * v))
        for r in (0, 13, 14, 15):
            _, Bop = h.get_layer(r)
            assert np.max(np.abs(Bop + D)) <= 16 * n * U * 4.0 * np.max(a), r   # kappa(K) < 4
    finally:
        h.close()
