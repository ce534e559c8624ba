"""Blocks that the QR must not factor from their Gram matrix although every Cholesky pivot keeps a good
part of its column's norm: their condition, squared, is what the Gram matrix's rounding is multiplied
by, and many moderate pivots multiply up to a large one.

P = Q R with Q orthogonal and R as named, columns of unit norm; beside it in the batch a
well-conditioned P. Held to the bound of the QR elsewhere: Q^T Q = I to 1e-5, and Q^T P upper
triangular to 1e-5 of ||P||_F with a non-negative diagonal."""
import numpy as np
import pytest
import torch

from paper_2607_20548_gb300 import soap as S

pytestmark = pytest.mark.gpu
TOL = 2e-5
N = 512


def _bidiagonal(n, rho):
    """Each column: sqrt(rho) of its own, the rest along the previous direction."""
    R = np.diag(np.full(n, np.sqrt(rho))) + np.diag(np.full(n - 1, np.sqrt(1 - rho)), 1)
    R[0, 0] = 1
    return R


def _random(n, rho, rng):
    """Squared diagonal rho, the rest of each column in a random direction above it."""
    R = np.triu(rng.standard_normal((n, n)), 1)
    R[:, 1:] *= np.sqrt(1 - rho) / np.linalg.norm(R[:, 1:], axis=0)
    return R + np.diag(np.r_[1, np.full(n - 1, np.sqrt(rho))])


def _previous(n, rho, rng):
    """Each column sqrt(rho) of its own, the rest along the previous column (not direction)."""
    R = np.zeros((n, n))
    R[0, 0] = 1
    for j in range(1, n):
        R[:, j] = np.sqrt(1 - rho) * R[:, j - 1]
        R[j, j] += np.sqrt(rho)
    return R


def _one_small(n, lam):
    """Blocks of 128 columns with one singular value squared of 1 / lam, spread over all of them."""
    k = 128
    G = np.eye(k) - (1 - 1 / lam) / k
    return np.kron(np.eye(n // k), np.linalg.cholesky(G / G[0, 0]).T)


def _well(n, rng):
    F = rng.standard_normal((n, 4 * n))
    return F @ F.T / (4 * n) + np.eye(n)


@pytest.mark.parametrize("kind,rho", [
    ("random", 0.27), ("random", 0.35), ("random", 0.5), ("random", 0.7), ("random", 0.8), ("bidiagonal", 0.3),
    ("bidiagonal", 0.4), ("bidiagonal", 0.8), ("plain bidiagonal", 0.35), ("previous", 0.45), ("one small", 256),
    ("one small", 32), ("one small", 20)])
def test_ill_conditioned_blocks(cuda, kind, rho):
    rng = np.random.default_rng(int(100 * rho))
    R = {"random": lambda: _random(N, rho, rng), "bidiagonal": lambda: _bidiagonal(N, rho),
         "plain bidiagonal": lambda: _bidiagonal(N, rho), "previous": lambda: _previous(N, rho, rng),
         "one small": lambda: _one_small(N, rho)}[kind]()
    A = R if kind == "plain bidiagonal" else np.linalg.qr(rng.standard_normal((N, N)))[0] @ R
    P = np.stack([A, _well(N, rng)]).astype(np.float32)
    Q, skip, status = S.soap_qr(torch.from_numpy(P).to(cuda), TOL, return_status=True)
    torch.cuda.synchronize()
    assert status.item() == 0
    assert not skip.any().item()
    eye = np.eye(N)
    for b in range(2):
        q = Q[b].double().cpu().numpy()
        r = q.T @ P[b].astype(np.float64)
        assert np.abs(q.T @ q - eye).max() <= 1e-5, b
        assert np.abs(np.tril(r, -1)).max() <= 1e-5 * np.linalg.norm(r), b
        assert np.diag(r).min() >= -1e-6 * np.linalg.norm(r), b
