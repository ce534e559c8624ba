"""The QR's blocks factored from their Gram matrix, next to blocks left to the column loop and
blocks of zero columns, against the oracle's Householder QR on identical fp32 inputs.

Tolerances as for the QR elsewhere: Q within 4x the oracle's own fp32 twin of fp64 (or 1e-5),
Q^T Q = I to 1e-5, the zero-column flags equal."""
import numpy as np
import pytest
import torch

from oracle.soap_ref import householder_q
from paper_2607_20548_gb300 import soap as S

pytestmark = pytest.mark.gpu
TOL = 2e-5


def _steady(n, rng):
    """P = F Q with Q the eigenbasis of a factor that one more gradient has moved: nearly
    orthogonal columns, as a refresh in the steady state of a run meets them."""
    U = np.linalg.qr(rng.standard_normal((n, n)))[0]
    s = np.arange(1, n + 1) ** -1.5
    s /= np.linalg.norm(s)
    G = (U * s) @ rng.standard_normal((n, n)) / np.sqrt(n) + 0.3 * rng.standard_normal((n, n)) / np.sqrt(n)
    F = 0.95 * ((U * (s * s + 0.09)) @ U.T) + 0.05 * G @ G.T
    return F @ U


def _case(n, kind, seed):
    rng = np.random.default_rng(seed)
    P = _steady(n, rng)
    if kind == "scaled":  # a small expert: squared column norms around 1e-14
        P = P * 1e-7
    elif kind == "zero_blocks":  # the columns from a block's start on are zero
        P[:, 128:] = 0.0
    elif kind == "mixed":  # a block with zero columns in it: the column loop
        P[:, n // 2 + 3:] = 0.0
    elif kind == "repeated":  # a column that repeats an earlier one of its block: the column loop
        P[:, 5] = P[:, 1] + 1e-3 * P[:, 5]
    return P.astype(np.float32)


@pytest.mark.parametrize("n,batch,kind", [
    (4, 3, "steady"), (28, 2, "steady"), (124, 1, "steady"), (128, 2, "steady"), (132, 2, "steady"),
    (252, 1, "steady"), (256, 2, "scaled"), (260, 1, "steady"), (272, 1, "scaled"), (644, 2, "steady"),
    (1028, 1, "steady"), (384, 2, "zero_blocks"), (260, 2, "mixed"), (516, 1, "mixed"), (256, 17, "repeated"),
    (1156, 1, "repeated"), (1156, 2, "mixed")])
def test_block_factorisation_matches_oracle(cuda, n, batch, kind):
    P = np.stack([_case(n, kind, 100 * n + b) for b in range(batch)])
    if batch > 1:  # neighbours in a batch may go different ways
        P[1] = _case(n, "steady", 7 * n)
    Q, skip, status = S.soap_qr(torch.from_numpy(P).to(cuda), TOL, return_status=True)
    Q, skip = Q.cpu().numpy(), skip.cpu().numpy().astype(bool)
    assert status.item() == 0
    for b in range(min(batch, 3)):
        Q64, s64, _ = householder_q(P[b].astype(np.float64), TOL)
        Q32 = householder_q(P[b], TOL)[0]
        assert np.array_equal(skip[b], s64)
        assert np.abs(Q[b].astype(np.float64).T @ Q[b] - np.eye(n)).max() <= 1e-5
        rel = lambda x: np.linalg.norm(x.astype(np.float64) - Q64) / np.linalg.norm(Q64)  # noqa: E731
        assert rel(Q[b]) <= max(1e-5, 4 * rel(Q32)), (b, rel(Q[b]), rel(Q32))


@pytest.mark.parametrize("n,batch,kind", [
    (380, 1, "steady"), (384, 2, "steady"), (388, 2, "steady"), (512, 1, "mixed"), (516, 3, "steady"),
    (768, 2, "zero_blocks"), (1020, 1, "steady"), (1024, 1, "steady"), (1028, 2, "mixed"), (1540, 1, "steady")])
def test_superblocks_match_oracle(cuda, n, batch, kind):
    """Around the widths (384 columns, 512 from n = 1024) at which the accumulation of Q goes on to
    another superblock, with a last one of several blocks, of one, and of 4 columns."""
    test_block_factorisation_matches_oracle(cuda, n, batch, kind)
