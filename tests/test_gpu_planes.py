"""One step from a steady state at the edges of the products' tiles (128 and 256 rows and columns,
K blocks of 64, sides that are odd multiples of 4), against the fp64 oracle.

In the steady state (the factors the mean outer products, the bases their eigenbases, the moments
stationary) every stage is well-conditioned: the refreshed bases are within about 1e-6 of fp64,
each product within 2e-7, v is bounded below by the noise's square. The update's and the state's
relative errors add these up over a handful of stages; they are held to 2e-5."""
import numpy as np
import pytest
import torch

from oracle.soap_ref import MatrixState, soap_step
from paper_2607_20548_gb300 import soap as S

from tests.parity_tools import oracle_hparams

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))


def _steady(m, n, left, right, seed):
    rng = np.random.default_rng(seed)
    k = min(m, n)
    s = np.arange(1, k + 1) ** -1.5
    s /= np.linalg.norm(s)
    U = np.linalg.qr(rng.standard_normal((m, m)))[0]
    V = np.linalg.qr(rng.standard_normal((n, n)))[0]
    A = (U[:, :k] * s) @ V[:, :k].T
    noise = 0.3 / np.sqrt(n)
    rot = A
    if left:
        rot = U.T @ rot
    if right:
        rot = rot @ V
    st = {"M": A + 0.16 * noise * rng.standard_normal((m, n)), "V": rot ** 2 + noise ** 2}
    if left:
        st.update(L=A @ A.T + 0.09 * np.eye(m), QL=U)
    if right:
        st.update(R=A.T @ A + 0.09 * m / n * np.eye(n), QR=V)
    W = 0.02 * rng.standard_normal((m, n))
    G = A + noise * rng.standard_normal((m, n))
    f = lambda x: x.astype(np.float32)  # noqa: E731
    return {p: f(x) for p, x in st.items()}, f(W), f(G)


PIECES = {"M": S.STATE_MHAT, "V": S.STATE_V, "L": S.STATE_L, "QL": S.STATE_QL, "R": S.STATE_R, "QR": S.STATE_QR}


@pytest.mark.parametrize("m,n,left,right,kl", [
    (124, 260, True, True, 0), (132, 136, True, True, 0), (128, 256, True, True, 0), (260, 516, True, True, 0),
    (516, 252, True, True, 1), (68, 60, True, True, 1), (132, 1028, True, False, 0), (1028, 132, False, True, 0),
    (260, 388, False, True, 1), (12, 20, True, True, 0), (640, 320, True, True, 0)])
def test_step_at_tile_edges(cuda, m, n, left, right, kl):
    count = 3  # a batch of one shape
    hp = S.default_hparams(kl=kl)
    ohp = oracle_hparams(hp)
    opt = S.SoapOptimizer([(m, n, left, right)] * count, hp)
    Ws, Gs, refs = [], [], []
    for i in range(count):
        st, W, G = _steady(m, n, left, right, 1000 * m + 10 * n + i)
        for p, x in st.items():
            opt.state_set(i, PIECES[p], torch.from_numpy(x).to(cuda))
        x = {p: v.astype(np.float64) for p, v in st.items()}
        ms = MatrixState(m, n, left, right, np.float64)
        ms.v = x["V"]
        ms.m = x["M"]
        if left:
            ms.L, ms.QL = x["L"], x["QL"]
            ms.m = ms.QL.T @ ms.m
        if right:
            ms.R, ms.QR = x["R"], x["QR"]
            ms.m = ms.m @ ms.QR
        ms.t = 1000
        W64, _ = soap_step(ms, W.astype(np.float64), G, ohp)
        refs.append((ms, W64 - W.astype(np.float64)))
        Ws.append(torch.from_numpy(W).to(cuda))
        Gs.append(torch.from_numpy(G).to(cuda))
    opt.t = 1000
    W0 = [w.double().cpu().numpy() for w in Ws]
    opt.step(Ws, Gs)
    torch.cuda.synchronize()
    assert opt.status() == 0, opt.last_error()
    for i, (ms, dW) in enumerate(refs):
        got = lambda which: opt.state_get(i, which).cpu().numpy()  # noqa: E731
        assert _rel(Ws[i].double().cpu().numpy() - W0[i], dW) <= 2e-5
        assert _rel(got(S.STATE_M), ms.m) <= 2e-5
        assert _rel(got(S.STATE_V), ms.v) <= 2e-5
        for on, F, Q, wf, wq in ((left, "L", "QL", S.STATE_L, S.STATE_QL), (right, "R", "QR", S.STATE_R, S.STATE_QR)):
            if on:
                assert _rel(got(wf), getattr(ms, F)) <= 2e-5
                assert _rel(got(wq), getattr(ms, Q)) <= 2e-5
    opt.destroy()
