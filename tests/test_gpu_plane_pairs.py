"""One step from a steady state of classes large enough that their products run on pairs of CTAs
(256 x 256 tiles), with sides whose last tile is ragged: 132 of its 256 rows (the second CTA has 4) or
68 (it has none). As in tests/test_gpu_planes.py, whose bound of 2e-5 holds here for the same
reasons; three matrices of each class are compared with the fp64 oracle.

The cases are chosen by the rule that splits the products between single CTAs and pairs, restated in
`pair`, so that over them every kind of product runs on pairs: gradient and moment into the basis
(transposed planes, fp32), the factors (symmetric, mirrored), Q^T F, the update into the weights, as
they are and transposed."""
import numpy as np
import pytest
import torch

from oracle.soap_ref import MatrixState, soap_step
from paper_2607_20548_gb300 import soap as S

from tests.parity_tools import oracle_hparams
from tests.test_gpu_planes import PIECES, _rel, _steady

SMS = 152


def pair(M, N, batch, symmetric=False):
    def waves(t, slots):
        a, b = -(-M // t), -(-N // t)
        return -(-((a * (a + 1) // 2 if symmetric else a * b) * batch) // slots)
    return M > 128 and N > 128 and 6 * waves(128, SMS) >= 10 * waves(256, SMS // 2)


def products(m, n, count, left, right, kl):
    """Which of the step's kinds of product run on pairs."""
    out = {}
    rr, cc = (n, m) if left and not right else (m, n)  # working orientation
    out["into the basis"] = pair(rr, cc, 2 * count)
    out["update"] = pair(rr, cc, count)
    for on, a, o, side in ((left, m, n, "L"), (right, n, m, "R")):
        if on:
            out["factor " + side] = pair(a, a, count, True)
            out["Q^T F " + side] = pair(a, a, count)
            if kl and left and right:
                out["KL " + side] = pair(a, o, count)
    return out


CASES = [
    # m, n, count, left, right, kl
    (388, 388, 16, True, True, 1),
    (644, 388, 12, True, True, 0),
    (1092, 388, 36, True, True, 0),
    (388, 1092, 36, True, False, 0),
    (1092, 388, 24, False, True, 1),
    (1092, 132, 5, True, False, 0),
]


def test_cases_run_on_pairs():
    reached = set()
    for m, n, count, left, right, kl in CASES:
        p = products(m, n, count, left, right, kl)
        reached |= {k for k, on in p.items() if on}
        assert any(p.values())
    assert {"into the basis", "update", "factor L", "factor R", "Q^T F L", "Q^T F R", "KL L", "KL R"} <= reached


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,count,left,right,kl", CASES)
def test_step_on_pairs(cuda, m, n, count, left, right, kl):
    hp = S.default_hparams(kl=kl)
    ohp = oracle_hparams(hp)
    opt = S.SoapOptimizer([(m, n, left, right)] * count, hp)
    distinct = 3  # inputs; the class is filled with copies of them in turn
    data = [_steady(m, n, left, right, 1000 * m + 10 * n + i) for i in range(distinct)]
    Ws, Gs = [], []
    for i in range(count):
        st, W, G = data[i % distinct]
        for p, x in st.items():
            opt.state_set(i, PIECES[p], torch.from_numpy(x).to(cuda))
        Ws.append(torch.from_numpy(W).to(cuda))
        Gs.append(torch.from_numpy(G).to(cuda))
    opt.t = 1000
    opt.step(Ws, Gs)
    torch.cuda.synchronize()
    assert opt.status() == 0, opt.last_error()
    for i, (st, W, G) in enumerate(data):
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
        dW = W64 - W.astype(np.float64)
        for j in (i, count - distinct + (i - count) % distinct):  # its first and its last copy
            assert j % distinct == i
            got = lambda which: opt.state_get(j, which).cpu().numpy()  # noqa: E731, B023
            assert _rel(Ws[j].double().cpu().numpy() - W.astype(np.float64), dW) <= 2e-5
            assert _rel(got(S.STATE_M), ms.m) <= 2e-5
            assert _rel(got(S.STATE_V), ms.v) <= 2e-5
            for on, F, Q, wf, wq in ((left, "L", "QL", S.STATE_L, S.STATE_QL), (right, "R", "QR", S.STATE_R, S.STATE_QR)):
                if on:
                    assert _rel(got(wf), getattr(ms, F)) <= 2e-5
                    assert _rel(got(wq), getattr(ms, Q)) <= 2e-5
    opt.destroy()
