"""Muon's products in every form they run in: one CTA or a pair of CTAs per tile, and a symmetric
product whole or as its lower tiles, mirrored. The forms are chosen by the estimated times that `form`
restates; the cases reach all of them with sides whose last 256-wide tile is ragged (136 or 200 rows of
it, or 72: then the second CTA has none). Against the oracle and with the bounds of
tests/test_gpu_muon.py, on two matrices of each class."""
import numpy as np
import pytest
import torch

from oracle.muon_ref import MuonParams, MuonState, muon_step
from paper_2607_20548_gb300 import soap as S

from tests.test_gpu_muon import QUINTIC, _ok, _rel

SMS = 152


def form(M, N, K, batch, symmetric):
    def us(cg, lower, launch, a_slice, epilogue):
        a, b = -(-M // (128 * cg)), -(-N // (128 * cg))
        tiles = (a * (a + 1) // 2 if lower else a * b) * batch
        return launch + -(-tiles // (SMS // cg)) * (-(-K // 64) * a_slice + epilogue)
    if not symmetric:
        two = M > 128 and N > 128 and us(2, False, 6.4, 0.24, 9.9) < us(1, False, 4.3, 0.27, 3.5)
        return "pairs" if two else "singles"
    whole, lower = us(1, False, 4.4, 0.26, 1.6), us(1, True, 4.0, 0.30, 1.9)
    if M > 128 and us(2, True, 5.9, 0.33, 4.0) < min(whole, lower):
        return "lower pairs"
    return "lower singles" if lower < whole else "symmetric singles"


CASES = [(904, 1160, 24), (1096, 904, 15), (712, 712, 32), (1096, 1096, 6), (1096, 1096, 4), (904, 904, 12), (136, 520, 3)]


def test_cases_reach_every_form():
    reached = set()
    for r, c, count in CASES:
        r, c = min(r, c), max(r, c)
        reached |= {form(r, r, c, count, True), form(r, r, r, count, True), form(r, c, r, count, False)}
    assert reached == {"singles", "pairs", "symmetric singles", "lower singles", "lower pairs"}
    assert form(904, 1096, 904, 15, False) == form(1096, 1096, 1096, 6, False) == "pairs"
    assert form(1096, 1096, 1096, 4, True) == "lower pairs"


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,count", CASES)
def test_muon_in_every_form(cuda, rows, cols, count):
    coeffs = QUINTIC[:3]
    rng = np.random.default_rng(rows + cols)
    f = lambda x: x.astype(np.float32)  # noqa: E731
    data = []  # weights, momentum, gradient; the class is filled with copies of two in turn
    for _ in range(2):
        A = rng.standard_normal((rows, cols)) / np.sqrt(rows * cols)
        noise = 0.3 / np.sqrt(rows * cols)
        data.append((f(0.02 * rng.standard_normal((rows, cols))), f(A + 0.2 * noise * rng.standard_normal((rows, cols))),
                     f(A + noise * rng.standard_normal((rows, cols)))))
    opt = S.MuonOptimizer([(rows, cols)] * count, coeffs=coeffs)
    W = [torch.from_numpy(data[i % 2][0]).to(cuda) for i in range(count)]
    G = [torch.from_numpy(data[i % 2][2]).to(cuda) for i in range(count)]
    for i in range(count):
        opt.state_set(i, torch.from_numpy(data[i % 2][1]).to(cuda))
    opt.step(W, G)
    torch.cuda.synchronize()
    assert opt.status() == 0
    for i, (W0, M0, G0) in enumerate(data):
        out = {}
        for name, hp in (("fp64", MuonParams(coeffs=list(coeffs))), ("bf16", MuonParams(coeffs=list(coeffs), ns_bf16=True))):
            st = MuonState(rows, cols, np.float64, 0, M0.astype(np.float64))
            out[name] = (muon_step(st, W0.astype(np.float64), G0.astype(np.float64), hp)[0], st.M)
        dW = {name: x[0] - W0 for name, x in out.items()}
        for j in (i, count - 2 + (i - count) % 2):  # its first and its last copy
            assert j % 2 == i
            d = W[j].cpu().numpy().astype(np.float64) - W0
            x = dict(e64=_rel(d, dW["fp64"]), e16=_rel(d, dW["bf16"]), e_twin=_rel(dW["bf16"], dW["fp64"]),
                     e_m=_rel(opt.state_get(j).cpu().numpy(), out["fp64"][1]))
            assert _ok(x), (j, x)
    opt.destroy()
