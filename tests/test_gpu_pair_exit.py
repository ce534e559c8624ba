"""The end of the products that run on pairs of CTAs: a wait that gives up leaves nothing in flight
towards either CTA's shared memory, whichever of the two producers had gone further, and the
products after it are those of an undisturbed context.

The class (16 of 388 x 388, two-sided) is large enough that every product of its step runs on pairs
(16 of 388 x 388 are 4 waves of 128 x 128 tiles on 152 SMs and one of 256 x 256 tiles on 76 pairs)."""
import numpy as np
import pytest
import torch

from paper_2607_20548_gb300 import soap as S

pytestmark = pytest.mark.gpu

COUNT, SIDE = 16, 388
LIMIT_NS = 1_000_000  # 1 ms: the bound the waits get


def _step(cuda):
    g = torch.Generator(device=cuda).manual_seed(17)
    W = list((0.02 * torch.randn(COUNT, SIDE, SIDE, device=cuda, generator=g)).unbind(0))
    G = list((torch.randn(COUNT, SIDE, SIDE, device=cuda, generator=g) / np.sqrt(SIDE)).unbind(0))
    opt = S.SoapOptimizer([(SIDE, SIDE, True, True)] * COUNT)
    return opt, W, G


def test_pair_wait_runs_out_and_the_next_step_is_undisturbed(cuda):
    opt, W, G = _step(cuda)
    opt.step(W, G)
    torch.cuda.synchronize()
    assert opt.status() == 0
    opt.destroy()

    held, Wh, Gh = _step(cuda)
    hold = torch.zeros(1, dtype=torch.int32, device=cuda)
    try:
        S.soap_wait_limit(LIMIT_NS, hold)
        held.step(Wh, Gh)
        torch.cuda.synchronize()
    finally:
        S.soap_wait_limit(0, None)
    assert held.status() == 6  # SOAP_ERR_TIMEOUT
    held.destroy()

    again, Wa, Ga = _step(cuda)
    again.step(Wa, Ga)
    torch.cuda.synchronize()
    assert again.status() == 0
    for a, b in zip(W, Wa):
        assert torch.equal(a, b)
    again.destroy()
