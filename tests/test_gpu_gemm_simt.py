"""The CUDA-core product at the edges of its tiles and of the rule that chooses them, and the tf32 parts."""
import pytest
import torch

from paper_2607_20548_gb300 import soap as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ta,tb", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("batch,M,N,K", [
    (1, 1, 1, 1), (2, 33, 63, 31), (3, 32, 65, 97),      # 32 x 64 tiles, steps of 32
    (114, 33, 64, 9), (9, 257, 191, 70),                 # 64 x 64 tiles
    (304, 65, 129, 17), (5, 1023, 1027, 33),             # 128 x 128 tiles, steps of 16
])
def test_simt_tiles(ta, tb, batch, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M * 7 + K)
    A = torch.randn((batch, K, M) if ta else (batch, M, K), device="cuda", generator=g)
    B = torch.randn((batch, N, K) if tb else (batch, K, N), device="cuda", generator=g)
    C = S.soap_gemm(A, B, trans_a=ta, trans_b=tb, alpha=0.75)
    a = A.double().transpose(1, 2) if ta else A.double()
    b = B.double().transpose(1, 2) if tb else B.double()
    # a chain of K fused multiply-adds and one product by alpha: gamma_(K+1) |a| |b|
    bound = (K + 1) * 2.0 ** -24 * 1.01 * 0.75 * (a.abs() @ b.abs())
    assert ((C.double() - 0.75 * (a @ b)).abs() <= bound + 1e-37).all()


@pytest.mark.parametrize("n", [1, 3, 5, 4096, 8 * 152 * 256 * 16 + 7])
@pytest.mark.parametrize("offset", [0, 1])
def test_split_parts(n, offset):
    """16-byte and 4-byte accesses give the same two parts: hi truncated to tf32, lo the rest rounded."""
    x = torch.randn(n + offset, device="cuda")[offset:]
    hi, lo = S.soap_split_tf32(x)
    assert torch.equal(hi.view(torch.int32), x.view(torch.int32) & ~0x1FFF)
    rest = (x - hi).view(torch.int32)  # exact; nearest tf32, ties away from zero
    assert torch.equal(lo.view(torch.int32), (rest + 0x1000) & ~0x1FFF)
