"""Residual GEMM + LayerNorm on tiles of 16, 32 and 64 rows: the same bits as the two launches they replace, at the edges of the
tiles, with K in fewer stages than the ring has and in more, and rows that are not finite keeping to themselves."""
import pytest
import torch

from paper_2107_05377_b200 import binding as mt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [16, 32, 64])
@pytest.mark.parametrize("M,N,K", [(1, 768, 768), (15, 768, 768), (16, 768, 768), (17, 768, 128), (33, 768, 768), (64, 1024, 1024),
                                   (65, 768, 3072), (171, 1024, 1024), (512, 768, 768), (300, 768, 1152)])
def test_same_bits_as_gemm_then_layernorm(M, N, K, rows):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    draw = lambda *shape, std=1.0, mean=0.0: torch.randn(*shape, device="cuda", generator=g) * std + mean  # noqa: E731
    x, w = draw(M, K).bfloat16(), draw(N, K, std=0.05).bfloat16()
    bias, gamma, beta = draw(N, std=0.1).bfloat16(), draw(N, std=0.2, mean=1.0).bfloat16(), draw(N, std=0.2).bfloat16()
    res = draw(M, N)
    if M > 16:
        x[M // 2, 3] = float("inf")      # one row without a finite result
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    u, want, want32 = torch.empty_like(res), torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), torch.empty_like(res)
    mt.mt_kernel_linear(x, w, bias, res, u, 2)
    mt.mt_kernel_layernorm(u, gamma, beta, want, 1e-12, y_f32=want32)
    for _ in range(3):
        got, got32 = torch.full_like(want, 7.0), torch.full_like(want32, 7.0)
        mt.mt_kernel_linear_layernorm_low(x, w, bias, res, gamma, beta, got, got32, 1e-12, rows, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        finite = torch.isfinite(want32).all(1)
        assert finite.sum() == (M - 1 if M > 16 else M)
        assert torch.equal(got32[finite], want32[finite]) and torch.equal(got[finite], want[finite])
        assert not torch.isfinite(got32[~finite]).any()
