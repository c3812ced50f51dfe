"""Linear maps on tiles of 16, 32 and 64 rows, taken transposed: the bits of the full tiles with every epilogue, at the edges of the
tiles, with K in fewer stages than the ring has, as many and more, with ranges of K, and with fewer rows in use than planned; nothing
is written beyond the rows, and a row that is not finite keeps to itself."""
import pytest
import torch

from paper_2107_05377_b200 import binding as mt

pytestmark = pytest.mark.gpu

SIZES = [(1, 768, 768), (15, 768, 128), (16, 128, 768), (17, 2304, 768), (33, 1024, 1024), (63, 768, 1152), (65, 3072, 768), (171, 768, 3072)]


def draw(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    rnd = lambda *shape, std=1.0: torch.randn(*shape, device="cuda", generator=g) * std   # noqa: E731
    x, w, bias, res = rnd(M, K).bfloat16(), rnd(N, K, std=0.05).bfloat16(), rnd(N, std=0.1).bfloat16(), rnd(M, N)
    if M > 1:
        x[M // 2, 3] = float("inf")
    return x, w, bias, res, torch.zeros(1, dtype=torch.int32, device="cuda")


def same(got, want, M):
    finite = torch.isfinite(want).all(1)
    assert finite.sum() == (M - 1 if M > 1 else M)
    assert torch.equal(got[finite], want[finite]) and not torch.isfinite(got[~finite]).all(1).any()


@pytest.mark.parametrize("rows", [16, 32, 64])
@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("epilogue", [0, 1, 2, 3])
def test_same_bits_as_full_tiles(M, N, K, rows, epilogue):
    x, w, bias, res, status = draw(M, N, K)
    kind = torch.bfloat16 if epilogue < 2 else torch.float32
    want = torch.empty(M, N, dtype=kind, device="cuda")
    if epilogue == 3:
        res.zero_()
    mt.mt_kernel_linear(x, w, bias, res, want, min(epilogue, 2))
    got = torch.full((M + 70, N), 7.0, dtype=kind, device="cuda")
    mt.mt_kernel_linear_low(x, w, bias, res, got, epilogue, rows, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    if epilogue == 3:
        # (tanh(inf) is finite; tanhf is exact to 2 units in the last place, and so is the tanh it is compared with)
        want = torch.tanh(want)
        assert torch.allclose(got[:M], want, rtol=0, atol=4 * 2 ** -24)
    else:
        same(got[:M], want, M)
    assert (got[M:] == 7.0).all(), "rows beyond M must be left alone"


@pytest.mark.parametrize("rows", [16, 32, 64])
@pytest.mark.parametrize("M,N,K,splits", [(1, 768, 3072, 4), (17, 768, 3072, 1), (33, 1024, 4096, 4), (64, 768, 256, 2), (171, 768, 3072, 4)])
def test_same_partial_sums_as_full_tiles(M, N, K, splits, rows):
    x, w, _, _, status = draw(M, N, K)
    pitch = (M + 127) // 128 * 128
    want, got = (torch.full((splits * pitch, N), 7.0, device="cuda") for _ in range(2))
    mt.mt_kernel_linear_partial(x, w, want, splits, pitch)
    mt.mt_kernel_linear_low(x, w, None, None, got, 4, rows, k_splits=splits, split_pitch=pitch, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for s in range(splits):
        part, whole = got[s * pitch:s * pitch + M], want[s * pitch:s * pitch + M]
        finite = torch.isfinite(whole).all(1)
        assert finite.sum() >= M - 1 and torch.equal(part[finite], whole[finite])
        assert (got[s * pitch + M:(s + 1) * pitch] == 7.0).all(), "rows beyond M must be left alone"


@pytest.mark.parametrize("rows", [16, 32, 64])
@pytest.mark.parametrize("in_use", [1, 16, 31, 64, 100, 200])
def test_only_the_rows_in_use_are_written(in_use, rows):
    M, N, K = 171, 768, 768
    x, w, bias, res, status = draw(M, N, K)
    want = torch.empty(M, N, device="cuda")
    mt.mt_kernel_linear(x, w, bias, res, want, 2)
    got = torch.full((M, N), 7.0, device="cuda")
    mt.mt_kernel_linear_low(x, w, bias, res, got, 2, rows, rows=torch.tensor([in_use], dtype=torch.int32, device="cuda"), status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    n = min(in_use, M)
    finite = torch.isfinite(want[:n]).all(1)
    assert torch.equal(got[:n][finite], want[:n][finite]) and (got[n:] == 7.0).all()
