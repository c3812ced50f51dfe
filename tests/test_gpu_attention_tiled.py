"""Attention over tiles of 128 queries and keys: lengths at the edges of tiles, of halves and of the sixteens that an MMA takes,
rows whose maximum grows from tile to tile by more and by less than the exponentials may lag, and values that are not finite in
other sequences' rows."""
import pytest
import torch

from paper_2107_05377_b200 import binding as mt

pytestmark = pytest.mark.gpu


def run(qkv, lens, S, heads, kernel=1):
    B, H = len(lens), heads * 64
    x = qkv.to(torch.bfloat16)
    for b, n in enumerate(lens):
        x[b * S + n:(b + 1) * S] = float("nan")
    ctx = torch.full((B * S, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    mt.mt_kernel_attention(x, torch.tensor(lens, dtype=torch.int32, device="cuda"), ctx, B, S, heads, tensor_memory=kernel, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return x, ctx


def check(x, ctx, lens, S, heads):
    H = heads * 64
    for b, n in enumerate(lens):
        q, k, v = (x[b * S:b * S + n, i * H:(i + 1) * H].double().view(n, heads, 64).transpose(0, 1) for i in range(3))
        p = torch.softmax(q @ k.transpose(1, 2) / 8.0, -1)
        want = (p @ v).transpose(0, 1).reshape(n, H)
        got = ctx[b * S:b * S + n].double()
        assert torch.isfinite(got).all()
        # probabilities and results rounded to bf16: 2^-9 relative per term of a sum whose terms have |v| for a bound
        assert ((got - want).norm() / want.norm()).item() <= 5e-3
        bound = (p @ v.abs()).transpose(0, 1).reshape(n, H) * 2 ** -8 + want.abs() * 2 ** -8 + 1e-5
        assert ((got - want).abs() <= bound).all()
        assert (ctx[b * S + n:(b + 1) * S] == 0).all(), "padded query rows must be written as zero"


@pytest.mark.parametrize("kernel", [1, 2])     # two threads per query row; one (with 8-bit projections)
@pytest.mark.parametrize("S,lens", [(100, [100, 65, 96, 17]), (128, [128, 112, 113, 1]), (129, [1, 15, 16, 17, 63, 64, 65, 127, 128, 129]), (200, [200, 144, 145, 192, 193, 33]),
                                    (300, [256, 257, 272, 300, 129, 5]), (512, [512, 511, 385, 384, 400, 448, 449, 1])])
def test_lengths_at_every_edge(S, lens, kernel):
    g = torch.Generator(device="cuda").manual_seed(S)
    qkv = torch.randn(len(lens) * S, 3 * 128, device="cuda", generator=g) * 1.5
    x, ctx = run(qkv, lens, S, 2, kernel)
    check(x, ctx, lens, S, 2)


@pytest.mark.parametrize("growth", [1.0, 1.7, 4.0])   # of the keys from tile to tile; scores of the first: standard deviation 2
def test_maxima_that_grow_from_tile_to_tile(growth):
    S, lens = 512, [512, 470, 260]
    g = torch.Generator(device="cuda").manual_seed(9)
    qkv = torch.randn(len(lens) * S, 3 * 64, device="cuda", generator=g) * 1.4
    tile = torch.arange(S, device="cuda").repeat(len(lens)) // 128
    qkv[:, 64:128] *= growth ** tile[:, None].float()
    qkv[::3, :64] *= -1.0
    x, ctx = run(qkv, lens, S, 1)
    check(x, ctx, lens, S, 1)
