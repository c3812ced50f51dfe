"""Attention over tiles of 128 queries and keys: lengths at the edges of tiles, of halves and of the sixteens that an MMA takes,
rows whose maximum grows from tile to tile, values that are not finite in other sequences' rows, and the same bits from every
kernel that a sequence can be given to."""
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch

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


EDGES = [(129, [1, 15, 16, 17, 63, 64, 65, 127, 128, 129]), (200, [200, 144, 145, 192, 193, 33]), (300, [256, 257, 272, 300, 129, 5]),
         (512, [512, 511, 385, 384, 400, 448, 449, 1])]


# up to 128 tokens there is one kernel; beyond, one with two threads per query row (1) and one with one (2: 8-bit projections)
@pytest.mark.parametrize("S,lens,kernel", [(100, [100, 65, 96, 17], 1), (128, [128, 112, 113, 1], 1)] + [e + (k,) for k in (1, 2) for e in EDGES])
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


@pytest.mark.parametrize("growth", [1.0, 1.7])
@pytest.mark.parametrize("S,lens", EDGES)
def test_one_and_two_threads_per_row_have_the_same_bits(S, lens, growth):
    g = torch.Generator(device="cuda").manual_seed(S)
    qkv = torch.randn(len(lens) * S, 3 * 128, device="cuda", generator=g) * 1.3
    tile = torch.arange(S, device="cuda").repeat(len(lens)) // 128
    qkv[:, 128:256] *= growth ** tile[:, None].float()
    two, one = (run(qkv, lens, S, 2, kernel)[1] for kernel in (1, 2))
    assert torch.equal(two, one)


@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("S", [129, 257, 512])
def test_a_short_sequence_has_the_same_bits_at_any_padding(S, kernel):
    lens = [1, 16, 31, 64, 65, 100, 127, 128]
    g = torch.Generator(device="cuda").manual_seed(S)
    qkv = torch.randn(len(lens), S, 3 * 128, device="cuda", generator=g) * 1.5
    wide = run(qkv.view(-1, 3 * 128), lens, S, 2, kernel)[1].view(len(lens), S, 128)
    for seq in (100, 128):
        some = [b for b, n in enumerate(lens) if n <= seq]
        near = run(qkv[some, :seq].reshape(-1, 3 * 128), [lens[b] for b in some], seq, 2)[1].view(len(some), seq, 128)
        for i, b in enumerate(some):
            assert torch.equal(near[i, :lens[b]], wide[b, :lens[b]])


def test_logits_of_short_sequences_do_not_depend_on_a_padding_beyond_128_tokens():
    """(From 65 tokens and more than 512 rows on: below, other choices that may change bits depend on the padded size; with 8-bit
    projections the first-token attention of the last layers has another kernel beyond 128 tokens.)"""
    cfg = synth.TreeConfig(trunk_layers=2, vocab_size=2000, tasks=(synth.TaskSpec(2, 2, 2), synth.TaskSpec(1, 1, 3), synth.TaskSpec(2, 0, 2)))
    _, blob, _ = cached_weights(cfg, 1)
    B = 8
    short = synth.make_batch(cfg, B, 100, 30, 100, seed=3)
    want = None
    for S in (100, 128, 129, 300, 512):
        model = mt.MTModel(cfg, B, S)
        model.load_weights(blob)
        tok, seg, lens = dev_batch(short)
        tok, seg = (torch.nn.functional.pad(t, (0, S - 100)) for t in (tok, seg))
        logits = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
        model.forward(tok.contiguous(), seg.contiguous(), lens, logits)
        torch.cuda.synchronize()
        assert model.poll_status() == 0
        want = logits if want is None else want
        assert torch.equal(logits, want), S
        model.close()
