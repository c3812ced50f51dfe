"""The row-wise quantiser where its short division can go wrong: every row length it holds in registers and one that it does
not, quotients over the whole range of the format (its subnormals and the ties between codes too), zeros of both signs, rows
of zeros, scales outside the range of the short division and of every significand that a scale can have.  Codes and scales
equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from oracle import fp8_oracle as f8
from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(65, 256), (300, 768), (17, 1024), (300, 3072), (9, 4096)])
def test_codes_and_scales_equal_the_oracle(rows, cols):
    rng = np.random.default_rng(cols)
    x = rng.standard_normal((rows, cols)) * np.exp2(rng.integers(-22, 1, (rows, cols)))
    x *= np.exp2(rng.integers(-90, 90, (rows, 1)).astype(np.float64))     # scales inside and outside 2^-60 .. 2^60
    x[1::8] = np.exp2(rng.integers(-14, 9, x[1::8].shape)) * rng.integers(8, 32, x[1::8].shape)   # few significant bits:
    x[1::8, 0] = 448.0 * 32.0                                             # scale 32 exactly, quotients on the ties
    x[2::8, ::3] = 0.0
    x[3::8, ::3] = -0.0
    x[4] = 0.0
    xt = torch.from_numpy(x).to(torch.bfloat16)
    q = torch.zeros(rows, cols, dtype=torch.uint8, device="cuda")
    s = torch.zeros(rows, device="cuda")
    mt.mt_kernel_quantize_rows(xt.cuda(), q, s)
    torch.cuda.synchronize()
    want_q, want_s = f8.quantize_rows(xt.float().numpy().astype(np.float64))
    assert np.array_equal(s.cpu().numpy(), want_s)
    assert np.array_equal(q.cpu().numpy(), want_q)


def test_every_significand_of_a_scale():
    """The scales of the 128 bf16 values of a binade: none has the all-ones significand that the short division cannot take, and
    every bf16 value from 2^-12 to the largest of its row gets the oracle's code (rows of 768: held in registers)."""
    amax = torch.arange(0x3F80, 0x4000, dtype=torch.int32).to(torch.int16).view(torch.bfloat16)
    scale = (amax.float() * np.float32(1.0 / 448.0)).view(torch.int32) & 0x7FFFFF
    assert int(scale.max()) < 0x7FFFFF
    values = torch.arange(0x3980, 0x4000, dtype=torch.int32).to(torch.int16).view(torch.bfloat16)   # 2^-12 .. 2
    for piece in values.split(767):
        rows = torch.zeros(128, 768, dtype=torch.bfloat16)
        rows[:, 0] = amax
        rows[:, 1:1 + len(piece)] = torch.where(piece[None] <= amax[:, None], piece[None], torch.zeros_like(piece[None]))
        q = torch.zeros(128, 768, dtype=torch.uint8, device="cuda")
        s = torch.zeros(128, device="cuda")
        mt.mt_kernel_quantize_rows(rows.cuda(), q, s)
        torch.cuda.synchronize()
        want_q, want_s = f8.quantize_rows(rows.float().numpy().astype(np.float64))
        assert np.array_equal(s.cpu().numpy(), want_s) and np.array_equal(q.cpu().numpy(), want_q)


BASE = synth.TreeConfig(trunk_layers=2, tasks=(synth.TaskSpec(2, 2, 3), synth.TaskSpec(1, 1, 2), synth.TaskSpec(2, 0, 2)))
WIDE = synth.TreeConfig(hidden=1024, heads=16, ffn=4096, trunk_layers=2, vocab_size=2000, tasks=BASE.tasks)


@pytest.mark.parametrize("cfg,B,S", [(BASE, 1, 31), (BASE, 20, 64), (BASE, 48, 128), (WIDE, 5, 128), (WIDE, 41, 128)])
def test_layernorm_that_quantises_gives_the_bits_of_the_separate_launch(cfg, B, S):
    """fused_ln 0: the LayerNorm before the FFN writes the codes (a CTA or a warp per row, by the rows of the launch); 1 and
    3: it is part of the projection (beyond 512 rows) and the rows are quantised by a launch of its own."""
    _, blob, _ = cached_weights(cfg, 5, random_affine=True)
    batch = synth.make_batch(cfg, B, S, max(1, S // 4), S, seed=2)
    model = mt.MTModel(cfg, B, S, fp8_gemm=True)
    model.load_weights(blob)
    out = {}
    for fused in (0, 1, 3):
        model.set_option("fused_ln", fused)
        out[fused] = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
        model.forward(*dev_batch(batch), out[fused])
        torch.cuda.synchronize()
        assert model.poll_status() == 0
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[3])
