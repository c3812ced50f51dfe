"""Forwards of few rows: GEMM tiles of 16, 32 and 64 rows taken transposed, the attention output with its LayerNorm on such tiles, the
FFN-down projection as partial sums, a LayerNorm CTA per row.  Parity with the oracle at every hidden state where the sizes can go
wrong: a single row, tiles just full and just begun, the last size before full tiles and the first after, and a hidden size of 1024
(more k-blocks than the ring of stages holds); and the same bits from run to run."""
import numpy as np
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch
from test_gpu_forward import check_against_oracle

pytestmark = pytest.mark.gpu

TASKS = (synth.TaskSpec(2, 2, 3), synth.TaskSpec(1, 1, 2), synth.TaskSpec(2, 0, 2))
BASE = synth.TreeConfig(trunk_layers=2, tasks=TASKS)
WIDE = synth.TreeConfig(hidden=1024, heads=16, ffn=4096, trunk_layers=2, vocab_size=2000, tasks=TASKS)


@pytest.mark.parametrize("cfg,B,S", [(BASE, 1, 1), (BASE, 1, 31), (BASE, 2, 16), (BASE, 1, 33), (BASE, 2, 32), (BASE, 1, 65),
                                     (BASE, 4, 128), (BASE, 4, 129), (WIDE, 1, 32), (WIDE, 1, 100)])
def test_forwards_of_few_rows_match_the_oracle(cfg, B, S):
    w, blob, wf = cached_weights(cfg, 5, random_affine=True)
    batch = synth.make_batch(cfg, B, S, max(1, S // 4), S, seed=8 + B)
    model = mt.MTModel(cfg, B, S, debug_capture=True)
    model.load_weights(blob)
    tok, seg, lens = dev_batch(batch)
    logits = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
    model.forward(tok, seg, lens, logits)
    torch.cuda.synchronize()
    assert model.poll_status() == 0
    check_against_oracle(cfg, wf, batch, model, logits, rows=range(B))
    again = torch.empty_like(logits)
    for _ in range(5):
        model.forward(tok, seg, lens, again)
        torch.cuda.synchronize()
        assert torch.equal(again, logits)


@pytest.mark.parametrize("cfg,B,S", [(BASE, 1, 8), (BASE, 3, 57), (BASE, 4, 128), (WIDE, 1, 100)])
def test_only_the_ffn_down_projection_is_summed_range_by_range(cfg, B, S):
    """With FFN-down weights of zero its partial sums are zero in every order, so option "ffn_down_split" must not change a
    bit: the attention-output projection of a launch of few rows is summed over K in one sequence like every other."""
    w = synth.make_weights(cfg, seed=5, random_affine=True)
    for layer in w["trunk"] + [one for task in w["tasks"] for one in task["layers"]]:
        layer["w2"] = np.zeros_like(layer["w2"])
    batch = synth.make_batch(cfg, B, S, max(1, S // 4), S, seed=8)
    model = mt.MTModel(cfg, B, S)
    model.load_weights(synth.pack_weights(cfg, w))
    out = {}
    for split in (0, 1):
        model.set_option("ffn_down_split", split)
        out[split] = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
        model.forward(*dev_batch(batch), out[split])
        torch.cuda.synchronize()
        assert model.poll_status() == 0
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("rows,hidden,n_parts", [(1, 768, 1), (512, 1024, 4), (4736, 768, 2), (4737, 768, 3)])
def test_rows_put_together_from_partial_sums_at_any_number_of_rows(rows, hidden, n_parts):
    """residual + ((part_0 + part_1 + ...) + bias), in this order and in fp32, then the LayerNorm: the bits of the plain kernel on
    the sum formed here, also beyond the rows up to which the plain kernel takes a CTA per row (4736)."""
    gen = torch.Generator(device="cuda").manual_seed(rows)
    rnd = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)   # noqa: E731
    pitch = (rows + 127) // 128 * 128
    part, residual = rnd(n_parts * pitch, hidden), rnd(rows, hidden)
    bias, gamma, beta = (rnd(hidden).bfloat16() for _ in range(3))
    y, y32, want, want32 = (torch.full((rows, hidden), float("nan"), dtype=t, device="cuda")
                            for t in (torch.bfloat16, torch.float32) * 2)
    mt.mt_kernel_layernorm_partial(part, n_parts, pitch, residual, bias, gamma, beta, y, 1e-12, y_f32=y32)
    total = part[:rows].clone()
    for s in range(1, n_parts):
        total += part[s * pitch:s * pitch + rows]
    mt.mt_kernel_layernorm(residual + (total + bias.float()), gamma, beta, want, 1e-12, y_f32=want32)
    torch.cuda.synchronize()
    assert torch.equal(y, want) and torch.equal(y32, want32)
