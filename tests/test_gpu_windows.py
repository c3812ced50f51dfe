"""Q/K/V projection + attention in one launch over windows of short sequences (option "qkv_attention"): parity with the
oracle and agreement with the two separate launches where windows can go wrong - one sequence per window, windows that
are exactly full, single-token sequences (128 of them in a window), a last window of one row - and where a CTA takes many units
(window, layer, head): both accumulators, the four sets of biases, the next window's rows asked for a unit ahead."""
import numpy as np
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, captured_kernels, dev_batch, rel_l2
from test_gpu_forward import check_against_oracle

pytestmark = pytest.mark.gpu


def lengths_of(kind, B, S):
    rng = np.random.default_rng(B * 1000 + S)
    return {"full": np.full(B, S), "ones": np.ones(B), "ragged": rng.integers(1, S + 1, B),
            "last_alone": np.array([S] * (B - 1) + [1])}[kind].astype(np.int32)


@pytest.mark.parametrize("B,S,kind", [(4, 64, "full"), (5, 64, "last_alone"), (9, 43, "ragged"), (300, 1, "ones"),
                                      (130, 2, "ones"), (8, 33, "full"), (40, 17, "ragged")])
def test_windows_match_oracle_and_separate_launches(B, S, kind):
    cfg = synth.TreeConfig(trunk_layers=2, tasks=(synth.TaskSpec(2, 2, 3), synth.TaskSpec(1, 1, 2), synth.TaskSpec(2, 0, 2)))
    w, blob, wf = cached_weights(cfg, 5, random_affine=True)
    lens = lengths_of(kind, B, S)
    batch = synth.make_batch(cfg, B, S, 1, S, seed=3)
    batch.lengths[:] = lens
    out = {}
    for fused in (1, 0):
        model = mt.MTModel(cfg, B, S, debug_capture=True)
        model.set_option("qkv_attention", fused)
        model.load_weights(blob)
        logits = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
        tok, seg, dev_lens = dev_batch(batch)   # (the lengths stay alive: the captured states are unpacked by them)
        model.forward(tok, seg, dev_lens, logits)
        torch.cuda.synchronize()
        assert model.poll_status() == 0
        rows = sorted({0, 1, B // 2, B - 2, B - 1})
        check_against_oracle(cfg, wf, batch, model, logits, rows=rows)
        out[fused] = logits
    # bf16 probabilities and context rounded once either way: the bound is that of two roundings of the packed layout
    assert float((out[1] - out[0]).abs().max()) <= 2e-3


# four layers on all tokens in the second wave
MANY = (synth.TaskSpec(1, 2, 2), synth.TaskSpec(1, 2, 3), synth.TaskSpec(1, 2, 2), synth.TaskSpec(2, 0, 2))
DEEP = synth.TreeConfig(trunk_layers=2, vocab_size=2000, tasks=MANY)
WIDE = synth.TreeConfig(hidden=1024, heads=16, ffn=4096, trunk_layers=2, vocab_size=2000, tasks=MANY)


@pytest.mark.parametrize("cfg,B,S,lo", [(DEEP, 256, 16, 16), (DEEP, 256, 64, 64), (DEEP, 256, 64, 1), (WIDE, 100, 64, 8)])
def test_ctas_that_take_many_units(cfg, B, S, lo):
    w, blob, wf = cached_weights(cfg, 5, random_affine=True)
    batch = synth.make_batch(cfg, B, S, lo, S, seed=3)
    windows, filled = 1, 0
    for n in batch.lengths:              # next fit, as the row starts are laid out
        windows, filled = (windows + 1, n) if filled + n > 128 else (windows, filled + n)
    ids = dev_batch(batch)
    model = mt.MTModel(cfg, B, S, debug_capture=True)
    model.load_weights(blob)
    logits = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
    grids = [grid[0] for name, grid, _ in captured_kernels(lambda: model.forward(*ids, logits)) if "qkv_attention" in name]
    assert windows * 4 * cfg.heads >= 5 * max(grids), "a CTA takes five units or more, so that the sets of biases wrap"
    model.forward(*ids, logits)
    torch.cuda.synchronize()
    assert model.poll_status() == 0
    check_against_oracle(cfg, wf, batch, model, logits, rows=sorted({0, 1, B // 2, B - 2, B - 1}))
    for _ in range(5):
        again = torch.full_like(logits, float("nan"))
        model.forward(*ids, again)
        torch.cuda.synchronize()
        assert torch.equal(again, logits)
    model.set_option("qkv_attention", 0)
    apart = torch.full_like(logits, float("nan"))
    model.forward(*ids, apart)
    # each route is within 5e-3 of fp64 on the logits of a whole batch (a few bf16 roundings per layer, three layers)
    assert rel_l2(logits.cpu().double().numpy(), apart.cpu().double().numpy()) <= 1e-2
    # a task alone gets the bits that it gets in the tree
    for task in (0, 1):
        alone = mt.MTModel(synth.config_single_task(cfg, task), B, S)
        alone.load_weights(synth.pack_weights(alone.cfg, synth.select_task_weights(w, task)))
        mine = torch.full((B, alone.cfg.total_classes), float("nan"), device="cuda")
        alone.forward(*ids, mine)
        torch.cuda.synchronize()
        at = cfg.logit_offsets[task]
        assert torch.equal(mine, logits[:, at:at + alone.cfg.total_classes])


@pytest.mark.parametrize("B,S", [(16, 40), (300, 3)])
def test_values_that_are_not_finite_stay_in_their_sequence(B, S):
    """One sequence holds a token whose embedding is NaN: its own logits are NaN, and those of the sequences that share its
    windows are what they are without it."""
    cfg = synth.TreeConfig(trunk_layers=2, vocab_size=2000, tasks=(synth.TaskSpec(2, 2, 3), synth.TaskSpec(2, 0, 2)))
    w = synth.make_weights(cfg, seed=5, random_affine=True)
    w["emb"]["word"][1500] = 0x7FC0
    model = mt.MTModel(cfg, B, S)
    model.load_weights(synth.pack_weights(cfg, w))
    batch = synth.make_batch(cfg, B, S, 2, S, seed=3)
    batch.token_ids[batch.token_ids == 1500] = 1501
    out = {}
    for token in (1501, 1500, 1501):          # (and nothing of it is left for the next forward)
        batch.token_ids[3, 1] = token
        logits = torch.full((B, cfg.total_classes), float("inf"), device="cuda")
        model.forward(*dev_batch(batch), logits)
        torch.cuda.synchronize()
        assert model.poll_status() == 0
        if token in out:
            assert torch.equal(out[token], logits)
        out[token] = logits
    others = [b for b in range(B) if b != 3]
    assert torch.isfinite(out[1501]).all()
    assert torch.equal(out[1500][others], out[1501][others])
    assert torch.isnan(out[1500][3]).all()
