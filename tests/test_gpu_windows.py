"""Q/K/V projection + attention in one launch over windows of short sequences (option "qkv_attention"): parity with the
oracle and agreement with the two separate launches where windows can go wrong - one sequence per window, windows that
are exactly full, single-token sequences (128 of them in a window), a last window of one row."""
import numpy as np
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch
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
