"""Forwards of few rows: low GEMM tiles (64 and 32 rows), projections as partial sums, a LayerNorm CTA per row.  Parity with
the oracle at every hidden state where the sizes can go wrong: a single row, tiles just full and just begun, the last
size before full tiles and the first after, and a hidden size of 1024 (more k-blocks than the ring of stages holds);
and the same bits from run to run."""
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
