"""First-token attention without keys and values (option "cls_pool"): parity with the oracle where sizes can go wrong - the
first size beyond the threshold, batches around the 16, 32 and 64 sequences of a CTA, sequences of one token, one step of 16
keys just full and just begun, the shortest sequences that take the path, a hidden size of 1024 - with branches of one
layer at two depths (their input is a trunk state that outlives its wave), and the same bits in every schedule."""
import numpy as np
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch
from test_gpu_forward import check_against_oracle

pytestmark = pytest.mark.gpu

TASKS = (synth.TaskSpec(1, 1, 3), synth.TaskSpec(2, 1, 2), synth.TaskSpec(2, 3, 2), synth.TaskSpec(3, 2, 2), synth.TaskSpec(1, 1, 2),
         synth.TaskSpec(2, 0, 2))
BASE = synth.TreeConfig(trunk_layers=3, tasks=TASKS)
WIDE = synth.TreeConfig(hidden=1024, heads=16, ffn=4096, trunk_layers=3, vocab_size=2000, tasks=TASKS)
EDGES = (1, 15, 16, 17, 31, 32, 33, 48, 49)


@pytest.mark.parametrize("cfg,B,S", [(BASE, 4, 129), (BASE, 3, 200), (BASE, 16, 49), (BASE, 17, 33), (BASE, 33, 16), (BASE, 65, 8),
                                     (WIDE, 6, 100), (WIDE, 47, 11)])
def test_first_token_attention_matches_the_oracle_in_every_schedule(cfg, B, S):
    w, blob, wf = cached_weights(cfg, 5, random_affine=True)
    batch = synth.make_batch(cfg, B, S, 1, S, seed=4)
    batch.lengths[:] = np.array([min(EDGES[b % len(EDGES)], S) if b else S for b in range(B)], np.int32)
    model = mt.MTModel(cfg, B, S, debug_capture=True)
    model.load_weights(blob)
    tok, seg, lens = dev_batch(batch)
    logits = torch.full((B, cfg.total_classes), float("nan"), device="cuda")
    model.forward(tok, seg, lens, logits)
    torch.cuda.synchronize()
    assert model.poll_status() == 0
    check_against_oracle(cfg, wf, batch, model, logits, rows=sorted({0, 1, 2, B // 2, B - 2, B - 1}))
    # beside the other waves or in line with them, with the tails at the end or each after its wave
    for option, value, usual in (("overlap_cls", 0, 1), ("early_heads", 1, 0), ("overlap_cls", 1, 1)):
        model.set_option(option, value)
        again = torch.full_like(logits, float("nan"))
        model.forward(tok, seg, lens, again)
        torch.cuda.synchronize()
        assert torch.equal(again, logits), option
        model.set_option(option, usual)
    model.set_option("cls_pool", 0)
    other = torch.full_like(logits, float("nan"))
    model.forward(tok, seg, lens, other)
    check_against_oracle(cfg, wf, batch, model, other, rows=[0, 1, B - 1])
