"""First-token attention without keys and values (option "cls_pool"): parity with the oracle where sizes can go wrong - the
first size beyond the threshold, batches around the 16, 32 and 64 sequences of a CTA, sequences of one token, one step of 16
keys just full and just begun, the shortest sequences that take the path, a hidden size of 1024 - with branches of one
layer at two depths (their input is a trunk state that outlives its wave), and the same bits in every schedule."""
import numpy as np
import pytest
import torch

from oracle import mt_oracle as orc
from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch, dev_bf16_to_f64, rel_l2
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


@pytest.mark.parametrize("alike", [0.02, 0.1])   # spread of what all tokens share, beside 0.02 of what they do not
@pytest.mark.parametrize("base,B,S", [(BASE, 48, 40), (WIDE, 24, 40)])
def test_no_less_exact_than_over_keys_and_values(base, B, S, alike):
    """A tree that is one layer on the embedding, its FFN zero and its attention output scaled up, so that the state is the
    first token's context and little else: its distance from fp64 (the layer's inputs as the GPU rounds them) is no larger
    than that of the route over keys and values.  5 %: twice the sampling error of a root mean square over 24 x 1024
    roundings is 1 %, one rounding more (of the probabilities or of the mean of the inputs) is 15 % and more."""
    cfg = synth.TreeConfig(hidden=base.hidden, heads=base.heads, ffn=256, trunk_layers=0, vocab_size=2000,
                           tasks=(synth.TaskSpec(0, 1, 2),))
    w = synth.make_weights(cfg, seed=3, random_affine=True)
    layer, H = w["tasks"][0]["layers"][0], cfg.hidden
    rng = np.random.default_rng(7)
    bits = lambda x: synth.f32_to_bf16_bits(np.asarray(x, np.float32))   # noqa: E731
    w["emb"]["type"] = bits(np.broadcast_to(rng.normal(0, alike, H), (cfg.type_vocab, H)))
    layer["wo"] = bits(rng.normal(0, 0.5, (H, H)))
    for name in ("w1", "b1", "w2", "b2"):
        layer[name] = np.zeros_like(layer[name])
    batch = synth.make_batch(cfg, B, S, S // 2, S, seed=2)
    model = mt.MTModel(cfg, B, S, debug_capture=True)
    model.load_weights(synth.pack_weights(cfg, w))
    tok, seg, lens = dev_batch(batch)
    logits = torch.empty(B, cfg.total_classes, device="cuda")
    state = {}
    for pool in (0, 1):
        model.set_option("cls_pool", pool)
        model.forward(tok, seg, lens, logits)
        assert model.poll_status() == 0
        state[pool] = dev_bf16_to_f64(model.debug_hidden(0, 1, B, S)).reshape(B, S, H)[:, 0]
    x = dev_bf16_to_f64(model.debug_hidden(-1, 0, B, S)).reshape(B, S, H)
    wide = synth.widen(w)
    one = wide["tasks"][0]["layers"][0]
    want = np.empty((B, H))
    for b in range(B):
        n = int(batch.lengths[b])
        h0 = orc.embed(batch.token_ids[b, :n], batch.segment_ids[b, :n], wide["emb"], cfg.ln_eps)[0]   # (fp32 residual)
        ctx = orc.attention(x[b, :n], one, cfg.heads)[0]
        h1 = orc.layer_norm(h0 + orc.linear(ctx, one["wo"], one["bo"]), one["ln1_g"], one["ln1_b"], cfg.ln_eps)
        want[b] = orc.layer_norm(h1, one["ln2_g"], one["ln2_b"], cfg.ln_eps)
    over_keys, pooled = rel_l2(state[0], want), rel_l2(state[1], want)
    print(f"rel-L2 of the state: over keys and values {over_keys:.3e}, without {pooled:.3e}")
    assert not np.array_equal(state[0], state[1])   # (the option chose two routes)
    assert pooled <= 1.05 * over_keys
