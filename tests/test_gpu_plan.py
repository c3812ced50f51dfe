"""What a forward launches, read from a captured graph: which kernel carries the residual projections of a plan that does not know
how many of its rows are in use, whether options choose the path that they name, the number of launches that the library
states, and how many CTAs a limit on the SMs leaves each persistent kernel."""
import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, captured_kernels, dev_batch

pytestmark = pytest.mark.gpu

# two layers on all tokens, one per wave, and a last branch layer
ONE = synth.TreeConfig(trunk_layers=2, vocab_size=2000, tasks=(synth.TaskSpec(2, 1, 2),))
WIDE = synth.TreeConfig(hidden=1024, heads=16, ffn=4096, trunk_layers=2, vocab_size=2000, tasks=(synth.TaskSpec(2, 1, 2),))


def model_and_run(cfg, B, S, lo=16, **options):
    _, blob, _ = cached_weights(cfg, 1)
    model = mt.MTModel(cfg, B, S)
    model.load_weights(blob)
    for key, value in options.items():
        model.set_option(key, value)
    batch = synth.make_batch(cfg, B, S, lo, S, seed=4)
    ids = dev_batch(batch)
    logits = torch.empty(B, cfg.total_classes, device="cuda")
    return model, lambda: model.forward(*ids, logits)


# Row blocks that need every branch of the rule for launches of one layer: a single round of narrow tiles, the separate
# projection in one round of its own, narrow tiles in up to 16/9 rounds, pairs that fill their rounds, pairs whose two
# planned rounds are one of use.  (Both ends of 16/9: 25 and 39 blocks at 22 resident clusters.)
@pytest.mark.parametrize("cfg,B,known,kind", [
    (ONE, 20, False, "narrow"), (ONE, 24, False, "separate"), (ONE, 25, False, "narrow"), (ONE, 28, False, "narrow"),
    (ONE, 39, False, "narrow"), (ONE, 40, False, "pair"), (ONE, 48, False, "pair"), (ONE, 64, False, "pair"),
    (ONE, 28, True, "separate"), (ONE, 32, True, "separate"), (ONE, 40, True, "pair"), (ONE, 48, True, "separate"),
    (WIDE, 18, False, "separate"), (WIDE, 24, False, "narrow"), (WIDE, 28, False, "pair"), (WIDE, 32, False, "separate")])
def test_kernel_of_the_residual_projections_of_one_layer(cfg, B, known, kind):
    S = 128
    model, run = model_and_run(cfg, B, S, **({"expected_tokens": B * S} if known else {}))
    names = [name for name, _, _ in captured_kernels(run)]
    count = {"narrow": sum("gemm_ln_tcgen05" in n for n in names), "pair": sum("gemm_ln_pair_tcgen05" in n for n in names)}
    want = {"narrow": 0, "pair": 0}
    if kind != "separate":
        want[kind] = 4                       # attention output and FFN-down of the two layers on all tokens
    assert count == want, names
    assert model.poll_status() == 0


PERSISTENT = ("gemm_bf16_tcgen05", "gemm_ln_tcgen05", "gemm_ln_pair_tcgen05", "qkv_attention_tcgen05")


@pytest.mark.parametrize("cfg,B,S,fused_ln", [(ONE, 28, 128, 2), (ONE, 48, 128, 2), (ONE, 48, 128, 1), (ONE, 48, 128, 3), (WIDE, 28, 128, 3),
                                              (ONE, 64, 64, 0)])
def test_sm_limit_holds_for_every_persistent_kernel(cfg, B, S, fused_ln):
    limit = 40
    model, run = model_and_run(cfg, B, S, fused_ln=fused_ln, sm_limit=limit)
    seen = {}
    for name, grid, _ in captured_kernels(run):
        for kind in PERSISTENT:
            if kind in name:
                seen[kind] = max(seen.get(kind, 0), grid[0] * grid[1] * grid[2])
    assert seen and max(seen.values()) <= limit, seen
    assert model.poll_status() == 0


def test_a_limit_of_one_sm_computes_the_same():
    """96 x 128 rows are projected on CTA pairs, of which one SM holds none: one pair runs all the same."""
    model, _ = model_and_run(ONE, 96, 128)
    batch = synth.make_batch(ONE, 96, 128, 16, 128, seed=4)
    out = {}
    for limit in (1, 0):
        model.workspace.zero_()              # (no earlier forward's activations)
        model.set_option("sm_limit", limit)
        out[limit] = torch.full((96, ONE.total_classes), float("nan"), device="cuda")
        model.forward(*dev_batch(batch), out[limit])
        torch.cuda.synchronize()
        assert model.poll_status() == 0
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


# branches of one, two and three layers at three depths, a task on the trunk, a token-level one; more than eight tails
TREE = synth.TreeConfig(trunk_layers=3, vocab_size=2000, tasks=(
    synth.TaskSpec(1, 1, 3), synth.TaskSpec(2, 1, 2), synth.TaskSpec(2, 3, 2), synth.TaskSpec(3, 2, 2), synth.TaskSpec(2, 0, 2),
    synth.TaskSpec(1, 2, 3, token_level=True)) + (synth.TaskSpec(3, 1, 2),) * 6)


@pytest.mark.parametrize("B,S", [(2, 50), (40, 17), (6, 100), (20, 128)])   # few rows, windows, pooled first tokens, both sizes of it
@pytest.mark.parametrize("options", [{}, {"cls_pool": 0}, {"qkv_attention": 0}, {"early_heads": 1}, {"cls_only_last_layer": 0},
                                     {"fused_ln": 0}, {"fused_ln": 3}, {"fp8_gemm": 1}, {"max_groups": 2}, {"ffn_down_split": 0}])
def test_stated_launches_are_those_of_a_captured_forward(B, S, options):
    cfg, options = TREE, dict(options)
    _, blob, _ = cached_weights(cfg, 1)
    model = mt.MTModel(cfg, B, S, fp8_gemm=bool(options.pop("fp8_gemm", 0)), max_groups=options.pop("max_groups", None))
    model.load_weights(blob)
    for key, value in options.items():
        model.set_option(key, value)
    ids = dev_batch(synth.make_batch(cfg, B, S, 1, S, seed=4))
    logits = torch.empty(B, cfg.total_classes, device="cuda")
    token_logits = torch.empty(B, S, cfg.total_token_classes, device="cuda")
    names = [name for name, _, _ in captured_kernels(lambda: model.forward_tokens(*ids, logits, token_logits))]
    assert model.plan_launches(model.full_mask()) == len(names), names
    bf16 = model.weights_bytes() == mt.MTModel(cfg, B, S, bind=False).weights_bytes()
    pooled = bf16 and B * S > 512 and 3 * S >= 2 * cfg.heads and options.get("cls_pool", 1) and options.get("cls_only_last_layer", 1)
    windows = bf16 and B * S >= 256 and S <= 64 and options.get("qkv_attention", 1)
    assert any("cls_pool_kernel" in n for n in names) == bool(pooled)
    assert any("qkv_attention_tcgen05" in n for n in names) == bool(windows)
    model.set_option("profile", 1)
    model.forward_tokens(*ids, logits, token_logits)
    assert sum(n for _, n in model.profile_read().values()) == len(names) - 1   # (the row starts are not timed)
    assert model.poll_status() == 0
