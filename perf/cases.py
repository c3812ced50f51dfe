"""What the speed of this framework is measured on: merged multi-task forwards through its public entry points.

A case is one request shape of a serving process: a model tree (a configuration of ``synth``), a padded batch of
token sequences with their valid lengths, the tasks asked for, and the call that is made (``forward`` on device
tensors, ``forward_tokens`` for trees with token-level tasks, ``forward_host`` from and to pinned host buffers).
``prepare`` builds what a server keeps (the model with its weights loaded) and what a request brings (ids, segments,
lengths, the output array); ``run`` is the call.
"""
import math
import struct

import torch

from paper_2107_05377_b200 import binding, synth

MIXED = "ours (mixed, c = 1)"
KD1 = "ours (KD-1)"


def _case(tree, batch, seq, lo, tasks, call="device", fp8=False, expect=False):
    """``lo``: shortest valid length (lengths are uniform in [lo, seq]); ``tasks``: the task mask, 0 for every task;
    ``expect``: the server tells the library how many valid tokens its batches have on average."""
    return {"tree": tree, "batch": batch, "seq": seq, "lo": lo, "tasks": tasks, "call": call, "fp8": fp8, "expect": expect}


def listed():
    cases = {
        # the smallest model and batch of the tests: two short queries, two one-layer branches; launches count
        "tiny_2x32": _case("tiny", 2, 32, 32, 0),
        # one query answered for all eight tasks: the latency of an online service
        "query_1x128": _case("glue8", 1, 128, 128, 0),
        # a handful of short ragged queries for one task, from host buffers to host logits and back: a request of a
        # server without batching (this tree: four shared layers and three of the task's own)
        "one_task_host_3x57": _case("glue8", 3, 57, 9, 1 << 6, call="host"),
        # a small batch, half of the tasks asked for
        "half_tasks_4x128": _case("glue8", 4, 128, 128, 0xE4),
        # the headline benchmark: eight tasks, ragged lengths, inputs resident
        "headline_32x128": _case("glue8", 32, 128, 16, 0, expect=True),
        # one of the paper's own merged trees (33 layers, branches of one to eight layers), odd batch and length
        "mixed_23x101": _case(MIXED, 23, 101, 7, 0),
        # the production-shaped tree: 21 tasks, a third of them token-level
        "production21_32x128": _case("production21", 32, 128, 16, 0),
        # documents: long sequences, ragged
        "long_16x512": _case("glue8", 16, 512, 128, 0),
        # reduced precision (8-bit projections)
        "fp8_64x128": _case("glue8", 64, 128, 16, 0, fp8=True),
        # bulk scoring for one task of the tree
        "bulk_one_task_128x128": _case("glue8", 128, 128, 16, 1 << 7),
        # the wide tree (BERT-large width, 34 layers)
        "large_64x128": _case("large8", 64, 128, 32, 0),
        # the largest batch of the serving sweep, no padding: throughput of bulk processing
        "bulk_256x128": _case("glue8", 256, 128, 128, 0),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def draw(rng):
    tree = rng.choice(["glue8", "glue8", "glue8", "glue8", "tiny", MIXED, KD1, "production21", "large8"])
    layers = {"tiny": 6, "production21": 40, "large8": 34 * 16 / 9, MIXED: 33, KD1: 15}.get(tree, 24)
    seq = int(round(math.exp(rng.uniform(math.log(8), math.log(512)))))
    # at most the tokens of the largest listed case, fewer on the trees with more or wider layers
    most = min(256, int(256 * 128 * 24 / max(24, layers) * 0.9 / seq))
    batch = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    lo = rng.choice([seq, max(1, seq // 8), rng.randint(1, seq)])
    n = _config(tree).n_tasks
    tasks = rng.choice([0, 0, 1 << rng.randrange(n), rng.randrange(1, 1 << n)])
    if tree == "production21":
        return _case(tree, batch, seq, lo, tasks)
    return _case(tree, batch, seq, lo, tasks, call=rng.choice(["device", "device", "host"]),
                 fp8=tree == "glue8" and rng.random() < 0.2, expect=rng.random() < 0.3)


def _config(tree):
    named = {"tiny": synth.config_tiny, "glue8": synth.config_glue8, "large8": synth.config_large8,
             "production21": synth.config_production21}
    return named[tree]() if tree in named else synth.config_paper_tree(tree)


def _active(case, cfg):
    mask = case["tasks"] or (1 << cfg.n_tasks) - 1
    return mask, [t for i, t in enumerate(cfg.tasks) if mask >> i & 1]


def _blob(cfg, nbytes, gen):
    """A weight blob in pinned host memory: matrices, biases and tables N(0, 0.02), LayerNorm gammas N(1, 0.1) and
    betas N(0, 0.1), as the parity tests draw them (here on the GPU, for speed)."""
    body = torch.empty((nbytes - synth.BLOB_HEADER_BYTES) // 2, dtype=torch.bfloat16, device="cuda")
    body.normal_(0.0, 0.02, generator=gen)
    pad = lambda n: (n + 127) // 128 * 128  # noqa: E731  (every tensor starts on 256 bytes)
    at = 0

    def layer():
        nonlocal at
        for name, shape in synth.layer_shapes(cfg).items():
            if name.startswith("ln"):
                body[at:at + shape[0]].mul_(5.0).add_(1.0 if name.endswith("_g") else 0.0)
            at += pad(math.prod(shape))

    H = cfg.hidden
    for rows in (cfg.vocab_size, cfg.max_position, cfg.type_vocab):
        at += pad(rows * H)
    for mean in (1.0, 0.0):
        body[at:at + H].mul_(5.0).add_(mean)
        at += pad(H)
    for _ in range(cfg.trunk_layers):
        layer()
    for t in cfg.tasks:
        for _ in range(t.branch_layers):
            layer()
        at += pad(H * H) + pad(H) + pad(t.num_classes * H) + pad(t.num_classes)
    assert at == body.numel(), "the blob's layout"
    blob = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
    head = struct.pack("<IIIiiiiiiiiiiiiiQ", synth.BLOB_MAGIC, synth.BLOB_VERSION, synth.KIND_FULL, cfg.hidden, cfg.heads,
                       cfg.ffn, cfg.trunk_layers, cfg.vocab_size, cfg.max_position, cfg.type_vocab, cfg.n_tasks, -1,
                       0, 0, 0, 0, nbytes - synth.BLOB_HEADER_BYTES)
    blob[:synth.BLOB_HEADER_BYTES].zero_()
    blob[:len(head)] = torch.frombuffer(bytearray(head), dtype=torch.uint8)
    blob[synth.BLOB_HEADER_BYTES:].copy_(body.view(torch.uint8))
    return blob


def prepare(case, seed):
    cfg = _config(case["tree"])
    B, S = case["batch"], case["seq"]
    mask, _ = _active(case, cfg)
    model = binding.MTModel(cfg, B, S, fp8_gemm=case["fp8"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    model.load_weights(_blob(cfg, model.blob_bytes(), gen))
    if case["expect"]:
        model.set_option("expected_tokens", max(1, B * (case["lo"] + S) // 2))
    batch = synth.make_batch(cfg, B, S, case["lo"], S, seed=seed)
    ids = [torch.from_numpy(a) for a in (batch.token_ids, batch.segment_ids, batch.lengths)]
    shape, token_shape = (B, cfg.total_classes), (B, S, cfg.total_token_classes)
    if case["call"] == "host":
        ids = [a.pin_memory() for a in ids]
        out, token_out = torch.zeros(shape).pin_memory(), None
    else:
        ids = [a.cuda() for a in ids]
        out = torch.zeros(shape, device="cuda") if shape[1] else None
        token_out = torch.zeros(token_shape, device="cuda") if token_shape[2] else None
    return {"model": model, "ids": ids, "mask": mask, "out": out, "token_out": token_out, "call": case["call"]}


def run(state):
    model, out, token_out = state["model"], state["out"], state["token_out"]
    if state["call"] == "host":
        model.forward_host(*state["ids"], out, task_mask=state["mask"])
    elif token_out is not None:
        model.forward_tokens(*state["ids"], out, token_out, task_mask=state["mask"])
    else:
        model.forward(*state["ids"], out, task_mask=state["mask"])
    return {"logits": out, "token_logits": token_out}


def work(case):
    """Valid tokens only (their expected number).  The last layer of a sequence-level branch is needed for the first
    token of a sequence: its key and value projections can be moved to that token's side of the two products, so it
    takes the linear maps on one row per sequence and one query per head over the layer's inputs."""
    cfg = _config(case["tree"])
    _, tasks = _active(case, cfg)
    B, S, lo, H, F = case["batch"], case["seq"], case["lo"], cfg.hidden, cfg.ffn
    n = (lo + S) / 2
    n2 = n * n + ((S - lo + 1) ** 2 - 1) / 12
    depth = max(t.fork_depth for t in tasks)
    first = sum(1 for t in tasks if t.branch_layers and not t.token_level)
    every = depth + sum(t.branch_layers for t in tasks) - first
    row = 2.0 * (4 * H * H + 2 * H * F)
    flops = every * B * (n * row + 4.0 * H * n2) + first * B * (row + 4.0 * H * cfg.heads * n)
    flops += sum(2.0 * B * (n if t.token_level else 1) * t.num_classes * H for t in tasks)
    flops += sum(2.0 * B * H * H for t in tasks if not t.token_level)
    wide, narrow = 4 * H * H + 2 * H * F, 3 * H * H + 2 * H * F
    layer = 2 * wide - (narrow if case["fp8"] else 0)
    weights = (every + first) * layer + sum(2 * t.num_classes * H + (0 if t.token_level else 2 * H * H) for t in tasks)
    outputs = 4 * B * sum(t.num_classes * (n if t.token_level else 1) for t in tasks)
    return {"bytes": weights + 2 * H * (min(B * n, cfg.vocab_size) + min(S, cfg.max_position)) + 4 * B * (2 * S + 1) + outputs,
            "flops": flops}


def tolerance(case):
    # logits after up to 20 layers whose matrix products take bf16 operands (a 1e-2 relative error of the hidden
    # state is what the parity tests allow); 8-bit operands: a few codes in a hundred fall on the other side of a step
    return {"rel": 3e-2, "max": 0.3} if case["fp8"] else {"rel": 1e-2, "max": 0.1}
