"""Forwards of a plan in frequent use run as a CUDA graph (option "replay"): the same bits as launched kernels, with the pointers of
each call, whatever comes between the calls - and they do run as one, from the call on that the plan has been launched often enough."""
import ctypes as C
import threading

import pytest
import torch

from paper_2107_05377_b200 import binding as mt
from paper_2107_05377_b200 import synth
from gpu_util import cached_weights, dev_batch

pytestmark = pytest.mark.gpu

LAUNCHED = 32     # times that a plan is launched kernel by kernel first

# sequence- and token-level tasks, a task that pools the trunk, first-token attention of both kinds by batch size
TREE = synth.TreeConfig(trunk_layers=3, vocab_size=2000,
                        tasks=(synth.TaskSpec(2, 2, 2), synth.TaskSpec(3, 0, 3), synth.TaskSpec(1, 1, 4, token_level=True),
                               synth.TaskSpec(1, 2, 1)))


def models(B, S):
    _, blob, _ = cached_weights(TREE, 1)
    out = []
    for replay in (1, 0):
        m = mt.MTModel(TREE, B, S)
        m.load_weights(blob)
        m.set_option("replay", replay)
        out.append(m)
    return out


def call(model, ids, mask=None, stream=None):
    B, S = ids[0].shape
    out = torch.zeros(B, TREE.total_classes, device="cuda"), torch.zeros(B, S, TREE.total_token_classes, device="cuda")
    torch.cuda.synchronize()     # (the zeros are there before another stream writes)
    model.forward_tokens(*ids, *out, task_mask=mask, stream=stream)
    return out


def same(a, b):
    torch.cuda.synchronize()
    return all(torch.equal(x, y) for x, y in zip(a, b))


# few rows; more than 512 (pooled first-token attention on the second stream); windows
@pytest.mark.parametrize("B,S", [(2, 40), (6, 128), (9, 60)])
def test_replayed_and_launched_forwards_have_the_same_bits(B, S):
    often, plain = models(B, S)
    inputs = [dev_batch(synth.make_batch(TREE, B, S, 1, S, seed=k)) for k in range(3)]
    want = [call(plain, ids) for ids in inputs]
    other = torch.cuda.Stream()
    for k in range(LAUNCHED + 32):   # (new output arrays in every call)
        assert same(call(often, inputs[k % 3], stream=other if k % 5 == 4 else None), want[k % 3]), k
        assert often.replayed_forwards() == max(0, k + 1 - LAUNCHED)
    # calls in a row, unsynchronised, on buffers that change under the same graph
    outs = [call(often, inputs[k % 3]) for k in range(7)]
    assert all(same(outs[k], want[k % 3]) for k in range(7))
    assert often.replayed_forwards() == 32 + 7 and plain.replayed_forwards() == 0
    assert often.poll_status() == 0


def test_captures_options_and_other_plans_between_replays():
    B, S = 3, 40
    often, plain = models(B, S)
    ids = dev_batch(synth.make_batch(TREE, B, S, 1, S, seed=5))
    want = call(plain, ids)
    for _ in range(LAUNCHED + 4):
        got = call(often, ids)
    assert same(got, want) and often.replayed_forwards() == 4
    # the caller's own capture records the kernels themselves
    graph, outs = torch.cuda.CUDAGraph(), (torch.zeros_like(want[0]), torch.zeros_like(want[1]))
    with torch.cuda.graph(graph):
        often.forward_tokens(*ids, *outs)
    assert often.replayed_forwards() == 4
    graph.replay()
    assert same(outs, want) and same(call(often, ids), want) and often.replayed_forwards() == 5
    # events of tasks and per-launch timing lie between the launches
    out = (torch.zeros_like(want[0]), torch.zeros_like(want[1]))
    events = [torch.cuda.Event() for _ in TREE.tasks]
    for e in events:
        e.record()
    torch.cuda.synchronize()
    rc = mt.lib().mt_forward_tokens(often.handle, *(t.data_ptr() for t in ids), often.full_mask(), B, S, *(t.data_ptr() for t in out),
                                    (C.c_void_p * len(events))(*(e.cuda_event for e in events)), None)
    assert rc == 0 and same(out, want) and often.replayed_forwards() == 5
    often.set_option("profile", 1)
    assert same(call(often, ids), want) and often.replayed_forwards() == 5
    often.set_option("profile", 0)
    assert same(call(often, ids), want) and often.replayed_forwards() == 6
    # a bad length in a replayed forward is flagged as in a launched one
    bad = ids[2].clone()
    bad[1] = S + 3
    call(often, (ids[0], ids[1], bad))
    assert often.poll_status() & 4
    # plans dropped while replays may be under way: by the cache's limit, by an option
    often.set_option("plan_cache", 1)
    for mask in (1, 2, 1, 15):
        expect = call(plain, ids, mask)
        before = often.replayed_forwards()
        for _ in range(LAUNCHED + 2):
            got = call(often, ids, mask)
        assert same(got, expect) and often.replayed_forwards() == before + 2
    often.set_option("overlap_cls", 0)
    assert same(call(often, ids), want)
    often.close()


def test_a_callers_capture_outlives_what_becomes_of_graphs_meanwhile():
    """While a stream is being captured (in the mode that forbids what might disturb it, from every thread), forwards on another
    stream are made a graph, replayed with new pointers and dropped, and the captured forward itself drops one."""
    B, S = 3, 40
    often, plain = models(B, S)
    inputs = [dev_batch(synth.make_batch(TREE, B, S, 1, S, seed=k)) for k in range(2)]
    short = dev_batch(synth.make_batch(TREE, B, 25, 1, 25, seed=7))
    want, want_short = [call(plain, ids) for ids in inputs], call(plain, short)
    often.set_option("plan_cache", 1)
    for _ in range(LAUNCHED):
        call(often, inputs[0])
    outs = [(torch.zeros_like(want[0][0]), torch.zeros_like(want[0][1])) for _ in range(4)]
    out_short = [tuple(torch.zeros_like(t) for t in want_short) for _ in range(2)]
    other, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        plain.forward_tokens(*inputs[0], *outs[3])
        for k in range(3):
            often.forward_tokens(*inputs[k % 2], *outs[k], stream=other)
        assert often.replayed_forwards() == 3
        often.forward_tokens(*short, *out_short[0], stream=other)
        for _ in range(LAUNCHED + 1):
            often.forward_tokens(*inputs[0], *outs[2], stream=other)
        assert often.replayed_forwards() == 4
        often.forward_tokens(*short, *out_short[1])     # captured: drops the graph under way
    torch.cuda.synchronize()
    assert all(same(outs[k], want[k % 2]) for k in range(3)) and same(out_short[0], want_short)
    graph.replay()
    assert same(outs[3], want[0]) and same(out_short[1], want_short)
    assert often.poll_status() == 0


def test_graphs_are_built_beside_a_thread_that_waits_for_the_device():
    """A wait for the whole device fails while any stream is being captured, so a graph is not built by capturing one."""
    cfg = synth.config_tiny()
    _, blob, _ = cached_weights(cfg, 0)
    model = mt.MTModel(cfg, 1, 24)
    model.load_weights(blob)
    ids = [dev_batch(synth.make_batch(cfg, 1, S, S, S, seed=S)) for S in range(1, 25)]
    out = torch.zeros(1, cfg.total_classes, device="cuda")
    errors, waits, done = [], [0], threading.Event()

    def wait():
        try:
            while not done.is_set():
                torch.cuda.synchronize()
                waits[0] += 1
        except Exception as e:   # noqa: BLE001
            errors.append(e)
    thread = threading.Thread(target=wait)
    thread.start()
    for rep in range(4):
        for one in ids:
            for _ in range(LAUNCHED + 1):
                model.forward(*one, out)
        assert model.replayed_forwards() == (rep + 1) * len(ids)
        model.set_option("replay", 1)        # (drops the plans: the graphs are built anew)
    done.set()
    thread.join()
    assert not errors and waits[0] > 0
    assert model.poll_status() == 0


def test_a_model_has_at_most_32_graphs():
    cfg = synth.config_tiny()
    _, blob, _ = cached_weights(cfg, 0)
    model = mt.MTModel(cfg, 1, 33)
    model.load_weights(blob)
    model.set_option("plan_cache", 64)
    ids = [dev_batch(synth.make_batch(cfg, 1, S, S, S, seed=S)) for S in range(1, 34)]
    out = torch.zeros(1, cfg.total_classes, device="cuda")
    for k, one in enumerate(ids):
        for _ in range(LAUNCHED + 1):
            model.forward(*one, out)
        assert model.replayed_forwards() == k + 1
    assert model.plan_cache_size() == 33
    # the first one's graph went when the last one's was built, the others are there
    for k in (1, 32, 0, 2):
        before = model.replayed_forwards()
        model.forward(*ids[k], out)
        assert model.replayed_forwards() == before + (k != 0)
    torch.cuda.synchronize()
    assert model.poll_status() == 0


def test_host_calls_are_replayed_too():
    cfg = synth.config_tiny()
    _, blob, _ = cached_weights(cfg, 0)
    B, S = 2, 32
    model = mt.MTModel(cfg, B, S)
    model.load_weights(blob)
    batches = [synth.make_batch(cfg, B, S, 1, S, seed=k) for k in range(2)]
    want = []
    for k in range(LAUNCHED + 24):
        b = batches[k % 2]
        out = torch.zeros(B, cfg.total_classes).pin_memory()
        model.forward_host(*[torch.from_numpy(a).pin_memory() for a in (b.token_ids, b.segment_ids, b.lengths)], out)
        if k < 2:
            want.append(out)
        assert torch.equal(out, want[k % 2]), k
    assert model.replayed_forwards() == 24
