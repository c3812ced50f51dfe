#!/usr/bin/env python
"""Throughput of the merged multi-task forward pass: the 8-task BERT-base tree at
batch 32 x seq 128 (valid lengths uniform in [16, 128]), sequences per second.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

A step is one mt_forward over one synthetic batch (all 24 transformer layers of the
tree, embeddings, poolers and heads).  Prints ONE JSON line (rank 0).  With N > 1
(launched by torch.distributed.run) every rank runs an independent replica on its own
GPU - sequences are independent, the path has no exchange step - and the value is the
sum over ranks divided by the slowest rank's time.

--impl reference times the fp64 CPU oracle on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from paper_2107_05377_b200 import synth  # noqa: E402

METRIC = "8-task BERT-base seq/s (seq128, b32)"
UNIT = "sequences/s"
BATCH, SEQ, LEN_LO, LEN_HI = 32, 128, 16, 128
N_INPUT_BATCHES = 4
REFERENCE_SAMPLE = 8          # sequences per step of the oracle arm
L2_FLUSH_BYTES = 256 << 20    # larger than the 126 MB L2

# DRAM traffic of the dominant kernel comes from one ncu capture (bytes per launch, averaged over the GEMM
# launches of the forwards of `bench.py --steps 2`); the figure and the digest of the kernel sources it was
# taken on are two lines of the launch-list summary under profiles/, and it is reported only while the
# sources still have that digest.
GEMM_SOURCES = ("gemm_tcgen05.cu", "gemm_ln_tcgen05.cu", "gemm_ln_pair_tcgen05.cu", "gemm_ln_low_tcgen05.cu", "gemm_low_tcgen05.cu",
                "gemm_low.cuh", "cluster_ptx.cuh", "tc_ptx.cuh", "rowwise.cuh")
TRAFFIC_SUMMARY = os.path.join("profiles", "bench_glue8_b32_s128_launch_list.md")
NOMINAL_BF16_TFLOPS = 2250.0   # dense bf16 of the part, for context beside the measured peak
STEADY_SECONDS = 2.0


def ncu_traffic():
    """(digest, bytes per GEMM launch) as recorded in the launch-list summary, or (None, None)."""
    import re
    try:
        with open(os.path.join(ROOT, TRAFFIC_SUMMARY)) as f:
            text = f.read()
    except OSError:
        return None, None
    d = re.search(r"gemm_sources_sha256:\s*`?([0-9a-f]{64})", text)
    b = re.search(r"gemm_dram_bytes_per_launch:\s*`?(\d+)", text)
    return (d.group(1), int(b.group(1))) if d and b else (None, None)


def gemm_sources_digest():
    h = hashlib.sha256()
    for name in GEMM_SOURCES:
        with open(os.path.join(ROOT, "paper_2107_05377_b200", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {"tflops": float(p.get("bf16_tflops_sustained", p.get("bf16_tflops"))), "hbm_gbs": float(p["hbm_gbs"]),
                "source": "measured (sustained)"}
    return {"tflops": 1400.0, "hbm_gbs": 6650.0, "source": "fallback"}


def tasks_of(cfg):
    return [(t.fork_depth, t.branch_layers, t.num_classes) for t in cfg.tasks]


def gemm_flops_per_forward(cfg, n_layers, m_rows, first_token_layers=0, batch=0):
    """FLOPs of the four linear maps of n_layers encoder layers over m_rows tokens.  Of those layers,
    first_token_layers (the last layer of each task branch) need the attention output and FFN maps only on the first
    token of each of the `batch` sequences; their attention projects neither keys nor values (see
    first_token_attention_flops)."""
    h, f = cfg.hidden, cfg.ffn
    qkv, rest = 2.0 * 3 * h * h, 2.0 * (h * h + 2 * h * f)
    return (n_layers - first_token_layers) * m_rows * (qkv + rest) + first_token_layers * batch * rest


def first_token_attention_flops(cfg, lengths):
    """FLOPs of one last branch layer's attention for the first tokens of sequences of these lengths: three H x H products
    per sequence (query, query through the key matrix, attended mean through the value matrix) and, per head, a pass over
    the sequence's inputs for the scores and one for the mean."""
    h = cfg.hidden
    return len(lengths) * 2.0 * 3 * h * h + 4.0 * cfg.heads * h * float(lengths.sum())


def oracle_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads", 1) for i in threadpool_info() if i.get("user_api") == "blas"]
        return max(n) if n else 1
    except Exception:
        return os.cpu_count() or 1


def time_oracle(cfg, weights_f64, batch, rows):
    from oracle import mt_oracle as orc
    t0 = time.perf_counter()
    orc.forward_batch_mt(batch.token_ids, batch.segment_ids, batch.lengths, weights_f64, tasks_of(cfg), cfg.heads,
                         cfg.ln_eps, rows=rows)
    return time.perf_counter() - t0


class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap,utilization.gpu")

    def __init__(self, device_index: int):
        self.file = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                                          "-lms", "50", "-i", str(device_index)], stdout=self.file,
                                         stderr=subprocess.DEVNULL)
        except OSError:
            pass

    def stop(self):
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        if self.proc is None:
            return out
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.file.flush()
        self.file.seek(0)
        sm, mx, reasons, busy = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.file.read().splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            try:
                busy.append(float(parts[9]) >= 50.0)
            except (ValueError, IndexError):
                busy.append(True)
            for name, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        self.file.close()
        os.unlink(self.file.name)
        if sm:
            loaded = [c for c, b in zip(sm, busy) if b] or sm   # samples taken while the GPU was busy
            out.update(sm_mhz=statistics.median(loaded), sm_max_mhz=max(mx), reasons=sorted(reasons),
                       samples=len(sm), samples_under_load=len(loaded))
        return out


def max_over_ranks(values, device=None):
    """Element-wise maximum of a list of floats over all ranks (identity without a process group)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return [float(v) for v in values]
    t = torch.tensor(values, dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t]


def aggregate_throughput(world, sequences_per_rank_step, steps, seconds):
    """Whole-job sequences/s: every rank processed the same number of sequences (replicas), the job
    took as long as its slowest rank."""
    return world * sequences_per_rank_step * steps / seconds


def run_reference(args, rank):
    if rank != 0:
        return
    cfg = synth.config_glue8()
    wf = synth.widen(synth.make_weights(cfg, seed=0))
    batch = synth.batch_glue8(cfg, BATCH, SEQ, LEN_LO, LEN_HI, seed=1)
    rows_of = lambda i: [(i * REFERENCE_SAMPLE + j) % BATCH for j in range(REFERENCE_SAMPLE)]  # noqa: E731
    for i in range(args.warmup):
        time_oracle(cfg, wf, batch, rows_of(i)[:2])
    total = 0.0
    for i in range(args.steps):
        total += time_oracle(cfg, wf, batch, rows_of(i))
    value = REFERENCE_SAMPLE * args.steps / total
    cores = oracle_threads()
    sample = f"{REFERENCE_SAMPLE} of the {BATCH} sequences per step (sequences are independent)"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "glue8 tree (8 tasks, 24 layers), batch 32 x seq 128, lengths U[16,128]",
                   "sample": sample},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true", help="skip timing the oracle (N=1 only)")
    ap.add_argument("--no-fp8", action="store_true", help="skip the extra leg with the 8-bit projections")
    ap.add_argument("--eager", action="store_true",
                    help="launch every kernel from the host in the timed passes instead of replaying CUDA graphs")
    ap.add_argument("--set", action="append", default=[], metavar="KEY=VALUE",
                    help="library option (mt_set_option) to set before the run, e.g. --set fused_ln=0; repeatable")
    args = ap.parse_args()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        if args.steps == 200:
            args.steps = 10
        run_reference(args, rank)
        return

    import torch
    import torch.distributed as dist

    from paper_2107_05377_b200 import binding
    from paper_2107_05377_b200 import build as builder

    args.warmup = max(args.warmup, 3)
    distributed = world > 1
    if distributed:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    if rank == 0:
        builder.build()   # a no-op when the library is up to date
    if distributed:
        dist.barrier()    # the other ranks load the library only after rank 0 has (re)built it
    device = torch.device("cuda", local_rank)
    torch.cuda.set_device(device)

    cfg = synth.config_glue8()
    weights = synth.make_weights(cfg, seed=0)
    model = binding.MTModel(cfg, BATCH, SEQ, device=str(device))
    blob = torch.from_numpy(synth.pack_weights(cfg, weights)).pin_memory()
    model.load_weights(blob)
    mask = model.full_mask()

    batches = [synth.batch_glue8(cfg, BATCH, SEQ, LEN_LO, LEN_HI, seed=1 + i) for i in range(N_INPUT_BATCHES)]
    dev_in = [(torch.from_numpy(b.token_ids).to(device), torch.from_numpy(b.segment_ids).to(device),
               torch.from_numpy(b.lengths).to(device)) for b in batches]
    host_in = [(torch.from_numpy(b.token_ids).pin_memory(), torch.from_numpy(b.segment_ids).pin_memory(),
                torch.from_numpy(b.lengths).pin_memory()) for b in batches]
    logits = torch.zeros(BATCH, cfg.total_classes, dtype=torch.float32, device=device)
    # what a server knows about its traffic: the mean number of valid tokens per batch (tile shapes only)
    model.set_option("expected_tokens", int(round(float(np.mean([int(b.lengths.sum()) for b in batches])))))
    for kv in args.set:
        key, _, value = kv.partition("=")
        model.set_option(key, int(value))
    plan = model.plan_summary(mask)
    launches_per_step = model.plan_launches(mask)
    host_logits = torch.zeros(BATCH, cfg.total_classes, dtype=torch.float32).pin_memory()
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=device)
    stream = torch.cuda.current_stream()

    def sync_all():
        torch.cuda.synchronize()
        if distributed:
            dist.barrier()
            torch.cuda.synchronize()

    def capture(mdl, out):
        """One CUDA graph per input batch holding one mt_forward (the inputs are resident at fixed
        addresses; the library allocates nothing and its plan exists after the warm-up calls)."""
        graphs = []
        side = torch.cuda.Stream(device=device)
        for i in range(N_INPUT_BATCHES):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                mdl.forward(*dev_in[i], out, task_mask=mask)
            graphs.append(g)
        return graphs

    def timed_pass(steps, graphs=None):
        """K forwards, each between two events on the launching stream, L2 flushed (untimed) before each."""
        starts = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
        sync_all()
        for i in range(steps):
            flush.fill_(i & 0xFF)
            starts[i].record(stream)
            if graphs is not None:
                graphs[i % N_INPUT_BATCHES].replay()
            else:
                model.forward(*dev_in[i % N_INPUT_BATCHES], logits, task_mask=mask)
            ends[i].record(stream)
        sync_all()
        return [s.elapsed_time(e) for s, e in zip(starts, ends)]

    sampler = ClockSampler(local_rank) if rank == 0 else None   # samples through all passes below
    for i in range(args.warmup):
        model.forward(*dev_in[i % N_INPUT_BATCHES], logits, task_mask=mask)
    sync_all()

    graphs = None if args.eager else capture(model, logits)
    if graphs is not None:
        timed_pass(max(args.warmup, 3), graphs)
    step_ms = timed_pass(args.steps, graphs)
    total_ms = sum(step_ms)
    assert model.poll_status() == 0, "device status word set during the timed region"

    # steady state: at least STEADY_SECONDS of forwards back to back (graph replays, no flush: a forward streams
    # 340 MB of weights, more than L2), one timed region, with clock samples of its own - whatever --steps is,
    # the record shows sustained behaviour
    steady = None
    if graphs is not None:
        reps = max(int(STEADY_SECONDS * 1e3 / (total_ms / args.steps)) + 1, args.steps)
        steady_sampler = ClockSampler(local_rank) if rank == 0 else None
        t_s, t_e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        sync_all()
        t_s.record(stream)
        for i in range(reps):
            graphs[i % N_INPUT_BATCHES].replay()
        t_e.record(stream)
        sync_all()
        steady_ms = max_over_ranks([t_s.elapsed_time(t_e)], device)[0]
        steady = {"value": aggregate_throughput(world, BATCH, reps, steady_ms * 1e-3), "unit": UNIT, "steps": reps,
                  "ms_per_step": steady_ms / reps, "seconds": steady_ms * 1e-3,
                  "how": "forwards back to back on one stream, one timed region, no L2 flush",
                  "clocks": steady_sampler.stop() if steady_sampler else None}
        assert model.poll_status() == 0, "device status word set during the steady-state leg"

    # end to end through the host entry point: pinned host inputs -> device, forward, logits -> pinned host
    # buffer, and the host waits for every step's logits before it issues the next step.  Eagerly:
    # mt_forward_host.  Otherwise the same call without its final wait (mt_forward_host_async) is
    # captured once per input batch - copies included - and every step is one graph launch plus the wait.
    for i in range(3):
        model.forward_host(*host_in[i % N_INPUT_BATCHES], host_logits, task_mask=mask)
    sync_all()
    host_graphs = None
    if not args.eager:
        host_graphs = []
        side = torch.cuda.Stream(device=device)
        for i in range(N_INPUT_BATCHES):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                model.forward_host_async(*host_in[i], host_logits, task_mask=mask)
            host_graphs.append(g)
        for i in range(3):
            host_graphs[i % N_INPUT_BATCHES].replay()
            stream.synchronize()
    t0 = time.perf_counter()
    for i in range(args.steps):
        if host_graphs is not None:
            host_graphs[i % N_INPUT_BATCHES].replay()
            stream.synchronize()
        else:
            model.forward_host(*host_in[i % N_INPUT_BATCHES], host_logits, task_mask=mask)
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0

    # the same K steps with two batches in flight: a second model over the SAME weights arena (a workspace
    # of its own), one stream each, steps dealt alternately; timed as one region (no flush in between: each
    # step streams 340 MB of weights, more than L2).  Reported beside the headline, which stays one stream.
    second = binding.MTModel(cfg, BATCH, SEQ, device=str(device), share_weights_with=model)
    second.set_option("expected_tokens", int(round(float(np.mean([int(b.lengths.sum()) for b in batches])))))
    for kv in args.set:
        key, _, value = kv.partition("=")
        second.set_option(key, int(value))
    pair = [(model, torch.cuda.Stream(device=device), logits), (second, torch.cuda.Stream(device=device), torch.zeros_like(logits))]

    for mdl, s2, out in pair:   # plans exist before anything is captured
        mdl.forward(*dev_in[0], out, task_mask=mask, stream=s2)
    sync_all()
    pair_graphs = None if args.eager else [capture(mdl, out) for mdl, _, out in pair]

    def in_flight_pass(steps):
        fork, join = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        fork.record(stream)
        for _, s2, _ in pair:
            s2.wait_event(fork)
        for i in range(steps):
            mdl, s2, out = pair[i % 2]
            if pair_graphs is not None:
                with torch.cuda.stream(s2):
                    pair_graphs[i % 2][i % N_INPUT_BATCHES].replay()
            else:
                mdl.forward(*dev_in[i % N_INPUT_BATCHES], out, task_mask=mask, stream=s2)
        for _, s2, _ in pair:
            done = torch.cuda.Event()
            done.record(s2)
            stream.wait_event(done)
        join.record(stream)
        sync_all()
        return fork.elapsed_time(join)

    in_flight_pass(2 * max(args.warmup, 3))
    two_ms = in_flight_pass(args.steps)
    assert model.poll_status() == 0 and second.poll_status() == 0, "device status word set with two batches in flight"

    # the same K steps with the 8-bit projections (option "fp8_gemm": E4M3 operands, one scale per operand row;
    # a model of its own, since the option sizes the arenas), graph replay, L2 flushed before every step: an
    # extra key beside the bf16 headline, with the tolerance it was tested to
    fp8 = None
    if graphs is not None and not args.no_fp8:
        low = binding.MTModel(cfg, BATCH, SEQ, device=str(device), fp8_gemm=True)
        low.load_weights(blob)
        low.set_option("expected_tokens", int(round(float(np.mean([int(b.lengths.sum()) for b in batches])))))
        low_logits = torch.zeros_like(logits)
        for i in range(max(args.warmup, 3)):
            low.forward(*dev_in[i % N_INPUT_BATCHES], low_logits, task_mask=mask)
        sync_all()
        low_graphs = capture(low, low_logits)
        timed_pass(max(args.warmup, 3), low_graphs)
        low_ms = sum(timed_pass(args.steps, low_graphs))
        low.forward(*dev_in[0], low_logits, task_mask=mask)
        model.forward(*dev_in[0], logits, task_mask=mask)
        sync_all()
        assert low.poll_status() == 0
        low_ms = max_over_ranks([low_ms], device)[0]
        fp8 = {"value": aggregate_throughput(world, BATCH, args.steps, low_ms * 1e-3), "unit": UNIT,
               "ms_per_step": low_ms / args.steps, "dtype": "e4m3 operands (Q/K/V, FFN-up, FFN-down), fp32 accumulate",
               "gpu_launches_per_step": low.plan_launches(mask),
               "max_abs_logit_difference_from_bf16": float((low_logits - logits).abs().max()),
               "tested_tolerance": "hidden rel-L2 <= 8e-2, logits max-abs <= 1e-1 against the unquantised fp64 oracle"}
        del low_graphs, low

    # second pass of the same K steps with an event pair around every launch: per-kernel durations
    model.set_option("profile", 1)
    timed_pass(args.steps)
    prof = model.profile_read()
    model.set_option("profile", 0)
    clocks = sampler.stop() if sampler else None

    total_ms, e2e_s, two_ms = max_over_ranks([total_ms, e2e_s, two_ms], device)

    if rank == 0:
        peaks = measured_peaks()
        m_rows = BATCH * SEQ
        gemm_classes = ("qkv", "attn_out", "ffn_up", "ffn_down")
        gemm_ms = sum(prof[c][0] for c in gemm_classes)
        gemm_launches = sum(prof[c][1] for c in gemm_classes)
        # algorithmic work of the GEMM launches: valid tokens only (the path stores and computes no padded row)
        step_tokens = [float(batches[i % N_INPUT_BATCHES].lengths.sum()) for i in range(args.steps)]
        n_first = sum(1 for t in cfg.tasks if t.branch_layers > 0)   # last branch layers: first token only
        gemm_flops = sum(gemm_flops_per_forward(cfg, plan["layers"], t, n_first, BATCH) for t in step_tokens)
        achieved = gemm_flops / (gemm_ms * 1e-3) / 1e12 if gemm_ms > 0 else 0.0
        traffic_digest, traffic_bytes = ncu_traffic()
        traffic = traffic_bytes if traffic_digest == gemm_sources_digest() else None
        valid_tokens = float(np.mean(step_tokens))
        padded_flops = gemm_flops_per_forward(cfg, plan["layers"], m_rows) + \
            plan["layers"] * BATCH * 4.0 * cfg.hidden * SEQ * SEQ
        valid_flops = gemm_flops + sum(
            (plan["layers"] - n_first) * 4.0 * cfg.hidden * float((n.astype(np.float64) ** 2).sum())
            + n_first * first_token_attention_flops(cfg, n)
            for n in (batches[i % N_INPUT_BATCHES].lengths for i in range(args.steps)))
        value = aggregate_throughput(world, BATCH, args.steps, total_ms * 1e-3)
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic",
            "config": {"workload": "glue8 tree (8 tasks, 24 transformer layers run), batch 32 x seq 128, "
                                   "lengths U[16,128], bf16 weights N(0,0.02)",
                       "global_batch": BATCH * world, "seq_len": SEQ, "parallelism": f"replicas x{world}",
                       "l2": "256 MB buffer written before every timed step (untimed); each step also streams "
                             "340 MB of weights, larger than L2",
                       "layers_run": plan["layers"], "waves": plan["waves"], "groups_per_wave": plan["groups_per_wave"],
                       "launch": "every kernel launched from the host" if args.eager else
                                 "CUDA graph replay, one captured mt_forward per input batch",
                       "token_layout": "packed (valid tokens only); last branch layers on first tokens only",
                       "valid_tokens_per_step": valid_tokens, "padded_tokens_per_step": m_rows},
            "gpu_launches": launches_per_step * args.steps,
            "e2e": {"value": aggregate_throughput(world, BATCH, args.steps, e2e_s), "unit": UNIT,
                    "h2d_bytes_per_step": 2 * BATCH * SEQ * 4 + BATCH * 4,
                    "d2h_bytes_per_step": BATCH * cfg.total_classes * 4},
            "roofline": {"bound": "tensor", "kernel": "gemm_bf16_tcgen05, gemm_low_tcgen05, gemm_ln_tcgen05, gemm_ln_pair_tcgen05 and gemm_ln_low_tcgen05 "
                                   "(QKV, attention-out, FFN-up, FFN-down launches; the last three include the LayerNorm after the "
                                   "residual GEMM)",
                         "flops": "valid tokens only; the last layer of each branch counts its attention-output and FFN maps on one token "
                                  "per sequence",
                         "achieved": achieved, "peak": peaks["tflops"], "unit": "TFLOP/s",
                         "frac": achieved / peaks["tflops"], "peak_source": peaks["source"],
                         "peak_nominal": NOMINAL_BF16_TFLOPS, "frac_of_nominal": achieved / NOMINAL_BF16_TFLOPS,
                         "traffic": traffic,
                         "launches": int(gemm_launches), "avg_launch_us": 1e3 * gemm_ms / max(gemm_launches, 1)},
            "roofline_forward": {"what": "all algorithmic FLOPs of a forward (GEMMs and attention, valid tokens only) over "
                                         "the whole step time, every kernel and every launch gap included",
                                 "achieved": valid_flops / (total_ms * 1e-3) / 1e12, "unit": "TFLOP/s",
                                 "peak": peaks["tflops"], "frac": valid_flops / (total_ms * 1e-3) / 1e12 / peaks["tflops"],
                                 "peak_source": peaks["source"], "peak_nominal": NOMINAL_BF16_TFLOPS,
                                 "frac_of_nominal": valid_flops / (total_ms * 1e-3) / 1e12 / NOMINAL_BF16_TFLOPS},
            "steady_state": steady,
            "fp8_gemm": fp8,
            "forward_tflops_valid": valid_flops / (total_ms * 1e-3) / 1e12,
            "forward_tflops_padded_equivalent": padded_flops * args.steps / (total_ms * 1e-3) / 1e12,
            "kernel_ms_per_step": {k: v[0] / args.steps for k, v in prof.items()},
            "two_in_flight": {"value": aggregate_throughput(world, BATCH, args.steps, two_ms * 1e-3), "unit": UNIT,
                              "ms_per_step": two_ms / args.steps,
                              "how": "two models over one weights arena, one stream each, steps dealt alternately, "
                                     "one timed region of the same K steps without L2 flush"},
            "clocks": clocks,
        }
        if world == 1 and not args.no_cpu_baseline:
            wf = synth.widen(weights)
            secs = time_oracle(cfg, wf, batches[0], range(BATCH))
            out["cpu_baseline"] = {"value": BATCH / secs, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
                                   "sample": f"one forward of all {BATCH} sequences of the first batch ({secs:.1f} s)"}
        print(json.dumps(out))
    if distributed:
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
