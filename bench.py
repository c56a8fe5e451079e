"""Benchmark of the GB300 tree-verification step.

One step = one pass of the whole hot path on one synthetic batch: the
target's forward pass over the packed tree (ancestor-masked attention over the
committed cache), the fused LM-head argmax, the greedy acceptance walk, and
the KV compaction of the accepted path.  Default workload: the Qwen3-8B-shaped
bf16 decoder at T = 64 tree nodes over ctx_len = 2048 committed positions.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME] [--impl ours|reference]

Prints one JSON line.  N > 1 (under torchrun) runs independent replicas, one
per GPU (the step does not shard); value = tree tokens verified per second
summed over ranks.  `--impl reference` times the CPU checker (oracle) on the
host cores instead.
"""

import argparse
import dataclasses
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from synth import gen, trees  # noqa: E402
from synth.configs import WORKLOADS  # noqa: E402
from synth.model import ROOT as ROOT_KIND, TREE_SHAPE, SynthModel, synthetic_kv  # noqa: E402

METRIC = "tree-verify step µs and tree tokens/s at 1 GB300; achieved HBM GB/s vs ~8 TB/s"
UNIT = "tree tokens/s"
PLANTED = os.path.join(ROOT, "tests", "golden", "planted.json")
TRAFFIC = os.path.join(ROOT, "profiles", "traffic.json")


def log(*a):
    print(*a, file=sys.stderr, flush=True)


def workload_tree(name):
    """Tree of the workload: planted greedy path (from golden/planted.json,
    written by the CPU checker) plus uniform-random draft tokens."""
    w = WORKLOADS[name]
    cfg = w.model
    with open(PLANTED) as f:
        p = json.load(f).get(name)
    if p is None:   # no planted path for this shape yet: the tree's tokens are all random
        p = dict(seed=0, root=int(gen.uniform_int(gen.tensor_key(0, ROOT_KIND), 1, cfg.vocab)[0]), planted=[])
    seed, root = p["seed"], p["root"]
    tokens, parent, path = trees.make_tree(w.tree, w.T, root, p["planted"], cfg.vocab,
                                           gen.tensor_key(seed, TREE_SHAPE, w.T))
    return seed, tokens, parent, path


def step_bytes(cfg, ctx, T):
    """Algorithmic HBM bytes of one step: every weight matrix once (layers and
    LM head), K/V of ctx committed positions read, T positions written."""
    es = 2 if cfg.dtype == "bf16" else 4
    H, I = cfg.hidden, cfg.intermediate
    per_layer = (cfg.q_dim + 2 * cfg.kv_dim) * H + H * cfg.q_dim + 3 * H * I
    weights = (cfg.n_layers * per_layer + cfg.vocab * H) * es
    kv = cfg.n_layers * 2 * (ctx + T) * cfg.kv_dim * es
    return weights + kv


class ClockSampler:
    """nvidia-smi clocks and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, dev):
        self.proc = None
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(dev), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, ValueError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for n, v in zip(names, parts[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def traffic_for(kernel_key, src_files):
    """dram bytes per launch of a kernel from the committed ncu summary, or
    None when the kernel source changed since the counters were taken."""
    try:
        with open(TRAFFIC) as f:
            d = json.load(f)
    except (OSError, ValueError):
        return None
    e = d.get(kernel_key)
    if not e:
        return None
    h = hashlib.sha256()
    for p in src_files:
        with open(os.path.join(ROOT, p), "rb") as f:
            h.update(f.read())
    return e["dram_bytes_per_launch"] if e.get("source_sha256") == h.hexdigest() else None


def src_hash(src_files):
    h = hashlib.sha256()
    for p in src_files:
        with open(os.path.join(ROOT, p), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


GEMM_SRC = ["paper_2608_00814_gb300/csrc/gemm.cu", "paper_2608_00814_gb300/csrc/common.cuh"]


# ---------------------------------------------------------------- CPU checker timing

def _oracle_inputs(name, n_layers):
    """The checker's model view and fp64 caches for the first n_layers layers
    of the workload, and the workload's tree."""
    w = WORKLOADS[name]
    cfg = w.model
    seed, tokens, parent, _ = workload_tree(name)
    sub = dataclasses.replace(cfg, n_layers=n_layers)
    view = SynthModel(sub, seed).oracle_view()
    ck = [synthetic_kv(cfg, seed, l, w.ctx_len, "f64", "k") for l in range(n_layers)]
    cv = [synthetic_kv(cfg, seed, l, w.ctx_len, "f64", "v") for l in range(n_layers)]
    return view, ck, cv, tokens, parent


def oracle_step_estimate(name, n_layers_sample=2):
    """Time the CPU checker on a bounded sample of the workload: the full tree
    through the first n_layers_sample layers plus the LM head.  The sample runs
    once untimed first (the process's first call pays for thread start-up and
    first-touch of the checker's buffers), then once timed, with the LM head
    timed alone on the same rows; the per-layer time is extrapolated to all
    layers.  Returns (seconds per full step, seconds of CPU work spent)."""
    import oracle
    w = WORKLOADS[name]
    view, ck, cv, tokens, parent = _oracle_inputs(name, n_layers_sample)
    t_all = time.perf_counter()
    oracle.verify_tree(view, ck, cv, w.ctx_len, tokens, parent)
    t0 = time.perf_counter()
    r = oracle.verify_tree(view, ck, cv, w.ctx_len, tokens, parent)
    t_run = time.perf_counter() - t0
    t1 = time.perf_counter()
    oracle.lm_head_argmax(view, r["final_hidden"])
    lm_time = time.perf_counter() - t1
    spent = time.perf_counter() - t_all
    per_layer = max(t_run - lm_time, 0.0) / n_layers_sample
    return per_layer * w.model.n_layers + lm_time, spent


def cpu_cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count()


def run_reference(args, budget_s=60.0):
    """--impl reference: the CPU checker timed on the host cores (rank 0 only).
    Whole steps are timed, as many of the requested ones as fit in about a
    minute (at least one); `steps` reports how many ran."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle
    w = WORKLOADS[args.workload]
    if args.warmup > 0:
        oracle_step_estimate(args.workload, 1)   # one layer and the LM head: threads and buffers warm
    view, ck, cv, tokens, parent = _oracle_inputs(args.workload, w.model.n_layers)
    times = []
    t_start = time.perf_counter()
    while len(times) < max(1, args.steps):
        t0 = time.perf_counter()
        oracle.verify_tree(view, ck, cv, w.ctx_len, tokens, parent)   # every layer and the LM head
        times.append(time.perf_counter() - t0)
        if time.perf_counter() - t_start + times[-1] > budget_s:
            break
    step_s = statistics.mean(times)
    value = w.T / step_s
    sample = ("CPU checker (fp64 NumPy) on the %s tree (T=%d, ctx=%d): %d whole step(s) timed, all %d layers "
              "and the LM head for every node; warm-up: one layer and the LM head"
              % (args.workload, w.T, w.ctx_len, len(times), w.model.n_layers))
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": len(times), "warmup": 1 if args.warmup > 0 else 0, "ms_per_step": step_s * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "%s T=%d ctx_len=%d" % (args.workload, w.T, w.ctx_len), "T": w.T,
                   "ctx_len": w.ctx_len},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cpu_cores(), "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


# ---------------------------------------------------------------- replicas

def reduce_step_time(ms, world, dist=None, device="cuda"):
    """Step time of the whole job: the maximum over ranks of each rank's
    device-timed step (replicas exchange nothing else), then a barrier."""
    if world <= 1:
        return ms
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.barrier()
    return float(t.item())


def job_throughput(T, ms, world):
    """Tree tokens verified per second by all ranks together."""
    return world * T / (ms * 1e-3)


# ---------------------------------------------------------------- other workloads

OTHER_WORKLOADS = ("qwen3-0.6b", "llama3.1-8b", "qwen2.5-32b", "qwen3-4b", "qwen3-14b", "qwen3-32b")


def time_workload(B, name, steps, warmup, peak):
    """µs per verify + compaction step of another workload (graph replay,
    inputs resident, weights far larger than L2 except for the 0.6B model,
    whose 1.2 GB still exceed it)."""
    import torch
    from synth.device import upload_cache, upload_model
    w = WORKLOADS[name]
    cfg, T, ctx = w.model, w.T, w.ctx_len
    seed, tokens_np, parent_np, _ = workload_tree(name)
    weights = upload_model(SynthModel(cfg, seed))
    native = [(synthetic_kv(cfg, seed, l, ctx, "native", "k"), synthetic_kv(cfg, seed, l, ctx, "native", "v"))
              for l in range(cfg.n_layers)]
    k, v = upload_cache(cfg, native, ctx + T)
    del native
    kv = B.KVCache(k, v)
    model = B.OosModel(cfg, weights, max_T=T, use_graph=True)
    stream = torch.cuda.current_stream()
    tok = torch.as_tensor(tokens_np, dtype=torch.int32, device="cuda")
    par = torch.as_tensor(parent_np, dtype=torch.int32, device="cuda")
    outs = B.VerifyOutputs(T)

    def step():
        B.oos_tree_verify(model, kv, ctx, tok, par, T, outs.accepted_len, outs.accepted_nodes, outs.accepted_tokens,
                          outs.bonus, stream)
        B.oos_kv_compact(model, kv, ctx, outs.accepted_nodes, outs.accepted_len, T, stream)

    for _ in range(max(warmup, 3)):
        step()
    torch.cuda.synchronize()
    if B.oos_last_status(model) != B.OOS_OK:
        raise RuntimeError("%s: verify status %s" % (name, B.oos_status_string(B.oos_last_status(model))))
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    acc = int(outs.accepted_len.item())
    model.close()
    b = step_bytes(cfg, ctx, T)
    res = {"config": "%s T=%d ctx_len=%d%s" % (name, T, ctx, " kv=f16" if cfg.kv_dtype == "f16" else ""),
           "us_per_step": ms * 1e3, "tree_tokens_per_s": T / (ms * 1e-3), "step_gbs": b / (ms * 1e-3) / 1e9,
           "step_frac_of_measured_hbm": b / (ms * 1e-3) / 1e9 / peak, "accepted_len": acc}
    del weights, kv, k, v, model
    torch.cuda.empty_cache()
    return res


# ---------------------------------------------------------------- decode loop

def decode_leg(B, cfg, weights, native_cache, T, stream, n_vanilla=96, n_rounds=12, eos=2):
    """Committed tokens/s of the device decode loop and of vanilla decoding."""
    import torch
    from synth.device import upload_cache
    seed, ctx = native_cache
    cap = ctx + max(n_vanilla * T, n_rounds * T) + 8   # the plain T-node run below commits one token per T slots
    native = [(synthetic_kv(cfg, seed, l, ctx, "native", "k"), synthetic_kv(cfg, seed, l, ctx, "native", "v"))
              for l in range(cfg.n_layers)]
    k, v = upload_cache(cfg, native, cap)
    del native
    kv = B.KVCache(k, v)
    # the planted root: its first greedy decisions are well separated (golden/planted.json)
    with open(PLANTED) as f:
        p = json.load(f).get(cfg.name)
    root = int(p["root"]) if p else int(gen.uniform_int(gen.tensor_key(seed, ROOT_KIND), 1, cfg.vocab)[0])
    state = torch.zeros(3, dtype=torch.int32, device="cuda")

    def run(model, bank, max_nodes, rounds, depth=16, lanes=8):
        committed = torch.zeros(1 + rounds * max_nodes, dtype=torch.int32, device="cuda")
        committed[0] = root
        mat = torch.zeros(rounds, dtype=torch.int32, device="cuda")
        ws = torch.empty(B.oos_decode_workspace_bytes(int(bank.numel())) + 256, dtype=torch.uint8, device="cuda")
        wsa = ws[(-ws.data_ptr()) % 256:]
        B.oos_decode(model, kv, ctx, committed, 1, bank, eos, lanes, depth, max_nodes, rounds, mat, state, wsa,
                     stream)   # warm (capture, first touch)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        B.oos_decode(model, kv, ctx, committed, 1, bank, eos, lanes, depth, max_nodes, rounds, mat, state, wsa,
                     stream)
        b.record(stream)
        torch.cuda.synchronize()
        if B.oos_last_status(model) != B.OOS_OK:
            raise RuntimeError("decode status %s" % B.oos_status_string(B.oos_last_status(model)))
        n_tok = int(state[1].item()) - 1
        return committed[1:1 + n_tok].cpu().tolist(), mat.cpu().tolist(), a.elapsed_time(b) * 1e-3

    # vanilla: a bank of EOS only never matches, so every tree is the root alone (T = 1)
    eos_bank = torch.full((64,), eos, dtype=torch.int32, device="cuda")
    m1 = B.OosModel(cfg, weights, max_T=1, use_graph=True)
    van_toks, van_mat, van_s = run(m1, eos_bank, 1, n_vanilla)
    m1.close()
    # the continuation the bank is built from: the same loop on trees of T nodes
    # holding the root alone, so that it is computed by the kernels the
    # speculative run uses (a random-init model has near-tied greedy decisions,
    # which a different tree size can decide the other way)
    mT = B.OosModel(cfg, weights, max_T=T, use_graph=True)
    ref_toks, _, _ = run(mT, eos_bank, T, n_vanilla)
    seq = [root] + ref_toks
    rng = np.random.default_rng(seed)
    bank = []
    for a in range(0, len(seq) - 24, 12):
        view = list(seq[a:a + 28])
        for j in range(7, len(view), 8):
            view[j] = 3 + (view[j] + 11) % (cfg.vocab - 3)
        bank += rng.integers(3, cfg.vocab, size=16).tolist() + [eos] + view + [eos]
    spec_toks, spec_mat, spec_s = run(mT, torch.as_tensor(np.asarray(bank, np.int32), device="cuda"), T, n_rounds)
    mT.close()
    k_same = 0
    while k_same < min(len(spec_toks), len(ref_toks)) and spec_toks[k_same] == ref_toks[k_same]:
        k_same += 1
    return {"rounds": n_rounds, "tree_nodes": T, "mat": spec_mat, "mat_mean": sum(spec_mat) / len(spec_mat),
            "tokens_per_s": len(spec_toks) / spec_s, "vanilla_rounds": n_vanilla,
            "vanilla_tokens_per_s": len(van_toks) / van_s, "speedup": (len(spec_toks) / spec_s) / (len(van_toks) / van_s),
            "tokens_equal_plain": k_same, "bank_tokens": len(bank),
            "note": "device loop: hint-bank suffix match -> tree -> verify -> compaction -> commit per round, one "
                    "captured graph per round; vanilla = trees of the root alone (T=1); bank = views of the plain "
                    "greedy continuation (root-only trees of T nodes) with every 8th token altered; "
                    "tokens_equal_plain = leading committed tokens identical to that continuation"}


# ---------------------------------------------------------------- GPU arm

def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2608_00814_gb300 import binding as B
    from synth.device import upload_cache, upload_model

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.cuda.current_device()
    w = WORKLOADS[args.workload]
    cfg = w.model if not args.layers else dataclasses.replace(w.model, n_layers=args.layers)
    T, ctx = w.T, w.ctx_len
    seed, tokens_np, parent_np, path = workload_tree(args.workload)

    t0 = time.time()
    sm = SynthModel(cfg, seed)
    weights = upload_model(sm)
    native = [(synthetic_kv(cfg, seed, l, ctx, "native", "k"), synthetic_kv(cfg, seed, l, ctx, "native", "v"))
              for l in range(cfg.n_layers)]
    k, v = upload_cache(cfg, native, ctx + T)
    del native
    kv = B.KVCache(k, v)
    model = B.OosModel(cfg, weights, max_T=T, use_graph=True)
    log("setup %.1fs" % (time.time() - t0))

    stream = torch.cuda.current_stream()
    tok = torch.as_tensor(tokens_np, dtype=torch.int32, device="cuda")
    par = torch.as_tensor(parent_np, dtype=torch.int32, device="cuda")
    outs = B.VerifyOutputs(T)

    def step():
        B.oos_tree_verify(model, kv, ctx, tok, par, T, outs.accepted_len, outs.accepted_nodes, outs.accepted_tokens,
                          outs.bonus, stream)
        B.oos_kv_compact(model, kv, ctx, outs.accepted_nodes, outs.accepted_len, T, stream)

    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize()
    status = B.oos_last_status(model)
    if status != B.OOS_OK:
        raise RuntimeError("verify status %s" % B.oos_status_string(status))
    acc_len = int(outs.accepted_len.item())
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()

    # ---- device-timed steps (inputs resident in HBM; 15+ GB of weights per step: larger than L2)
    clocks = ClockSampler(dev)
    time.sleep(0.3)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    ms = reduce_step_time(e0.elapsed_time(e1) / args.steps, world, dist, "cuda")

    # ---- end to end through the C ABI with host buffers (pinned), copies inside the timed region
    h_tok = torch.as_tensor(tokens_np, dtype=torch.int32).pin_memory()
    h_par = torch.as_tensor(parent_np, dtype=torch.int32).pin_memory()
    h_len = torch.zeros(1, dtype=torch.int32).pin_memory()
    h_nodes = torch.zeros(T, dtype=torch.int32).pin_memory()
    h_toks = torch.zeros(T, dtype=torch.int32).pin_memory()
    h_bonus = torch.zeros(1, dtype=torch.int32).pin_memory()
    torch.cuda.synchronize()
    e2e_steps = max(3, args.steps // 2)
    t_start = time.perf_counter()
    for _ in range(e2e_steps):
        tok.copy_(h_tok, non_blocking=True)
        par.copy_(h_par, non_blocking=True)
        step()
        h_len.copy_(outs.accepted_len, non_blocking=True)
        h_nodes.copy_(outs.accepted_nodes, non_blocking=True)
        h_toks.copy_(outs.accepted_tokens, non_blocking=True)
        h_bonus.copy_(outs.bonus, non_blocking=True)
        stream.synchronize()
        assert int(h_len.item()) == acc_len
    e2e_s = (time.perf_counter() - t_start) / e2e_steps
    h2d = 2 * T * 4
    d2h = (2 + 2 * T) * 4

    # ---- dominant kernel: the gate/up weight GEMM, timed alone with events over every layer
    n_rep = 3
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(cfg.n_layers * n_rep)]
    for i in range(cfg.n_layers):   # warm
        B.oos_launch_stage(model, i, B.OOS_STAGE_GATE_UP, T, stream)
    torch.cuda.synchronize()
    for r in range(n_rep):
        for l in range(cfg.n_layers):
            a, b = ev[r * cfg.n_layers + l]
            a.record(stream)
            B.oos_launch_stage(model, l, B.OOS_STAGE_GATE_UP, T, stream)
            b.record(stream)
    torch.cuda.synchronize()
    k_ms = statistics.mean(a.elapsed_time(b) for a, b in ev)
    N, K = 2 * cfg.intermediate, cfg.hidden
    k_bytes = 2 * N * K + 2 * T * K + 2 * T * N
    with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) if os.path.exists(os.path.join(ROOT, "MEASURED_PEAKS.json")) \
            else open(os.devnull) as f:
        try:
            peaks = json.load(f)
            peak, peak_src = peaks["hbm_gbs"], "measured"
        except ValueError:
            peak, peak_src = 6800.0, "fallback"
    k_gbs = k_bytes / (k_ms * 1e-3) / 1e9
    traffic = traffic_for("gemm_gate_up_%s_T%d" % (args.workload, T), GEMM_SRC)

    # ---- target prefill: a ctx_len-token synthetic prompt (seeded) into slots [0, ctx) of the
    # cache (after every verify measurement: it overwrites the synthetic cache they read)
    prefill = None
    if not args.no_prefill:
        pf_model = B.OosModel(cfg, weights, max_T=128, use_graph=False)
        prompt = np.random.default_rng(seed).integers(0, cfg.vocab, size=ctx).astype(np.int32)
        p_tok = torch.as_tensor(prompt, device="cuda")
        nxt = torch.zeros(1, dtype=torch.int32, device="cuda")
        B.oos_prefill(pf_model, kv, 0, p_tok, ctx, nxt, stream)   # warm
        torch.cuda.synchronize()
        if B.oos_last_status(pf_model) != B.OOS_OK:
            raise RuntimeError("prefill status %s" % B.oos_status_string(B.oos_last_status(pf_model)))
        reps = 2
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(reps):
            B.oos_prefill(pf_model, kv, 0, p_tok, ctx, nxt, stream)
        b.record(stream)
        torch.cuda.synchronize()
        pf_ms = a.elapsed_time(b) / reps
        prefill = {"tokens": ctx, "ms": pf_ms, "tokens_per_s": ctx / (pf_ms * 1e-3), "chunk": 2048,
                   "note": "prompt in causal chunks of up to 2048 tokens; every chunk streams the weights once"}
        pf_model.close()

    # ---- hint-bank candidate step (suffix match + tree packing): a 64M-token bank (256 MB,
    # larger than L2) with a 7-token key planted at three places, and a 50k-token bank
    hint = None
    if not args.no_hint:
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        eos = 2
        key = torch.randint(3, cfg.vocab, (7,), dtype=torch.int32, device="cuda", generator=g)
        prefix = torch.cat([torch.randint(3, cfg.vocab, (30,), dtype=torch.int32, device="cuda", generator=g), key])
        tok_o = torch.zeros(T, dtype=torch.int32, device="cuda")
        par_o = torch.zeros(T, dtype=torch.int32, device="cuda")
        T_o = torch.zeros(1, dtype=torch.int32, device="cuda")
        info = torch.zeros(3, dtype=torch.int32, device="cuda")
        res = {}
        for label, nb in (("large", 64 << 20), ("request", 50_000)):
            bank = torch.randint(3, cfg.vocab, (nb,), dtype=torch.int32, device="cuda", generator=g)
            for f in (0.1, 0.5, 0.9):
                at = int(f * (nb - 20))
                bank[at:at + 7] = key
                bank[at + 7:at + 9] = torch.tensor([11 + at % 7, 12], dtype=torch.int32, device="cuda")
            ws = torch.empty(B.oos_hint_workspace_bytes(nb), dtype=torch.uint8, device="cuda")
            run_h = lambda: B.oos_hint_tree(bank, eos, prefix, None, None, 8, 16, T, ws, tok_o, par_o, T_o, info,
                                            stream)
            run_h()
            torch.cuda.synchronize()
            reps = 5
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            for _ in range(reps):
                run_h()
            b.record(stream)
            torch.cuda.synchronize()
            us = a.elapsed_time(b) / reps * 1e3
            res[label] = (nb, us, info.cpu().tolist(), int(T_o.item()))
        nb, us, inf, tn = res["large"]
        nr, us_r = res["request"][0], res["request"][1]
        h_bytes = 4 * nb   # bank tokens read (match bytes are written only where something matches)
        # the part of the call that grows with the bank (the match kernel's streaming): the
        # difference between the two banks cancels the fixed cost (launches, the
        # packing block)
        m_gbs = 4 * (nb - nr) / ((us - us_r) * 1e-6) / 1e9 if us > us_r else None
        hint = {"bank_tokens": nb, "us": us, "gbs": h_bytes / (us * 1e-6) / 1e9,
                "frac_of_measured_hbm": h_bytes / (us * 1e-6) / 1e9 / peak, "match_n": inf[0], "hint_lanes": inf[1],
                "tree_nodes": tn, "request_bank_tokens": nr, "request_us": us_r,
                "per_bank_token_gbs": m_gbs, "per_bank_token_frac_of_measured_hbm": m_gbs / peak if m_gbs else None,
                "note": "us: the whole call on the 64M-token bank; per_bank_token_*: 4 bytes per position over the "
                        "time the 64M-token bank adds to the 50k-token call"}
        del bank, ws

    # ---- multi-step decode loop on the device (hint-bank tree -> verify -> compaction -> commit,
    # no host round trip between rounds), against vanilla decoding (T = 1: the root alone) on the
    # same model.  The bank holds views of the target's own continuation (found by the vanilla run)
    # with every 8th token altered, so that acceptance stops inside the views the way a hint bank
    # that is only partly right makes it stop; tokens committed per call is the paper's #MAT.
    decode = None
    if not args.no_decode:
        decode = decode_leg(B, cfg, weights, native_cache=(seed, ctx), T=T, stream=stream)

    # ---- the other workload shapes, one after another (N = 1 only)
    workloads = None
    if world == 1 and not args.no_workloads:
        workloads = {}
        for name in OTHER_WORKLOADS:
            workloads[name] = time_workload(B, name, 10, 3, peak)
            log("%s: %.1f us/step" % (name, workloads[name]["us_per_step"]))

    # ---- CPU checker on the host cores (rank 0, N = 1 only)
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        s_est, spent = oracle_step_estimate(args.workload, 2)
        cpu = {"value": T / s_est, "unit": UNIT, "cores": cpu_cores(), "kind": "oracle",
               "sample": "fp64 NumPy checker on the same tree: first 2 of %d layers for all %d nodes plus the "
                         "LM head, run once untimed and once timed (%.1f s of CPU work), extrapolated to the "
                         "full step (%.2f s)"
                         % (cfg.n_layers, T, spent, s_est)}

    step_b = step_bytes(cfg, ctx, T)
    value = job_throughput(T, ms, world)
    launches_per_step = 2 + cfg.n_layers * 5 + 2 + 1   # prep, embed, 5 per layer, LM head, accept, compact
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "bf16" if cfg.dtype == "bf16" else "f32", "data": "synthetic",
            "config": {"workload": "%s T=%d ctx_len=%d%s" % (args.workload, T, ctx,
                                                               " layers=%d" % cfg.n_layers if args.layers else ""),
                       "T": T, "ctx_len": ctx,
                       "accepted_len": acc_len, "l2": "inputs larger than L2 (weights streamed once per step)",
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "us_per_step": ms * 1e3,
            "step_gbs": step_b / (ms * 1e-3) / 1e9,
            "step_frac_of_measured_hbm": step_b / (ms * 1e-3) / 1e9 / peak,
            "roofline": {"bound": "hbm", "kernel": "gate/up weight GEMM (tcgen05)",
                         "achieved": k_gbs, "peak": peak, "unit": "GB/s", "frac": k_gbs / peak,
                         "traffic": traffic, "peak_source": peak_src, "bytes_per_launch": k_bytes,
                         "ms_per_launch": k_ms},
            "cpu_baseline": cpu,
            "e2e": {"value": world * T / e2e_s, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
            "gpu_launches": launches_per_step * args.steps,
            "clocks": clk,
            "prefill": prefill,
            "hint": hint,
            "decode": decode,
            "workloads": workloads,
        }), flush=True)
    model.close()
    if world > 1:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--workload", default="qwen3-8b", choices=sorted(n for n, w in WORKLOADS.items()
                                                                      if w.model.dtype == "bf16"))
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-prefill", action="store_true", help="skip the prefill measurement")
    ap.add_argument("--no-hint", action="store_true", help="skip the hint-bank step measurement")
    ap.add_argument("--no-decode", action="store_true", help="skip the decode-loop measurement")
    ap.add_argument("--no-workloads", action="store_true", help="skip timing the other workload shapes")
    ap.add_argument("--layers", type=int, default=0,
                    help="profiling captures only: keep the first N layers of the workload's model")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
