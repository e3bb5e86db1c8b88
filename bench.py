#!/usr/bin/env python
"""Benchmark of the HSD hot path.

Workload: the 8B-shape, 3-level hierarchy at batch 1 (Llama-style 32 layers, d=4096, 32 q / 8 kv heads,
SwiGLU 14336, vocab 32000, bf16, early exits at layers 4 and 12, prompt 1024, 256 new tokens), random-init
weights and uniform-random prompts.  A step is one hsd_generate call; `value` is generated tokens per
second over the generation loop (prompt pass excluded, reported separately), inputs resident in HBM; `e2e`
times the same call from pinned host memory (prompt upload, prompt pass, generation, token download).

T is chosen as the contract asks: a short calibration run measures the per-level forward costs and
acceptance rates, then the library's own search minimises the expected latency of Theorem 3.2.

`--impl reference` times the CPU oracle (the only reference implementation there is) on a bounded sample of
the same workload.  `--workload` selects a smaller shape for development runs.
"""
import argparse
import json
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import torch  # noqa: E402

METRIC = "hsd_generated_tokens_per_s_b1"
UNIT = "tokens/s"


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        p = json.load(open(path))
        return float(p["hbm_gbs"]), "measured"
    return 6650.0, "fallback"


class ClockSampler:
    """Samples nvidia-smi clocks / throttle reasons while the timed region runs."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.rows, self.proc = index, [], None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], 0, set()
        for r in self.rows:
            try:
                sm.append(float(r[0]))
                mx = max(mx, float(r[1]))
            except (ValueError, IndexError):
                continue
            for name, v in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), r[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        sm.sort()
        return {"sm_mhz": sm[len(sm) // 2] if sm else None, "sm_max_mhz": mx or None, "reasons": sorted(reasons),
                "samples": len(sm)}


def reduce_max_over_ranks(values, device="cuda"):
    """Element-wise maximum of a list of floats over all ranks (identity without a process group)."""
    import torch.distributed as dist
    t = torch.tensor(values, device=device, dtype=torch.float64)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.tolist()


def aggregate_tokens_per_s(world, n_new, ms_per_step):
    """Whole-job throughput of `world` independent replicas generating n_new tokens per step each."""
    return world * n_new / (ms_per_step / 1e3)


def weight_bytes(cfg, n_layers):
    es = 2 if cfg["dtype"] == "bf16" else 4
    d, hd, ff, V = cfg["d_model"], cfg["head_dim"], cfg["d_ff"], cfg["vocab"]
    per_layer = (cfg["n_q_heads"] * hd * d * 2 + cfg["n_kv_heads"] * hd * d * 2 + 3 * ff * d + 2 * d) * es
    return n_layers * per_layer + (V * d + d) * es


def pass_bytes(cfg, n_layers, ctx, rows, logit_rows):
    """Algorithmic bytes of one level forward: weights once, KV read for the context, KV write and
    embedding rows for the processed rows, logits written."""
    es = 2 if cfg["dtype"] == "bf16" else 4
    kv = 2 * cfg["n_kv_heads"] * cfg["head_dim"] * es
    return (weight_bytes(cfg, n_layers) + n_layers * kv * (ctx + rows) + rows * cfg["d_model"] * es
            + logit_rows * cfg["vocab"] * es)      # ctx = context tokens summed over the sequences of the pass


def to_cuda(w):
    return {k: (v.cuda() if k != "layers" else [{n: t.cuda() for n, t in l.items()} for l in v]) for k, v in w.items()}


def choose_T(binding, cfg, weights, wl, prompts, n_calib=160):
    """Calibration run with T = (2, ..., 2), then the Theorem 3.2 search (monotone T, T_max 15)."""
    exits = wl["exits"]
    K = len(exits) - 1
    T0 = [2] * K
    eng = binding.Hsd(cfg, weights, exits, T0, max_batch=prompts.shape[0], max_seq=wl["prompt"] + n_calib + 64,
                      page_size=wl["page"])
    eng.generate(prompts, 8, 12345)                      # warm-up
    _, stats, _ = eng.generate(prompts, n_calib, 12345)
    eng.close()
    costs = [s["ms"] / max(1, s["forwards"]) for s in stats]
    alphas = [min(0.999, max(0.001, stats[i]["accepted"] / max(1, stats[i]["tested"]))) for i in range(1, K + 1)]
    T, lat = binding.hsd_search_T(costs, alphas, 15, True)
    return list(T), costs, alphas, lat


def choose_hierarchy(binding, cfg, weights, wl, prompts, T_bar=15):
    """Section 4.2 end to end: acceptance rates between ALL exit layers measured on the prompts (shared head on
    every layer's hidden state), a linear cost model of an exit fitted to the measured level costs, then the
    latency-optimal (sigma, T).  Returns (exits, T, record)."""
    n_layers = cfg["n_layers"]
    layers = list(range(1, n_layers + 1))
    base_exits = list(wl["exits"])
    T0 = [2] * (len(base_exits) - 1)
    eng = binding.Hsd(cfg, weights, base_exits, T0, max_batch=1, max_seq=wl["prompt"] + 256, page_size=wl["page"])
    rows = [eng.layer_logits(prompts[b % prompts.shape[0], 128 * k:128 * (k + 1)].contiguous(), layers)
            for b, k in ((0, 0), (0, 1))]
    alpha = binding.hsd_pairwise_alpha(torch.cat(rows, dim=1)).cpu().tolist()
    del rows
    eng.generate(prompts[:1], 8, 12345)
    _, stats, _ = eng.generate(prompts[:1], 96, 12345)
    eng.close()
    ms = [s["ms"] / max(1, s["forwards"]) for s in stats]
    # least-squares line through (exit layer, measured pass time): cost(e) = a e + b
    n = len(base_exits)
    mx, my = sum(base_exits) / n, sum(ms) / n
    a = sum((x - mx) * (y - my) for x, y in zip(base_exits, ms)) / max(1e-12, sum((x - mx) ** 2 for x in base_exits))
    b = my - a * mx
    costs = [a * e + b for e in layers]
    lat, sigma, T = binding.hsd_search_hierarchy(costs, alpha, T_bar)
    exits = [layers[i] for i in sigma]
    rec = {"candidates": n_layers, "cost_ms_per_layer": round(a, 5), "cost_ms_fixed": round(b, 5),
           "alpha_to_target": [round(alpha[i][n_layers - 1], 3) for i in sigma[:-1]],
           "expected_ms_per_token": round(lat, 4), "exits": exits, "T": list(T)}
    return exits, list(T), rec


def run_ours(args):
    from paper_2510_19705_b200 import binding, inputs
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    wl = inputs.WORKLOADS[args.workload]
    cfg = wl["model"]
    n_new, P = (args.n_new or wl["n_new"]), (args.prompt_len or wl["prompt"])
    # replicas only: each rank runs its own independent sequence (no data-path collective)
    weights = inputs.make_weights(cfg, wl["weight_seed"], device="cuda")
    B = max(1, args.batch)
    prompts_host = inputs.make_prompts(cfg["vocab"], B, P, wl["prompt_seed"] + rank).pin_memory()
    prompts = prompts_host.cuda()
    hier = None
    if args.search_hierarchy:
        exits, T, hier = choose_hierarchy(binding, cfg, weights, wl, prompts)
        wl = dict(wl, exits=tuple(exits), T=tuple(T))
        if len(exits) == 1:
            T = []
    if args.search_hierarchy:
        calib = None
    elif args.T:
        T, calib = [int(v) for v in args.T.split(",")], None
    elif wl["T"] is None:
        T, costs, alphas, lat = choose_T(binding, cfg, weights, wl, prompts)
        calib = {"costs_ms": [round(c, 4) for c in costs], "alphas": [round(a, 4) for a in alphas],
                 "expected_ms_per_token": round(lat, 4),
                 "literal_algorithm_ms_per_token": round(binding.hsd_expected_latency_literal(costs, alphas, T), 4)}
    else:
        T, calib = list(wl["T"]), None
    eng = binding.Hsd(cfg, weights, wl["exits"], T, max_batch=B, max_seq=P + n_new + sum(T) + 16, page_size=wl["page"])
    if args.coin > 0:                                    # A/B runs of two builds: the same accept decisions whatever the logits
        eng.set_iid_acceptance([args.coin] * (len(wl["exits"]) - 1))
    if args.exit_heads:                                  # Section 5.1's other setting: one (random-init) head per drafting level
        eng.set_exit_heads(inputs.make_exit_heads(cfg, len(wl["exits"]), seed=4242, device="cuda"))

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            torch.distributed.barrier()
            torch.cuda.synchronize()

    for i in range(args.warmup):
        eng.generate(prompts, n_new, 1000 + i)
    barrier()
    launches0 = binding.hsd_kernel_launches()
    dec_ms = pre_ms = 0.0
    agg = None
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        ev0.record()
        for i in range(args.steps):
            _, stats, (t_pre, t_dec) = eng.generate(prompts, n_new, i)
            dec_ms += t_dec
            pre_ms += t_pre
            agg = stats if agg is None else [{k: a[k] + b[k] for k in a} for a, b in zip(agg, stats)]
        ev1.record()
        barrier()
    launches = binding.hsd_kernel_launches() - launches0
    step_ms = ev0.elapsed_time(ev1) / args.steps
    # end to end through the public call, host buffers: prompt upload + prompt pass + generation + download
    out_host = torch.empty(B, n_new, dtype=torch.int32).pin_memory()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    e2e_steps = max(1, min(args.steps, 3))
    for i in range(e2e_steps):
        d_prompt = prompts_host.cuda(non_blocking=True)
        toks, _, _ = eng.generate(d_prompt, n_new, i)
        out_host.copy_(toks, non_blocking=True)
        torch.cuda.synchronize()
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    dec_ms_step, step_ms, e2e_ms, pre_ms_step = reduce_max_over_ranks(
        [dec_ms / args.steps, step_ms, e2e_s * 1e3, pre_ms / args.steps])
    if rank != 0:
        return
    hbm_peak, peak_kind = peaks()
    # the pass is ~99 % reads: a read-only stream measured with the library's own kernel, beside the copy figure
    read_peak = binding.hsd_stream_read_gbs() if world == 1 else None
    K = len(wl["exits"]) - 1
    # dominant unit: the target level's verification forward (one pass streams every weight once)
    tgt = agg[K]
    tgt_ms = tgt["ms"] / max(1, tgt["forwards"])
    mean_rows = tgt["rows"] / max(1, tgt["forwards"])
    mean_ctx = B * (P + n_new / 2.0)
    levels = []
    for i, s in enumerate(agg):
        ms = s["ms"] / max(1, s["forwards"])
        rows = s["rows"] / max(1, s["forwards"])
        b = pass_bytes(cfg, wl["exits"][i], mean_ctx, rows, rows if i == 0 else (s["drafted"] / max(1, s["calls"]) + 1))
        levels.append({"level": i, "layers": wl["exits"][i], "forwards": s["forwards"], "ms_per_forward": round(ms, 4),
                       "rows_per_forward": round(rows, 2), "gbs": round(b / ms / 1e6, 1) if ms > 0 else None,
                       "accept_rate": round(s["accepted"] / s["tested"], 4) if s["tested"] else None})
    tgt_bytes = pass_bytes(cfg, wl["exits"][K], mean_ctx, mean_rows, tgt["drafted"] / max(1, tgt["calls"]) + 1)
    achieved = tgt_bytes / tgt_ms / 1e6 if tgt_ms > 0 else 0.0
    # DRAM traffic per launch: measured ratio to the algorithmic bytes from the committed ncu capture of the
    # same kernel on a smaller shape, scaled to this launch
    traffic = None
    ratio_file = os.path.join(ROOT, "profiles", "traffic_ratio.json")
    if os.path.exists(ratio_file):
        traffic = int(json.load(open(ratio_file))["dram_bytes_per_algorithmic_byte"] * tgt_bytes)
    line = {
        "metric": METRIC, "value": round(aggregate_tokens_per_s(world, B * n_new, dec_ms_step), 2), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(dec_ms_step, 3), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": cfg["dtype"], "data": "synthetic",
        "config": {"workload": args.workload, "batch": B, "prompt_len": P, "n_new": n_new, "exits": list(wl["exits"]),
                   "T": T, "T_search": calib, "hierarchy_search": hier, "exit_heads": bool(args.exit_heads), "l2": "inputs larger than L2 (weights %.1f GB per target pass)"
                   % (weight_bytes(cfg, cfg["n_layers"]) / 1e9), "replicas": "independent sequence per GPU"},
        "prefill_ms": round(pre_ms_step, 3), "step_ms_with_prefill": round(step_ms, 3),
        "e2e": {"value": round(aggregate_tokens_per_s(world, B * n_new, e2e_ms), 2), "unit": UNIT, "h2d_bytes_per_step": B * P * 4,
                "d2h_bytes_per_step": B * n_new * 4},
        "gpu_launches": int(launches),
        "clocks": clk.summary(),
        "roofline": {"bound": "hbm", "kernel": "fwd_persistent_kernel: one launch = the target level's whole "
                     "verification forward (32 layers + output head)",
                     "achieved": round(achieved, 1), "peak": hbm_peak, "peak_kind": peak_kind, "unit": "GB/s",
                     "frac": round(achieved / hbm_peak, 4), "frac_of_8000": round(achieved / 8000.0, 4),
                     "read_only_stream_gbs": round(read_peak, 1) if read_peak else None,
                     "frac_of_read_only_stream": round(achieved / read_peak, 4) if read_peak else None,
                     "traffic": traffic, "ms_per_launch": round(tgt_ms, 4), "bytes_per_launch": int(tgt_bytes)},
        "levels": levels,
    }
    if args.ablation and world == 1 and K >= 1:
        line["config"]["ablation"] = ablation_table(binding, eng, prompts, n_new, args.steps, agg, dec_ms, T)
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline(args.workload, T, weights)
    print(json.dumps(line))


def ablation_table(binding, eng, prompts, n_new, steps, real_stats, real_ms, T):
    """The paper's check of its two assumptions (appendix "Examining the assumptions of HSD"): latency per token with
    real or IID-coin acceptance (coin probability = the measured rate of each level), and with the measured time
    or a fixed artificial cost per forward (= the level's mean measured forward time, so it leaves out the sampling
    kernels and the host round trip).  ms per generated token (whole top-level rounds)."""
    def per_token(stats, ms, costs):
        toks = max(1, stats[-1]["emitted"])
        return ms / toks, sum(s["forwards"] * c for s, c in zip(stats, costs)) / toks
    costs = [s["ms"] / max(1, s["forwards"]) for s in real_stats]
    alphas = [s["accepted"] / max(1, s["tested"]) for s in real_stats[1:]]
    eng.set_iid_acceptance(alphas)
    iid_stats, iid_ms = None, 0.0
    for i in range(steps):
        _, st, (_, t_dec) = eng.generate(prompts, n_new, i)
        iid_ms += t_dec
        iid_stats = st if iid_stats is None else [{k: a[k] + b[k] for k in a} for a, b in zip(iid_stats, st)]
    eng.set_iid_acceptance(None)
    rr, ra = per_token(real_stats, real_ms, costs)
    ir, ia = per_token(iid_stats, iid_ms, costs)
    return {"ms_per_token": {"real_acceptance_real_cost": round(rr, 4), "iid_acceptance_real_cost": round(ir, 4),
                             "real_acceptance_artificial_cost": round(ra, 4), "iid_acceptance_artificial_cost": round(ia, 4)},
            "theorem_3_2_ms_per_token": round(binding.hsd_expected_latency(costs, alphas, T), 4),
            "literal_algorithm_ms_per_token": round(binding.hsd_expected_latency_literal(costs, alphas, T), 4),
            "alphas": [round(a, 4) for a in alphas], "costs_ms": [round(c, 4) for c in costs]}


def run_accept(args):
    """Stand-alone acceptance / resample workload (batch 64, 8 drafted positions, vocabulary 32000, bf16):
    one step = one hsd_verify_level call; four input sets are rotated so every call reads from HBM."""
    from paper_2510_19705_b200 import binding, inputs
    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    wl = inputs.WORKLOADS["accept"]
    B, t, V = wl["batch"], wl["t"], wl["vocab"]
    sets = []
    for i in range(4):
        p, q = inputs.make_accept_logits(B, t, V, seed=i, device="cuda")
        x = binding.hsd_draft_sample(q, 100 + i, 0)
        sets.append((p, q, x))
    ws = torch.empty(max(16, binding.hsd_verify_workspace_bytes(B, t)), dtype=torch.uint8, device="cuda")
    out = torch.empty(B, t + 1, dtype=torch.int32, device="cuda")
    n = torch.empty(B, dtype=torch.int32, device="cuda")
    steps, warm = max(args.steps, 20), max(args.warmup, 3)
    for i in range(warm):
        binding.hsd_verify_level(1, *sets[i % 4], 7, i, ws, out, n)
    torch.cuda.synchronize()
    l0 = binding.hsd_kernel_launches()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
    with ClockSampler(torch.cuda.current_device()) as clk:
        # a call is shorter than its submission from Python: the stream is held back for a few milliseconds first so
        # that the timed calls are queued back to back and the events bracket device time only
        torch.cuda._sleep(int(8e6))
        ev[0].record()
        for i in range(steps):
            binding.hsd_verify_level(1, *sets[i % 4], 7, i, ws, out, n)
            ev[i + 1].record()
        torch.cuda.synchronize()
    ms = ev[0].elapsed_time(ev[steps]) / steps
    launches = binding.hsd_kernel_launches() - l0
    # end to end from pinned host memory: logits upload, decision, result download
    hp, hq, hx = (a.cpu().pin_memory() for a in sets[0])
    ho = torch.empty(B, t + 1, dtype=torch.int32).pin_memory()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for i in range(3):
        dp, dq, dx = hp.cuda(non_blocking=True), hq.cuda(non_blocking=True), hx.cuda(non_blocking=True)
        binding.hsd_verify_level(1, dp, dq, dx, 7, i, ws, out, n)
        ho.copy_(out, non_blocking=True)
        torch.cuda.synchronize()
    e2e_ms = (time.perf_counter() - t0) / 3 * 1e3
    bytes_alg = (B * (t + 1) + B * t) * V * 2
    hbm_peak, peak_kind = peaks()
    achieved = bytes_alg / ms / 1e6
    line = {"metric": "accept_positions_per_s", "value": round(B * t / (ms / 1e3), 1), "unit": "positions/s", "n_gpus": 1,
            "steps": steps, "warmup": warm, "ms_per_step": round(ms, 5), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": {"workload": "accept", "batch": B, "t": t, "vocab": V,
                       "l2": "4 input sets of 69.6 MB rotated (278 MB > L2)"},
            "e2e": {"value": round(B * t / (e2e_ms / 1e3), 1), "unit": "positions/s", "h2d_bytes_per_step": bytes_alg + B * t * 4,
                    "d2h_bytes_per_step": B * (t + 1) * 4},
            "gpu_launches": int(launches), "clocks": clk.summary(),
            "roofline": {"bound": "hbm", "kernel": "row_stats_kernel and cluster_decide_kernel (one verification call: row statistics; accept tests and final draw)",
                         "achieved": round(achieved, 1), "peak": hbm_peak, "peak_kind": peak_kind, "unit": "GB/s",
                         "frac": round(achieved / hbm_peak, 4), "traffic": None, "bytes_per_launch": bytes_alg}}
    if not args.no_cpu_baseline:
        from oracle.hsd import SpecDecisions
        from oracle.verify import verify

        class Rows:
            def __init__(self, rows):
                self.r = rows

            def rows(self, idx, ctx, draft):
                return list(self.r)
        p_np, q_np, x_np = inputs.logits_to_numpy(sets[0][0]), inputs.logits_to_numpy(sets[0][1]), sets[0][2].cpu().numpy()
        t0 = time.perf_counter()
        nb = 16
        for b in range(nb):
            verify(1, list(x_np[b]), list(q_np[b]), [0], Rows(p_np[b]), SpecDecisions(7, b), 0)
        dt = time.perf_counter() - t0
        line["cpu_baseline"] = {"value": round(nb * t / dt, 1), "unit": "positions/s", "cores": 1, "kind": "oracle",
                                "sample": "%d of the %d sequences (%.1f s)" % (nb, B, dt)}
    print(json.dumps(line))


def cpu_baseline(workload, T, weights=None, rounds=2, prompt_len=64):
    """The oracle, as it stands, on a bounded sample: `rounds` top-level HSD rounds of the same model
    after a short prompt."""
    from paper_2510_19705_b200 import inputs
    from oracle.hsd import HSD, SpecDecisions
    from oracle.transformer import Transformer
    wl = inputs.WORKLOADS[workload]
    cfg = wl["model"]
    if weights is None:
        weights = inputs.make_weights(cfg, wl["weight_seed"], device="cuda" if torch.cuda.is_available() else "cpu")
    w_np = inputs.weights_to_numpy(weights)
    model = Transformer(cfg, w_np, wl["exits"])
    prompt = inputs.make_prompts(cfg["vocab"], 1, prompt_len, wl["prompt_seed"])[0].tolist()
    run = HSD(model, T, SpecDecisions(0))
    t0 = time.perf_counter()
    n = 0
    out = []
    for _ in range(rounds):
        toks, _ = run.hsd(run.K, prompt + out)
        out += toks
        n += len(toks)
    dt = time.perf_counter() - t0
    try:
        cores = len(os.sched_getaffinity(0))
    except AttributeError:
        cores = os.cpu_count()
    return {"value": round(n / dt, 4), "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": "%d top-level HSD round(s) (%d tokens, %.1f s) of the %s model after a %d-token prompt, T=%s"
                      % (rounds, n, dt, workload, prompt_len, list(T))}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2510_19705_b200 import inputs
    wl = inputs.WORKLOADS[args.workload]
    # the T our arm runs: given with --T, the workload's, else (1, ..., 1), which is what the latency search returns
    # for the 8B-shape workload on this hardware (the search itself needs the GPU's measured costs)
    if args.T:
        T = [int(v) for v in args.T.split(",")]
    else:
        T = list(wl["T"]) if wl["T"] is not None else [1] * (len(wl["exits"]) - 1)
    weights = inputs.make_weights(wl["model"], wl["weight_seed"], device="cuda" if torch.cuda.is_available() else "cpu")
    vals = []
    steps = max(1, min(args.steps, 2))
    for i in range(min(args.warmup, 1) + steps):
        cb = cpu_baseline(args.workload, T, weights)
        vals.append(cb)
    vals = vals[-steps:]
    v = sum(c["value"] for c in vals) / len(vals)
    cb = dict(vals[-1], value=round(v, 4))
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": round(v, 4), "unit": UNIT, "n_gpus": int(os.environ.get("WORLD_SIZE", "1")),
        "steps": steps, "warmup": min(args.warmup, 1), "ms_per_step": None, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "batch": 1, "T": T, "note": "CPU oracle on a bounded sample of the workload"},
        "cpu_baseline": cb, "e2e": {"value": round(v, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="8b3")
    ap.add_argument("--n-new", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--batch", type=int, default=1, help="sequences per GPU (the metric is quoted at 1)")
    ap.add_argument("--prompt-len", type=int, default=0, help="override the workload's prompt length (development runs)")
    ap.add_argument("--T", default="", help="fix T (comma separated) instead of calibrating / using the workload's")
    ap.add_argument("--coin", type=float, default=0.0,
                    help="accept every draft with this fixed probability instead of p/q (development: two builds then run "
                         "the same passes; not the benchmark's metric)")
    ap.add_argument("--ablation", action="store_true",
                    help="add the four-way latency table (real / IID-coin acceptance x measured / artificial cost)")
    ap.add_argument("--exit-heads", action="store_true",
                    help="give every drafting level its own output head and norm gain (not the default config)")
    ap.add_argument("--search-hierarchy", action="store_true",
                    help="choose the exit layers and T by the latency-optimal hierarchy search over all layers (not the default config)")
    args = ap.parse_args()
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        # started by hand with --gpus N: become the launcher of N ranks (one replica per GPU, no data-path collective)
        import socket
        with socket.socket() as sock:
            sock.bind(("127.0.0.1", 0))
            port = sock.getsockname()[1]
        cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", str(args.gpus),
               "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__)] + sys.argv[1:]
        raise SystemExit(subprocess.call(cmd))
    if args.impl == "reference":
        run_reference(args)
    else:
        if not torch.cuda.is_available():
            raise SystemExit("bench.py needs a CUDA device (there is no CPU fallback)")
        if args.workload == "accept":
            run_accept(args)
        else:
            run_ours(args)


if __name__ == "__main__":
    main()
