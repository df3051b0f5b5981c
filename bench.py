"""Benchmark of the affinity-aware sharding hot path on GB300.

One step = the whole hot path on one calibration layer of the Qwen3-0.6B
shape (d=1024, 8 KV groups, SwiGLU N=3072, T=16384 tokens, D=2 devices):
zero A, dtp_affinity_accumulate (tcgen05 bf16 GEMM with the fused SwiGLU
first-order epilogue and on-chip token reduction), then dtp_search_layout
(10 coordinate-ascent iterations).  Inputs (302 MB of activations) are larger
than the 129 MB L2, so no flush is needed between steps.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun each rank processes its own layer (seed + rank): the affinity
pass and the up-edge search are independent per layer, so there is no
collective on the data path ("weak" scaling); the timed region is bracketed by
barriers and the max over ranks is reported.  ``--impl reference`` times the
fp64 CPU oracle (the reference arm for this method) on a bounded token slice.
Rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import datetime
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2609_13846_gb300 import synth  # noqa: E402

WORKLOAD = "qwen3_0.6b_layer"
METRIC = "affinity tokens/s per layer (Qwen3-0.6B shape)"
UNIT = "tokens/s"


def flop_per_token(w) -> float:
    """2*d*(2N)*(G+1): X and every C_h against [W_gate | W_up]."""
    return 2.0 * w.d * 2 * w.N * (w.G + 1)


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        j = json.load(open(p))
        clk = j.get("clocks_under_load", {})
        return dict(bf16=float(j["bf16_tflops"]), bf16_sustained=float(j.get("bf16_tflops_sustained", 0)),
                    hbm=float(j["hbm_gbs"]), source="measured", sm_mhz=clk.get("sm_mhz_median"))
    return dict(bf16=1900.0, bf16_sustained=1700.0, hbm=6800.0, source="fallback", sm_mhz=None)


def profile_field(key: str, name: str = "affinity_fo_tc_qwen3_layer.txt"):
    """A number from a committed ncu summary under profiles/ (a line ``key: value ...``), or None."""
    p = os.path.join(ROOT, "profiles", name)
    if not os.path.exists(p):
        return None
    for line in open(p):
        if line.startswith(key + ":"):
            try:
                return float(line.split(":", 1)[1].split()[0])
            except ValueError:
                return None
    return None


def traffic_from_profile():
    """DRAM bytes per launch of the affinity kernel from the committed ncu summary."""
    return profile_field("dram_bytes_per_full_launch")


class Clocks:
    """Samples nvidia-smi clocks and throttle reasons during the timed region.

    mark_start() / mark_end() bracket the timed work; the summary uses the samples taken between
    the two marks (by nvidia-smi's own timestamps) when there are any, else every sample."""

    FIELDS = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None
        self.t0 = self.t1 = None

    def __enter__(self):
        # samples go to a git-ignored folder of the repository
        os.makedirs(os.path.join(ROOT, "_build"), exist_ok=True)
        fd, self.path = tempfile.mkstemp(suffix=".csv", prefix="clocks_", dir=os.path.join(ROOT, "_build"))
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "50"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (FileNotFoundError, OSError):
            self.proc = None
        time.sleep(0.25)
        return self

    def mark_start(self):
        self.t0 = time.time()

    def mark_end(self):
        self.t1 = time.time()

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if self.proc is None or not self.path:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows, smax = [], None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 10:
                continue
            try:
                sm = float(parts[2])
                smax = float(parts[3])
            except ValueError:
                continue
            try:
                ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
            except ValueError:
                ts = None       # an unexpected timestamp format: the sample still counts, outside the window
            rows.append((ts, sm, {n for n, v in zip(names, parts[6:10]) if v.lower().startswith("active")}))
        os.unlink(self.path)
        inside = [r for r in rows
                  if r[0] is not None and self.t0 is not None and self.t1 is not None and self.t0 <= r[0] <= self.t1]
        use = inside or rows
        sm = [r[1] for r in use]
        reasons = set().union(*[r[2] for r in use]) if use else set()
        busy = [x for x in sm if smax and x > 0.3 * smax] or sm
        return {"sm_mhz": statistics.median(busy) if busy else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(rows), "samples_in_timed_region": len(inside)}


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def run_reference(args, w):
    """The fp64 CPU oracle (the reference arm for this method) on a bounded token slice."""
    import oracle
    world, rank, _ = dist_env()
    if rank != 0:
        return
    T_slice = args.cpu_tokens
    L = synth.make_workload_layer(w, T=T_slice)
    X, C, Wg, Wu = (L[k].double().numpy() for k in ("X", "C", "W_gate", "W_up"))
    for _ in range(args.warmup):
        oracle.affinity_fo(X[:8], C[:, :8], Wg, Wu)
    times = []
    A = None
    for _ in range(args.steps):
        t0 = time.perf_counter()
        A = oracle.affinity_fo(X, C, Wg, Wu)
        oracle.search_layout(A.astype(np.float32), w.D[0], w.iters)
        times.append(time.perf_counter() - t0)
    total = sum(times)
    value = T_slice * args.steps / total
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "d": w.d, "G": w.G, "N": w.N, "T": w.T, "D": w.D[0],
                   "iters": w.iters, "token_slice": T_slice},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
                         "sample": f"{T_slice} of {w.T} tokens of one layer per step, then the D={w.D[0]} search"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def cpu_baseline(w, A_gpu, budget_s: float):
    """Oracle timed on the host cores on a bounded token slice (rank 0, N=1 only)."""
    import oracle
    T0 = 16
    L = synth.make_workload_layer(w, T=T0)
    X, C, Wg, Wu = (L[k].double().numpy() for k in ("X", "C", "W_gate", "W_up"))
    t0 = time.perf_counter()
    oracle.affinity_fo(X, C, Wg, Wu)
    per_tok = (time.perf_counter() - t0) / T0
    T_slice = int(max(T0, min(8192, budget_s / max(per_tok, 1e-9))))
    L = synth.make_workload_layer(w, T=T_slice)
    X, C, Wg, Wu = (L[k].double().numpy() for k in ("X", "C", "W_gate", "W_up"))
    t0 = time.perf_counter()
    oracle.affinity_fo(X, C, Wg, Wu)
    t_aff = time.perf_counter() - t0
    A_np = A_gpu.float().cpu().numpy()
    t0 = time.perf_counter()
    oracle.search_layout(A_np, w.D[0], w.iters)
    t_search = time.perf_counter() - t0
    return {"value": T_slice / t_aff, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": f"affinity on {T_slice} of {w.T} tokens of one layer (fp64); "
                      f"search on the GPU's A took {1e3 * t_search:.1f} ms",
            "search_ms": 1e3 * t_search}


# token slices on which the oracle is timed for each workload (the full tiny config; 256 tokens of one
# layer of the Qwen-shaped and Danube-shaped models; 64 tokens of the Llama-shaped layer)
ORACLE_SLICES = (("tiny", 256), ("qwen3_0.6b_layer", 256), ("qwen3_0.6b_model", 256),
                 ("danube3_500m_model", 256), ("llama3.1_8b_layer", 64))


def oracle_per_config():
    """The fp64 oracle's affinity time per token on a token slice of every workload (layer 0)."""
    import oracle
    out = {}
    for name, T in ORACLE_SLICES:
        wc = synth.WORKLOADS[name]
        L = synth.make_workload_layer(wc, T=T)
        X, C, Wg, Wu = (L[k].double().numpy() for k in ("X", "C", "W_gate", "W_up"))
        t0 = time.perf_counter()
        oracle.affinity_fo(X, C, Wg, Wu)
        dt = time.perf_counter() - t0
        out[name] = {"tokens": T, "s_per_token": dt / T, "tokens_per_s": T / dt,
                     "gflops": flop_per_token(wc) * T / dt / 1e9}
    return out


def oracle_model_search(A_model, gpu_results, iters):
    """The oracle's up-edge coordinate ascent over every layer of the model on the GPU's affinities,
    timed on the host, per device count; also whether its layouts equal the GPU's bit for bit."""
    import oracle
    out = {}
    for D, ref in gpu_results.items():
        t0 = time.perf_counter()
        res = [oracle.search_layout(A_model[i], D, iters) for i in range(A_model.shape[0])]
        dt = time.perf_counter() - t0
        same = all(r["score_q"] == int(ref["score_q"][i]) and np.array_equal(r["h"], ref["h"][i]) and
                   np.array_equal(r["nu"], ref["nu"][i]) for i, r in enumerate(res))
        out[f"D{D}_host_ms"] = 1e3 * dt
        out[f"D{D}_host_matches_gpu"] = bool(same)
    out["host_cores"] = oracle.num_threads()
    return out


def model_cpu_baseline(w, S_up, S_down, chain_gpu, searches):
    """The oracle beside a whole-model run, on the host cores: its affinity on a token slice of layer 0
    (256 tokens, 64 for the Llama-shaped layer), extrapolated to every layer's tokens, and its
    whole-model coordinate ascent (both edges) on the GPU's matrices, timed and checked layout for
    layout against the GPU's; the host times also go into each search entry."""
    import oracle
    T_slice = 64 if w.d >= 4096 else 256
    L = synth.make_workload_layer(w, 0, T=T_slice)
    X, C, Wg, Wu = (L[k].double().numpy() for k in ("X", "C", "W_gate", "W_up"))
    t0 = time.perf_counter()
    oracle.affinity_fo(X, C, Wg, Wu)
    per_tok = (time.perf_counter() - t0) / T_slice
    Su = S_up.cpu().numpy()
    Sd = S_down.cpu().numpy() if S_down is not None else None
    for D, ref in chain_gpu.items():
        t0 = time.perf_counter()
        r = oracle.chain_search(Su, Sd, D, w.iters)
        searches[f"D{D}"]["host_ms"] = 1e3 * (time.perf_counter() - t0)
        searches[f"D{D}"]["host_matches_gpu"] = bool(
            r["J_q"] == int(ref["J_q"]) and np.array_equal(r["h"], ref["h"]) and np.array_equal(r["nu"], ref["nu"]))
    return {"value": 1.0 / per_tok, "unit": "tokens/s", "cores": oracle.num_threads(), "kind": "oracle",
            "s_per_token": per_tok, "whole_model_affinity_s_extrapolated": per_tok * w.T * w.layers,
            "sample": f"affinity on {T_slice} tokens of layer 0 (fp64); the whole-model search on the host on "
                      f"the GPU's matrices (search.D*.host_ms)"}


def layout_suite(args, w, S_up, S_down, S_add, stream):
    """The layouts of Table 4 on this model's affinities at one device count: the optimised layout,
    the ablations (anti-optimised, heads only, neurons only, 4/8/12 evenly spaced layers), the ADD-score
    layout when S_add is given (searched on the ADD up edge, scored under the first-order objective),
    and eight random layouts (seeds 1000-1007) scored with chain_score.  Returns per-layout J and the
    device time of the whole suite."""
    from paper_2609_13846_gb300 import ablation, dtp
    Lyr, G, N = S_up.shape
    D = 4 if 4 in w.D else w.D[0]
    Sd = S_down if Lyr > 1 else None
    kinds = ["optimised", "anti", "heads_only", "neurons_only"] + \
        [f"layers{n}" for n in (4, 8, 12) if n < Lyr]
    masks = {k: ablation.ablation_masks(Lyr, k) for k in kinds}
    dev_masks = {k: (None if mh is None else torch.as_tensor(mh, device=S_up.device),
                     None if mn is None else torch.as_tensor(mn, device=S_up.device), mini)
                 for k, (mh, mn, mini) in masks.items()}
    rand = [tuple(torch.as_tensor(a, device=S_up.device) for a in ablation.random_layout(Lyr, G, N, D, 1000 + s))
            for s in range(8)]
    ws = torch.empty(dtp.search_chain_workspace_size(Lyr, G, N, D), dtype=torch.uint8, device=S_up.device)

    def run(check):
        out = {}
        for k, (mh, mn, mini) in dev_masks.items():
            r = dtp.search_chain(S_up, Sd, D, w.iters, workspace=ws, check=check, move_heads=mh,
                                 move_neurons=mn, minimize=mini)
            out[k] = {"J": r["J"].clone(), "iters": r["iters_done"].clone()}
            if k == "optimised":
                out[k].update(h=r["h"].clone(), nu=r["nu"].clone())
        if S_add is not None:
            r = dtp.search_chain(S_add, Sd, D, w.iters, workspace=ws, check=check)
            sc = dtp.chain_score(S_up, Sd, r["h"], r["nu"], D, workspace=ws, check=check)
            out["add_score"] = {"J": sc["J"].clone(), "iters": r["iters_done"].clone()}
        for j, (h, nu) in enumerate(rand):
            out[f"random{j}"] = {"J": dtp.chain_score(S_up, Sd, h, nu, D, workspace=ws, check=check)["J"].clone()}
        return out

    run(True)
    torch.cuda.synchronize()
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    s0.record(stream)
    res = run(False)
    s1.record(stream)
    torch.cuda.synchronize()
    if dtp.workspace_status(ws) != dtp.DTP_OK:
        raise RuntimeError("layout suite reported a device-side error")
    J = {k: round(float(v["J"]), 4) for k, v in res.items()}
    rnd = [J[f"random{j}"] for j in range(8)]
    return {"D": D, "ms": s0.elapsed_time(s1), "J": {k: v for k, v in J.items() if not k.startswith("random")},
            "J_random_mean": round(sum(rnd) / len(rnd), 4), "J_random_range": [min(rnd), max(rnd)],
            "J_random_expected": (2 * Lyr - 1) / D,
            "layouts": len(res)}, (res["optimised"]["h"], res["optimised"]["nu"], D)


def time_apply(w, h, nu, D, stream):
    """Apply the optimised layout to stacked synthetic weights of every layer (q/k/v/o, gate/up/down),
    captured once in a CUDA graph and timed over graph replays (inputs resident, 3 replays)."""
    from paper_2609_13846_gb300 import dtp
    Wt = synth.make_dense_weights(w.layers, w.d, w.G * w.q_per_group, w.G, w.head_dim, w.N, seed=w.seed + 3000,
                                  device=h.device)
    fn = lambda: dtp.apply_layout(Wt, h, nu, D, w.head_dim, check=False)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        fn()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out, ho, no = fn()
    g.replay()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(3):
        g.replay()
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / 3
    # the graph's result is the layout's: device l's groups and neurons are the l-th contiguous slice
    ok = all(bool((h[i][ho[i]] == torch.arange(D, device=h.device).repeat_interleave(w.G // D)).all())
             for i in range(w.layers))
    nbytes = 2 * sum(v.numel() * v.element_size() for v in Wt.values())
    return {"ms": ms, "bytes": nbytes, "GBs": nbytes / ms / 1e6, "launches": 3, "graph": True, "shards_ok": ok}


def run_model(args):
    """Whole-model pipeline timing: every layer's affinity pass with the down-edge term on all
    its tokens, the ||w^d||^2 finalize, ||b_gk||^2 and S_down, then the whole-model search per D.
    Inputs are drawn per layer on the device outside the timed intervals."""
    from paper_2609_13846_gb300 import dtp, shard
    w = synth.WORKLOADS[args.model]
    world, rank, local = dist_env()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    stream = torch.cuda.current_stream()
    Lyr, G, N, T, d = w.layers, w.G, w.N, w.T, w.d
    # under torchrun each rank scores its own block of layers (up edge and the down edge leaving
    # each), then one all-gather hands every rank the whole model's matrices
    mine = shard.layers_for_rank(Lyr, rank, world)
    S_up_loc = torch.zeros((len(mine), G, N), dtype=torch.float32, device=dev)
    S_down_loc = torch.zeros((len(mine), G, N), dtype=torch.float32, device=dev)
    ws = dtp.affinity_workspace(T, d, G, N, dtp.DTP_BF16, dev) if args.qheads == 1 else \
        torch.empty(dtp.affinity_grouped_workspace_size(T, d, G * args.qheads, args.qheads, N, dtp.DTP_BF16),
                    dtype=torch.uint8, device=dev)
    S_add_loc = torch.zeros((len(mine), G, N), dtype=torch.float32, device=dev) if args.add_score else None
    t_aff = t_down = t_add = 0.0
    q = args.qheads
    t_prod = 0.0
    if args.producer and q not in (1, w.q_per_group):
        raise SystemExit("--producer takes --qheads 1 (KV-group rows) or the model's query heads per group")
    with Clocks(local) as clk:
        clk.mark_start()
        for li, i in enumerate(mine):
            L = synth.make_workload_layer(w, i, device=dev) if q == 1 else \
                synth.make_layer(d, G * q, N, T, w.layer_seed(i), dtype=w.dtype, outliers=w.outliers, device=dev)
            if args.producer:
                # C from the attention outputs: one row per query head, or per KV group when q == 1
                P = synth.make_attention_inputs(T, d, G * w.q_per_group, w.head_dim, w.layer_seed(i) + 2000, device=dev)
                torch.cuda.synchronize()
                p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                p0.record(stream)
                L["C"] = dtp.head_writes(P["attn"], P["W_o"], P["gamma"], P["rms"], w.head_dim,
                                         1 if q > 1 else w.q_per_group, out=L["C"])
                p1.record(stream)
                torch.cuda.synchronize()
                t_prod += p0.elapsed_time(p1)
                del P
            Dn = synth.make_down_inputs(d, G, w.qkv_rows, N, T, seed=w.seed + 1000 + i, device=dev)
            act2 = torch.zeros(N, dtype=torch.float32, device=dev)
            A = S_up_loc[li]
            A.zero_()
            torch.cuda.synchronize()
            e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            e0.record(stream)
            if q == 1:
                dtp.affinity_accumulate_down(L["X"], L["C"], L["W_gate"], L["W_up"], Dn["rms"], A=A, act2=act2,
                                             workspace=ws)
            else:   # one row of C per query head, summed over each KV group's q query heads
                dtp.affinity_accumulate_grouped(L["X"], L["C"], L["W_gate"], L["W_up"], q, A=A, rms_next=Dn["rms"],
                                                act2=act2, workspace=ws)
            dtp.affinity_finalize(A, T, dtp.down_sqnorm(Dn["W_down"]))
            e1.record(stream)
            if i + 1 < Lyr:
                bn = dtp.down_weight_sqnorm(Dn["Wqkv"], Dn["gamma"], Dn["W_down"])
                S_down_loc[li].copy_(dtp.down_finalize(act2, bn, T))
            e2.record(stream)
            if args.add_score:
                e3 = torch.cuda.Event(enable_timing=True)
                if q == 1:
                    dtp.affinity_add_accumulate(L["C"], L["W_gate"], L["W_up"], A_add=S_add_loc[li])
                else:
                    dtp.affinity_add_accumulate_grouped(L["C"], L["W_gate"], L["W_up"], q, A_add=S_add_loc[li])
                e3.record(stream)
            torch.cuda.synchronize()
            t_aff += e0.elapsed_time(e1)
            t_down += e1.elapsed_time(e2)
            if args.add_score:
                t_add += e2.elapsed_time(e3)
            del L, Dn
        clk.mark_end()
    if dtp.workspace_status(ws) != dtp.DTP_OK:
        raise RuntimeError("affinity kernel reported a device-side error")
    torch.cuda.synchronize()
    g0 = time.perf_counter()
    S_up, S_down = shard.gather_model_affinities(S_up_loc, S_down_loc, Lyr, device=dev)
    S_add = shard.gather_layer_results({"a": S_add_loc}, Lyr, device=dev)["a"] if args.add_score else None
    torch.cuda.synchronize()
    t_gather = (time.perf_counter() - g0) * 1e3 if world > 1 else 0.0
    t_aff, t_down, t_add, t_prod = (shard.max_over_ranks(x, device=dev) for x in (t_aff, t_down, t_add, t_prod))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    if rank != 0:
        return
    if Lyr == 1:
        S_down = S_up[:0]
    searches = {}
    chain_gpu = {}
    for D in w.D:
        r = dtp.search_chain(S_up, S_down if Lyr > 1 else None, D, w.iters)
        torch.cuda.synchronize()
        s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        s0.record(stream)
        for _ in range(3):
            r = dtp.search_chain(S_up, S_down if Lyr > 1 else None, D, w.iters, check=False)
        s1.record(stream)
        torch.cuda.synchronize()
        searches[f"D{D}"] = {"ms": s0.elapsed_time(s1) / 3, "J": float(r["J"]), "J_random": (2 * Lyr - 1) / D,
                             "iters_done": int(r["iters_done"])}
        chain_gpu[D] = {k: r[k].cpu().numpy() for k in ("h", "nu", "J_q")}
    share = dtp.top_group_share(S_up).cpu()              # Sec. 5: largest KV group's share per neuron
    suite, (h_opt, nu_opt, D_opt) = layout_suite(args, w, S_up, S_down, S_add if args.add_score else None, stream)
    apply = time_apply(w, h_opt, nu_opt, D_opt, stream)
    total_ms = t_aff + t_down + sum(v["ms"] for v in searches.values()) + t_prod + t_add + t_gather
    chunk = (16 // q) * q                      # query heads per launch; each launch has its own X pass
    fl = 2.0 * d * 2 * N * (G * q + -(-(G * q) // chunk)) * T * Lyr
    line = {"metric": f"whole-model affinity + layout time ({args.model})", "value": total_ms / 1e3, "unit": "s",
            "higher_is_better": False, "n_gpus": world, "scaling": "strong", "dtype": "bf16", "data": "synthetic",
            "gather_ms": t_gather,
            "config": {"workload": args.model, "layers": Lyr, "d": d, "G": G, "N": N, "T_per_layer": T,
                       "query_heads_per_group": q, "producer": bool(args.producer),
                       "D": list(w.D), "iters": w.iters, "qkv_rows": w.qkv_rows},
            "affinity_ms": t_aff, "affinity_tflops": fl / (t_aff / 1e3) / 1e12,
            "layer_tokens_per_s": Lyr * T / (t_aff / 1e3), "down_edge_ms": t_down, "search": searches,
            "add_affinity_ms": t_add if args.add_score else None, "layout_suite": suite, "apply": apply,
            "top_group_share": {"min": float(share.min()), "max": float(share.max()), "mean": float(share.mean()),
                                "uniform": 1.0 / G},
            "pipeline_s": (total_ms + suite["ms"] + apply["ms"]) / 1e3,
            "producer_ms": t_prod if args.producer else None,
            "paper_context": "RTX 5090: affinity 49-51 s (incl. calibration forward), optimisation 38-47 s",
            "clocks": clk.summary(),
            "clocks_note": "sampled over the per-layer scoring loop (input generation included)"}
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = model_cpu_baseline(w, S_up, S_down if Lyr > 1 else None, chain_gpu, searches)
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-budget", type=float, default=10.0, help="seconds of oracle work for cpu_baseline")
    ap.add_argument("--cpu-tokens", type=int, default=64, help="token slice per step of --impl reference")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--sustained-s", type=float, default=2.0,
                    help="seconds of back-to-back steps for the sustained figure (0: skip)")
    ap.add_argument("--model", default=None, help="time a whole-model pipeline instead, e.g. qwen3_0.6b_model")
    ap.add_argument("--add-score", action="store_true", help="with --model: also the ADD affinity and its layout")
    ap.add_argument("--producer", action="store_true",
                    help="with --model: make C from synthetic attention outputs with the producer kernel")
    ap.add_argument("--qheads", type=int, default=1,
                    help="with --model: query heads per KV group; >1 scores each query head and sums per group")
    args = ap.parse_args()
    w = synth.WORKLOADS[WORKLOAD]
    if args.model:
        run_model(args)
        return

    if args.impl == "reference":
        run_reference(args, w)
        return

    from paper_2609_13846_gb300 import dtp, shard

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    peaks = load_peaks()

    # inputs resident in HBM; each rank owns one layer (world layers in all, one block each)
    layer = shard.layers_for_rank(world, rank, world)[0]
    L = synth.make_layer(w.d, w.G, w.N, w.T, w.seed + layer, dtype=w.dtype, outliers=w.outliers, device=dev)
    X, C, Wg, Wu = L["X"], L["C"], L["W_gate"], L["W_up"]
    D, iters = w.D[0], w.iters
    stream = torch.cuda.current_stream()
    side = torch.cuda.Stream(device=dev)
    n_sms = torch.cuda.get_device_properties(dev).multi_processor_count
    # Step pipeline: the affinity pass of step k is capped one CTA below the chip (max_ctas; the library
    # rounds that down to an even count, 150 of 152) while the layout search of step k-1 (a cluster of
    # two thread blocks) runs on the two SMs left, from a second stream.
    # A and the search workspace are double-buffered; events order each buffer's reuse.  (Moving
    # the 12 us partial-sum reduce to the second stream as well measured slower.)
    A_buf = [torch.zeros((w.G, w.N), dtype=torch.float32, device=dev) for _ in range(2)]
    ws_s_buf = [torch.empty(dtp.search_workspace_size(1, w.G, w.N, D), dtype=torch.uint8, device=dev)
                for _ in range(2)]
    A, ws_search = A_buf[0], ws_s_buf[0]
    ws_aff = dtp.affinity_workspace(w.T, w.d, w.G, w.N, dtp.DTP_BF16, dev)
    ready = [torch.cuda.Event() for _ in range(2)]
    free = [torch.cuda.Event() for _ in range(2)]
    used = [False, False]
    n_step = [0]

    aff_ev = []

    def step(record=False):
        b = n_step[0] % 2
        n_step[0] += 1
        if used[b]:
            stream.wait_event(free[b])           # the search of step k-2 has read A_buf[b]
        A_buf[b].zero_()
        if record:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
        dtp.affinity_accumulate(X, C, Wg, Wu, A=A_buf[b], workspace=ws_aff, max_ctas=n_sms - 1)
        if record:
            e1.record(stream)
            aff_ev.append((e0, e1))
        ready[b].record(stream)
        side.wait_event(ready[b])
        r = dtp.search_layout(A_buf[b], D, iters, workspace=ws_s_buf[b], stream=side, check=False)
        free[b].record(side)
        used[b] = True
        return r

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize()
    if any(dtp.workspace_status(x) != dtp.DTP_OK for x in ws_s_buf + [ws_aff]):
        raise RuntimeError("a kernel reported a device-side error")

    # ---- timed region: inputs resident on the device
    barrier()
    torch.cuda.synchronize()
    with Clocks(local) as clk:
        t0 = torch.cuda.Event(enable_timing=True)
        t1 = torch.cuda.Event(enable_timing=True)
        clk.mark_start()
        t0.record(stream)
        for _ in range(args.steps):
            res = step(record=True)
        stream.wait_stream(side)                 # the last step's search is inside the timed region
        t1.record(stream)
        torch.cuda.synchronize()
        clk.mark_end()
    barrier()
    elapsed_ms = shard.max_over_ranks(t0.elapsed_time(t1), device=dev)
    aff_ms = [a.elapsed_time(b) for a, b in aff_ev]
    ms_step = elapsed_ms / args.steps
    value = world * w.T * args.steps / (elapsed_ms / 1e3)
    clocks = clk.summary()

    # sustained: the same pipelined step back to back for about --sustained-s seconds (power-capped
    # steady state), timed on the device; the affinity launches of its second half give the
    # sustained kernel rate, compared with cuBLAS's sustained figure
    sus = None
    if args.sustained_s > 0:
        n_sus = max(10, int(args.sustained_s * 1e3 / ms_step))
        aff_ev.clear()
        barrier()
        torch.cuda.synchronize()
        with Clocks(local) as clk_s:
            u0, u1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            clk_s.mark_start()
            u0.record(stream)
            for k in range(n_sus):
                step(record=k >= n_sus // 2)
            stream.wait_stream(side)
            u1.record(stream)
            torch.cuda.synchronize()
            clk_s.mark_end()
        barrier()
        sus_ms = shard.max_over_ranks(u0.elapsed_time(u1), device=dev)
        sus_aff = float(np.mean([a.elapsed_time(b) for a, b in aff_ev]))
        sus = {"seconds": sus_ms / 1e3, "steps": n_sus, "value": world * w.T * n_sus / (sus_ms / 1e3),
               "unit": UNIT, "affinity_ms_second_half": sus_aff, "clocks": clk_s.summary()}
        aff_ev.clear()

    # search alone (same A, same launch) for the "search ms" part of the metric
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    s0.record(stream)
    for _ in range(5):
        dtp.search_layout(A, D, iters, workspace=ws_search, check=False)
    s1.record(stream)
    torch.cuda.synchronize()
    search_ms = s0.elapsed_time(s1) / 5

    # the 28-layer Qwen3-0.6B-shaped model search (up-edge objective, all layers batched), on
    # affinities from this kernel over a 1024-token slice of each layer (seed 100 + layer)
    model = synth.WORKLOADS["qwen3_0.6b_model"]
    A_model = torch.zeros((model.layers, model.G, model.N), dtype=torch.float32, device=dev)
    for i in range(model.layers):
        Li = synth.make_workload_layer(model, i, T=1024, device=dev)
        dtp.affinity_accumulate(Li["X"], Li["C"], Li["W_gate"], Li["W_up"], A=A_model[i])
        del Li
    model_search = {"layers": model.layers, "tokens_per_layer_for_A": 1024, "iters": model.iters}
    model_gpu = {}
    for Dm in model.D:
        wsm = torch.empty(dtp.search_workspace_size(model.layers, model.G, model.N, Dm), dtype=torch.uint8, device=dev)
        rm = dtp.search_layout_batched(A_model, Dm, model.iters, workspace=wsm)
        m0, m1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        m0.record(stream)
        for _ in range(5):
            rm = dtp.search_layout_batched(A_model, Dm, model.iters, workspace=wsm, check=False)
        m1.record(stream)
        torch.cuda.synchronize()
        if dtp.workspace_status(wsm) != dtp.DTP_OK:
            raise RuntimeError("model search reported a device-side error")
        model_search[f"D{Dm}_ms"] = m0.elapsed_time(m1) / 5
        model_search[f"D{Dm}_mean_score"] = float(rm["score"].mean())
        model_search[f"D{Dm}_max_iters_done"] = int(rm["iters_done"].max())
        # the exact optimum of every layer (all unlabelled head partitions), beside the ascent
        rg = dtp.search_global(A_model, Dm)
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        rg = dtp.search_global(A_model, Dm, check=False)
        g1.record(stream)
        torch.cuda.synchronize()
        model_search[f"D{Dm}_global_ms"] = g0.elapsed_time(g1)
        model_search[f"D{Dm}_global_mean_score"] = float(rg["score"].mean())
        model_search[f"D{Dm}_ascent_over_global_min"] = float((rm["score_q"].double() / rg["score_q"].double()).min())
        model_search[f"D{Dm}_layers_at_global"] = int((rm["score_q"] == rg["score_q"]).sum())
        model_gpu[Dm] = {k: rm[k].cpu().numpy() for k in ("h", "nu", "score_q")}
    A_model_host = A_model.cpu().numpy()
    del A_model

    # ---- end to end through the public API, host buffers in pinned memory.  Every step copies its
    # inputs (X, C, W_gate, W_up) host -> device and reads its result (A and the layout) back into
    # pinned host memory.  Steps are pipelined: the copy of step k+1 runs on a copy stream while step
    # k computes (inputs double-buffered on the device), and the search overlaps as in the device step.
    hostL = {k: v.cpu().pin_memory() for k, v in L.items()}
    h2d = sum(v.numel() * v.element_size() for v in hostL.values())
    e2e_steps = max(3, min(args.steps, 20))
    copy_s = torch.cuda.Stream(device=dev)
    dbuf = [{k: torch.empty(v.shape, dtype=v.dtype, device=dev) for k, v in hostL.items()} for _ in range(2)]
    Ae_buf = [torch.zeros((w.G, w.N), dtype=torch.float32, device=dev) for _ in range(2)]
    hA = [torch.empty((w.G, w.N), dtype=torch.float32).pin_memory() for _ in range(2)]
    hh = [torch.empty(w.G, dtype=torch.int32).pin_memory() for _ in range(2)]
    hnu = [torch.empty(w.N, dtype=torch.int32).pin_memory() for _ in range(2)]
    hsc = [torch.empty(1, dtype=torch.float64).pin_memory() for _ in range(2)]
    d2h = hA[0].numel() * 4 + hh[0].numel() * 4 + hnu[0].numel() * 4 + 8
    h2d_done = [torch.cuda.Event() for _ in range(2)]
    in_free = [torch.cuda.Event() for _ in range(2)]
    a_ready = [torch.cuda.Event() for _ in range(2)]
    a_free = [torch.cuda.Event() for _ in range(2)]
    keep = [None, None]
    e_used = [False, False]

    def e2e_step(k):
        b = k % 2
        with torch.cuda.stream(copy_s):
            if e_used[b]:
                copy_s.wait_event(in_free[b])     # step k-2's affinity has read dbuf[b]
            for key, hv in hostL.items():
                dbuf[b][key].copy_(hv, non_blocking=True)
            h2d_done[b].record(copy_s)
        stream.wait_event(h2d_done[b])
        if e_used[b]:
            stream.wait_event(a_free[b])          # step k-2's search has read Ae_buf[b]
        Ae_buf[b].zero_()
        dtp.affinity_accumulate(dbuf[b]["X"], dbuf[b]["C"], dbuf[b]["W_gate"], dbuf[b]["W_up"], A=Ae_buf[b],
                                workspace=ws_aff, max_ctas=n_sms - 1)
        in_free[b].record(stream)
        hA[b].copy_(Ae_buf[b], non_blocking=True)
        a_ready[b].record(stream)
        side.wait_event(a_ready[b])
        r = dtp.search_layout(Ae_buf[b], D, iters, workspace=ws_s_buf[b], stream=side, check=False)
        with torch.cuda.stream(side):
            hh[b].copy_(r["h"], non_blocking=True)
            hnu[b].copy_(r["nu"], non_blocking=True)
            hsc[b].copy_(r["score"].reshape(1), non_blocking=True)
        a_free[b].record(side)
        keep[b] = r
        e_used[b] = True

    for k in range(2):                            # warm the copy path and the allocator
        e2e_step(k)
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    w0 = time.perf_counter()
    for k in range(e2e_steps):
        e2e_step(k)
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - w0
    barrier()
    if not torch.equal(hA[(e2e_steps - 1) % 2], A_buf[0].cpu()):
        raise RuntimeError("end-to-end result differs from the device-resident step")

    # ---- the same, for a caller holding the attention outputs instead of C: each step ships X,
    # attn [T, Hq*hd], W_o, gamma, rms and the FFN weights, and the producer makes C on the device
    P = synth.make_attention_inputs(w.T, w.d, w.G * w.q_per_group, w.head_dim, w.seed + 2000, device=dev)
    hostP = {k: v.cpu().pin_memory() for k, v in P.items()}
    hostP.update({k: hostL[k] for k in ("X", "W_gate", "W_up")})
    h2d_att = sum(v.numel() * v.element_size() for v in hostP.values())
    pbuf = [{k: torch.empty(v.shape, dtype=v.dtype, device=dev) for k, v in hostP.items()} for _ in range(2)]
    Cdev = torch.empty((w.G, w.T, w.d), dtype=torch.bfloat16, device=dev)
    ws_hw = torch.empty(256, dtype=torch.uint8, device=dev)
    for k in range(2):
        e_used[k] = False

    def e2e_att_step(k):
        b = k % 2
        with torch.cuda.stream(copy_s):
            if e_used[b]:
                copy_s.wait_event(in_free[b])
            for key, hv in hostP.items():
                pbuf[b][key].copy_(hv, non_blocking=True)
            h2d_done[b].record(copy_s)
        stream.wait_event(h2d_done[b])
        if e_used[b]:
            stream.wait_event(a_free[b])
        Ae_buf[b].zero_()
        q = pbuf[b]
        dtp.head_writes(q["attn"], q["W_o"], q["gamma"], q["rms"], w.head_dim, w.q_per_group, out=Cdev,
                        workspace=ws_hw)
        dtp.affinity_accumulate(q["X"], Cdev, q["W_gate"], q["W_up"], A=Ae_buf[b], workspace=ws_aff,
                                max_ctas=n_sms - 1)
        in_free[b].record(stream)
        hA[b].copy_(Ae_buf[b], non_blocking=True)
        a_ready[b].record(stream)
        side.wait_event(a_ready[b])
        r = dtp.search_layout(Ae_buf[b], D, iters, workspace=ws_s_buf[b], stream=side, check=False)
        with torch.cuda.stream(side):
            hh[b].copy_(r["h"], non_blocking=True)
            hnu[b].copy_(r["nu"], non_blocking=True)
            hsc[b].copy_(r["score"].reshape(1), non_blocking=True)
        a_free[b].record(side)
        keep[b] = r
        e_used[b] = True

    for k in range(2):
        e2e_att_step(k)
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    w0 = time.perf_counter()
    for k in range(e2e_steps):
        e2e_att_step(k)
    torch.cuda.synchronize()
    e2e_att_s = time.perf_counter() - w0
    barrier()
    if dtp.workspace_status(ws_hw) != dtp.DTP_OK:
        raise RuntimeError("producer reported a device-side error")
    e2e_att = {"value": world * w.T * e2e_steps / e2e_att_s, "unit": UNIT, "h2d_bytes_per_step": h2d_att,
               "d2h_bytes_per_step": d2h, "ms_per_step": e2e_att_s * 1e3 / e2e_steps,
               "what": "inputs are the attention outputs (attn, W_o, gamma, rms) instead of C; the producer "
                       "kernel makes C per KV group on the device each step"}
    del P, pbuf, Cdev
    e2e_value = world * w.T * e2e_steps / e2e_s

    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    if rank != 0:
        return

    aff_mean_ms = float(np.mean(aff_ms))
    fl = flop_per_token(w) * w.T
    achieved = fl / (aff_mean_ms / 1e3) / 1e12
    roofline = {"bound": "tensor", "achieved": achieved, "peak": peaks["bf16"], "unit": "TFLOP/s",
                "frac": achieved / peaks["bf16"], "traffic": traffic_from_profile(),
                "kernel": "affinity_fo_tc_kernel (+ its partial-sum reduce)",
                "peak_source": f"{peaks['source']} bf16 burst (cuBLAS 8192^3)",
                "frac_of_sustained": achieved / peaks["bf16_sustained"] if peaks["bf16_sustained"] else None,
                # share of the kernel's active cycles with the tensor pipe busy (committed ncu summary)
                "tensor_pipe_active_pct": profile_field("tensor_pipe_active_pct_of_active")}
    if sus is not None:
        sus_tf = fl / (sus["affinity_ms_second_half"] / 1e3) / 1e12
        sus["affinity_tflops"] = sus_tf
        sus["frac_of_sustained_peak"] = sus_tf / peaks["bf16_sustained"] if peaks["bf16_sustained"] else None
        roofline["sustained"] = sus
        sus_mhz = sus["clocks"].get("sm_mhz")
        if peaks.get("sm_mhz") and sus_mhz and peaks["bf16_sustained"]:
            # work per SM clock cycle, the sustained affinity kernel against cuBLAS's sustained loop;
            # the peak file's median SM clock was sampled over that loop, so the two are like for like
            roofline["frac_clock_normalised"] = (sus_tf / sus_mhz) / (peaks["bf16_sustained"] / peaks["sm_mhz"])
            roofline["clock_normalisation"] = (
                f"(sustained {sus_tf:.0f} TFLOP/s / {sus_mhz:.0f} MHz median) / (cuBLAS sustained "
                f"{peaks['bf16_sustained']:.0f} TFLOP/s / {peaks['sm_mhz']:.0f} MHz median under load)")
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": WORKLOAD, "d": w.d, "G": w.G, "N": w.N, "T": w.T, "D": D, "iters": iters,
                   "layers_per_step": world, "l2": "inputs (302 MB) larger than L2; no flush",
                   "pipeline": "two streams: step k's affinity on all SMs but two, step k-1's search on "
                               "those two; A double-buffered"},
        "affinity_ms": aff_mean_ms, "affinity_tflops": achieved, "search_ms": search_ms,
        "search_iters_done": int(res["iters_done"]), "layout_score": float(res["score"]),
        "model_search": model_search,
        "roofline": roofline,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "steps": e2e_steps, "ms_per_step": e2e_s * 1e3 / e2e_steps,
                "h2d_GBs": h2d * e2e_steps / e2e_s / 1e9,
                "pipeline": "H2D of step k+1 on a copy stream during step k; D2H into pinned buffers"},
        "e2e_from_attention": e2e_att,
        "gpu_launches": 3 * args.steps,
        "clocks": clocks,
    }
    if world == 1 and not args.no_cpu_baseline:
        cb = cpu_baseline(w, A, args.cpu_budget)
        cb["per_config"] = oracle_per_config()
        cb["sample"] += ("; per_config: the oracle's affinity on a token slice of every workload; the 28-layer "
                         "model search on the host on the GPU's affinities (model_search.D*_host_ms)")
        model_search.update(oracle_model_search(A_model_host, model_gpu, model.iters))
        line["cpu_baseline"] = cb
    print(json.dumps(line), flush=True)


if __name__ == "__main__":
    main()
