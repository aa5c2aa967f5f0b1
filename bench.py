#!/usr/bin/env python
"""Benchmark of the H-Spec block-parallel draft step on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--workload NAME]
    python bench.py --sweep                    # only the concurrency x block-size sweep, more steps per cell
    python bench.py --case NAME [--reps N]     # one kernel on a small case, for profiler captures

One "step" = one call of hspec_draft_block (the whole hot path) over one batch of seeded synthetic requests.
The headline workload is the concurrency-128 configuration (32B-class shapes, B = 128, k = 16, contexts
log-uniform in [1024, 32768]); the concurrency-1 and concurrency-32 configurations, the two serving workloads with
the paper's 2048-token window, and the 18 cells of the concurrency x block-size sweep are measured in the same run
and reported under "by_concurrency", "window_2048" and "sweep".  Rank 0 prints those tables as "[bench] name: {...}" lines and
then, last, ONE JSON line with the headline.

Timing: W warm-up steps, then untimed steps for --settle-s seconds (so the GPU sits at the clocks it keeps under its
power cap, the condition the tensor peak was measured in), then --repeats timed regions of exactly K steps each, every
one bracketed by a synchronise and one pair of CUDA events; `value` is the median region, all of them are listed.

Multi-GPU: the step has no exchange between requests, so N > 1 runs N independent replicas (one process per
GPU, different requests per rank, no data-path collective); time is the max over ranks.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

import synth  # noqa: E402

METRIC = "draft tokens/s per B200 at concurrency 1/32/128; % of HBM roofline"
HEADLINE = "conc128_32b"
BY_CONCURRENCY = {"1": "latency_8b", "32": "serving_8b", "128": "conc128_32b"}
FALLBACK_PEAKS = dict(hbm_gbs=6650.0, bf16_tflops=1590.0, bf16_tflops_sustained=1400.0)


# ----------------------------------------------------------------------------- helpers

def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return dict(hbm_gbs=float(p["hbm_gbs"]), bf16_tflops=float(p["bf16_tflops"]),
                    bf16_tflops_sustained=float(p.get("bf16_tflops_sustained", p["bf16_tflops"])),
                    sustained_sm_mhz=float(p.get("clocks_under_load", {}).get("sm_mhz_median", 0.0)) or None,
                    source="measured")
    return dict(FALLBACK_PEAKS, sustained_sm_mhz=1300.0, source="fallback")


def load_traffic():
    """DRAM traffic per kernel as a ratio to its algorithmic bytes, from the profiler captures recorded in
    profiles/dram_traffic.json (kernel -> {dram_read_bytes, dram_write_bytes, algorithmic_bytes, case, ...})."""
    path = os.path.join(ROOT, "profiles", "dram_traffic.json")
    if not os.path.exists(path):
        return {}
    with open(path) as f:
        rec = json.load(f)
    out = {}
    for name, r in rec.get("kernels", {}).items():
        out[name] = dict(ratio=(r["dram_read_bytes"] + r["dram_write_bytes"]) / r["algorithmic_bytes"],
                         case=r.get("case", ""), captured=r.get("captured", ""))
    return out


def workload_accounting(cfg, ctx_lens, B, k):
    """Algorithmic bytes and flops of one step (weights read once, visible target-KV bytes, dense contractions)."""
    M = B * k
    mats = [(n, s) for n, (s, kind) in synth.weight_shapes(cfg).items() if kind == "mat" and n != "embed"]
    weight_bytes = sum(2 * s[0] * s[1] for _, s in mats)
    flops = 0.0
    for n, s in mats:
        rows = B if n in ("proj_r", "proj_ds") else M
        flops += 2.0 * rows * s[0] * s[1]
    n_attn = sum(cfg["has_attn"])
    W = cfg["window"]
    vis = [min(c, W - 1) if W > 0 else c for c in ctx_lens]
    kv_bytes_layer = sum(vis) * cfg["Hkv"] * cfg["dh"] * 2 * 2
    attn_flops_layer = sum(4.0 * k * cfg["Hq"] * cfg["dh"] * (v + (k + 1) / 2) for v in vis)
    return dict(weight_bytes=weight_bytes, kv_bytes=kv_bytes_layer * n_attn, kv_bytes_per_layer=kv_bytes_layer,
                gemm_flops=flops, attn_flops=attn_flops_layer * n_attn,
                s_init_bytes=B * cfg["d_S"] * 2 * (1 + cfg["L"]),
                drafter_kv_bytes_avoided=sum(ctx_lens) * n_attn * 2 * cfg["Hkv"] * cfg["dh"] * 2)


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu_index = gpu_index
        self.lines = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                          "-lms", "50", "-i", str(self.gpu_index)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def window(self, t0, t1):
        """Median SM clock and the throttle reasons seen between two wall-clock times."""
        sm, mx, reasons = [], [], set()
        for ts, line in list(self.lines):
            if not (t0 <= ts <= t1 + 0.1):
                continue
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return dict(sm_mhz=None, sm_max_mhz=None, reasons=["no samples in the timed region"], samples=0)
        return dict(sm_mhz=statistics.median(sm), sm_max_mhz=max(mx), reasons=sorted(reasons), samples=len(sm))

    def stop(self, t0=None, t1=None):
        if self.proc is None:
            return dict(sm_mhz=None, sm_max_mhz=None, reasons=["nvidia-smi unavailable"])
        time.sleep(0.15)
        self.proc.terminate()
        return self.window(t0 if t0 is not None else 0.0, t1 if t1 is not None else time.time())


def to_np(t):
    t = t.detach().cpu()
    return t.contiguous().view(torch.int16).numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.numpy()


def dist_info():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("LOCAL_RANK", 0)), int(os.environ.get("WORLD_SIZE", 1))


def max_over_ranks(value, device=None):
    """Max of a python float over all ranks (identity when not distributed)."""
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return value
    t = torch.tensor([value], dtype=torch.float64, device=device if device is not None else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier():
    import torch.distributed as dist
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.barrier()


# ----------------------------------------------------------------------------- the CUDA arm

def run_workload(name, steps, warmup, rank, clock_gpu=None, want_e2e=True, lean=False, repeats=1, settle_s=0.0,
                 want_graph=True, **cfg_over):
    import paper_2609_24197_b200 as hs
    cfg = synth.get_config(name, **cfg_over)
    B, k = cfg["B"], cfg["k"]
    dev = torch.device("cuda", torch.cuda.current_device())
    weights = synth.make_weights(cfg, device=dev)
    batch = synth.make_request_batch(cfg, device=dev, seed_offset=1000 * rank)
    ctx = batch["ctx_lens_host"]
    max_ctx = max(ctx)
    drafter = hs.Drafter(cfg, weights, B, k, max_ctx)
    del weights                                   # the library holds its own (fp16) copies
    torch.cuda.empty_cache()
    acct = workload_accounting(cfg, ctx, B, k)
    stream = torch.cuda.current_stream()

    ids = torch.empty((B, k), dtype=torch.int32, device=dev)

    def step():
        hs.hspec_draft_block(drafter.handle, batch["page_table"], batch["ctx_lens"], batch["last_hidden"],
                             batch["last_token"], k, batch["k_pools"], batch["v_pools"], drafter.workspace, ids,
                             max_ctx=max_ctx)

    for _ in range(max(warmup, 3)):
        step()
    torch.cuda.synchronize()
    sampler = ClockSampler(clock_gpu) if clock_gpu is not None else None
    if sampler:
        sampler.start()
    # ---- untimed steps until the GPU has settled under its power cap (the sustained-peak condition)
    settle_steps = 0
    t_end = time.time() + settle_s
    while time.time() < t_end:
        for _ in range(8):
            step()
        settle_steps += 8
        torch.cuda.synchronize()
    barrier()
    # ---- the timed regions: each exactly `steps` steps, nothing else on the stream, one pair of events around it
    regions = []
    for _ in range(max(1, repeats)):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        barrier()
        t0 = time.time()
        e0.record(stream)
        for _ in range(steps):
            step()
        e1.record(stream)
        torch.cuda.synchronize()
        t1 = time.time()
        barrier()
        ms = max_over_ranks(e0.elapsed_time(e1), dev)
        regions.append(dict(ms_per_step=ms / steps, t0=t0, t1=t1))
    t_first, t_last = regions[0]["t0"], regions[-1]["t1"]
    for r in regions:
        w = sampler.window(r["t0"], r["t1"]) if sampler else None
        r["sm_mhz"] = w["sm_mhz"] if w else None
    clocks = sampler.stop(t_first, t_last) if sampler else None
    by_ms = sorted(regions, key=lambda r: r["ms_per_step"])
    median = by_ms[(len(by_ms) - 1) // 2]          # an actual region (the lower median), with its own clock reading
    total_ms = median["ms_per_step"] * steps
    stats = drafter.stats()
    assert stats["rc"] == 0, f"device status block not clean: {stats}"
    launches = stats["launches_last_step"]
    # ---- the same steps again with a pair of CUDA events around every kernel launch (recorded by the library on
    # the step's stream): per-kernel durations for the roofline figures.  The events cost host time, which shows at
    # small batch sizes, so this pass is kept out of `value`; its own step time is reported beside it.
    hs.hspec_set_profiling(drafter.handle, True)
    step()
    torch.cuda.synchronize()
    prof = {}
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
    ev[0].record(stream)
    for i in range(steps):
        step()
        ev[i + 1].record(stream)
        for e in hs.hspec_get_profile(drafter.handle):       # reading them waits for the step
            a = prof.setdefault(e["name"], dict(ms=0.0, n=0, flops=0.0, bytes=0.0, io_bytes=0.0))
            a["ms"] += e["ms"]; a["n"] += 1; a["flops"] += e["flops"]; a["bytes"] += e["bytes"]
            a["io_bytes"] += e["io_bytes"]
    torch.cuda.synchronize()
    hs.hspec_set_profiling(drafter.handle, False)
    step_ms = [ev[i].elapsed_time(ev[i + 1]) for i in range(steps)]
    out = dict(name=name, B=B, k=k, ms_per_step=total_ms / steps, step_ms=step_ms, acct=acct, prof=prof,
               launches_per_step=launches, clocks=clocks, ctx_sum=sum(ctx), ctx_max=max_ctx, cfg=cfg,
               ms_per_step_profiled=sum(step_ms) / steps, settle_steps=settle_steps, sm_mhz=median["sm_mhz"],
               regions=[dict(ms_per_step=round(r["ms_per_step"], 4), sm_mhz=r["sm_mhz"]) for r in regions])
    # ---- the step captured once in a CUDA graph and replayed (what a serving loop does with a launch-bound step);
    # reported beside `value`, which stays on plain launches
    out["graph_replay_ms_per_step"] = None
    if not lean and want_graph:
        try:
            side = torch.cuda.Stream()
            side.wait_stream(stream)
            with torch.cuda.stream(side):
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=side):
                    step()
            torch.cuda.synchronize()
            for _ in range(3):
                graph.replay()
            g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            g0.record(stream)
            for _ in range(steps):
                graph.replay()
            g1.record(stream)
            torch.cuda.synchronize()
            out["graph_replay_ms_per_step"] = g0.elapsed_time(g1) / steps
            del graph
        except Exception as exc:                   # a capture failure must not cost the bench line
            print(f"[bench] graph capture skipped: {exc}", file=sys.stderr)
            torch.cuda.synchronize()
    if lean:                                       # launch-list captures: nothing more
        out["e2e"] = dict(ms_per_step=float("nan"), h2d_bytes_per_step=0, d2h_bytes_per_step=0)
        out["_keep"] = (drafter, batch)
        return out

    if want_e2e:
        # through the public call with HOST inputs: pinned page table, context lengths, last hidden state and last
        # token are copied to the device every step and the draft ids are read back.  The target's KV cache is
        # device-resident by definition of the method (it is the serving engine's cache, read in place).
        host = {n: batch[n].cpu().pin_memory() for n in ("page_table", "ctx_lens", "last_hidden", "last_token")}
        devb = {n: torch.empty_like(batch[n]) for n in host}
        ids_host = torch.empty((B, k), dtype=torch.int32).pin_memory()
        h2d = sum(t.numel() * t.element_size() for t in host.values())
        d2h = ids_host.numel() * 4

        def e2e_step():
            for n in host:
                devb[n].copy_(host[n], non_blocking=True)
            hs.hspec_draft_block(drafter.handle, devb["page_table"], devb["ctx_lens"], devb["last_hidden"],
                                 devb["last_token"], k, batch["k_pools"], batch["v_pools"], drafter.workspace, ids,
                                 max_ctx=max_ctx)
            ids_host.copy_(ids, non_blocking=True)
            stream.synchronize()
            return int(ids_host[0, 0])
        for _ in range(3):
            e2e_step()
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(steps):
            e2e_step()
        e1.record(stream)
        torch.cuda.synchronize()
        e2e_ms = max_over_ranks(e0.elapsed_time(e1), dev) / steps
        out["e2e"] = dict(ms_per_step=e2e_ms, h2d_bytes_per_step=h2d, d2h_bytes_per_step=d2h)
    out["_keep"] = (drafter, batch)
    return out


def kv_injection_counterexample(cfg, reps=10):
    """What a KV-injecting block drafter of the same shape adds to every step (Sec. 2.2 of the paper) and this
    drafter does not do: for the positions verified since the last step, fuse the target's hidden states, project
    them to keys and values for each attention layer and write them into a drafter-side paged cache.  Measured with
    the library's own GEMM and cache-write kernels on k new positions per request (the case where a whole block was
    accepted), beside the number of bytes the cache grows by per step."""
    import paper_2609_24197_b200 as hs
    dev = torch.device("cuda", torch.cuda.current_device())
    B, k, D, r = cfg["B"], cfg["k"], cfg["D"], cfg["r"]
    Hkv, dh, ps = cfg["Hkv"], cfg["dh"], cfg["page_size"]
    layers = int(sum(cfg["has_attn"]))
    T = B * k
    g = torch.Generator(device=dev).manual_seed(synth.BASE_SEED + 77)
    h = torch.randn((T, cfg["n_fuse"] * D), generator=g, device=dev).to(torch.float16)
    w_fuse = (torch.randn((r, cfg["n_fuse"] * D), generator=g, device=dev) * 0.02).to(torch.float16)
    w_kv = [(torch.randn((2 * Hkv * dh, r), generator=g, device=dev) * 0.02).to(torch.float16) for _ in range(layers)]
    kw = torch.ones(dh, device=dev)
    pages_per_req = (k + ps - 1) // ps
    page_table = torch.arange(B * pages_per_req, dtype=torch.int32, device=dev).reshape(B, pages_per_req).contiguous()
    pools = [(torch.zeros((B * pages_per_req, ps, Hkv, dh), dtype=torch.bfloat16, device=dev),
              torch.zeros((B * pages_per_req, ps, Hkv, dh), dtype=torch.bfloat16, device=dev)) for _ in range(layers)]
    req = torch.arange(B, dtype=torch.int32, device=dev).repeat_interleave(k).contiguous()
    pos = torch.arange(k, dtype=torch.int32, device=dev).repeat(B).contiguous()
    f = torch.empty((T, r), dtype=torch.float16, device=dev)
    kv = torch.empty((T, 2 * Hkv * dh), dtype=torch.float32, device=dev)
    ws = torch.empty(max(hs.hspec_gemm_workspace_bytes(T, r, cfg["n_fuse"] * D),
                         hs.hspec_gemm_workspace_bytes(T, 2 * Hkv * dh, r)), dtype=torch.uint8, device=dev)

    def once():
        hs.hspec_op_gemm(h, w_fuse, f, workspace=ws)
        for l in range(layers):
            hs.hspec_op_gemm(f, w_kv[l], kv, workspace=ws)
            hs.hspec_op_kv_inject_write(kv.view(T, 2, Hkv, dh), kw, req, pos, page_table, pools[l][0], pools[l][1],
                                        cfg["rope_theta"], cfg["rms_eps"], True)
    for _ in range(3):
        once()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        once()
    e1.record()
    torch.cuda.synchronize()
    return dict(positions_per_step=T, layers=layers, ms_per_step=round(e0.elapsed_time(e1) / reps, 4),
                cache_bytes_added_per_step=T * layers * 2 * Hkv * dh * 2,
                note="fusion GEMM + per-layer K/V GEMM + paged bf16 cache write for k new positions per request; "
                     "the draft step measured above does none of this and keeps no drafter-side cache")


def cpu_baseline(cfg_name, k_rows=None, rank=0):
    """Times the oracle as it stands on one request (median context) of the workload, on the host cores."""
    from oracle import hspec_oracle as O
    cfg = synth.get_config(cfg_name)
    k = k_rows or cfg["k"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    weights = {n: to_np(t) for n, t in synth.make_weights(cfg, device=dev).items()}
    if dev == "cuda":
        torch.cuda.empty_cache()
    ctx_all = synth.make_ctx_lens(cfg)
    b = int(np.argsort(ctx_all)[len(ctx_all) // 2])
    batch = synth.make_request_batch(cfg, ctx_lens=[ctx_all[b]], device="cpu", seed_offset=1000 * rank)
    t0 = time.time()
    out = O.draft_block(cfg, weights, [to_np(t) for t in batch["k_pools"]], [to_np(t) for t in batch["v_pools"]],
                        to_np(batch["page_table"]), batch["ctx_lens_host"], to_np(batch["last_hidden"]),
                        to_np(batch["last_token"]), k, dtype=np.float32)
    dt = time.time() - t0
    cores = len(os.sched_getaffinity(0))
    return dict(value=k / dt, unit="draft tokens/s", cores=cores, kind="oracle",
                sample=f"1 request of {cfg_name} (context {ctx_all[b]}, k={k}), numpy float32, {dt:.1f} s",
                seconds=dt, ids=out["draft_ids"][0].tolist()), (cfg, weights, batch)


def kernel_table(res):
    steps = len(res["step_ms"])
    total = sum(v["ms"] for v in res["prof"].values())
    rows = {}
    for name, v in sorted(res["prof"].items(), key=lambda kv: -kv[1]["ms"]):
        rows[name] = dict(ms_per_step=round(v["ms"] / steps, 4), launches_per_step=v["n"] // steps,
                          share=round(v["ms"] / total, 4))
    return rows


def serial_roofline_ms(launches, kv_bytes, peaks):
    """The kernels of a step run one after another, so the step cannot beat the SUM of its kernels' own rooflines: each
    GEMM launch at the slower of its two (weight bytes at the HBM peak, flops at the tensor peak), the attention and the
    scan at their HBM bytes.  Tighter than max(HBM, tensor) of the step's totals when a step mixes a weight-streaming
    projection with tensor-bound layers.  `launches`: (name, flops, bytes) of one step's launches."""
    hbm, tf = peaks["hbm_gbs"] * 1e9, peaks["bf16_tflops_sustained"] * 1e12
    t = sum(max(f / tf, b / hbm) for n, f, b in launches if n.startswith(("gemm:", "gemm2:", "mamba_scan")))
    return (t + kv_bytes / hbm) * 1e3


def summarize(res, peaks, traffic=None):
    """Roofline numbers of one workload from the per-launch event times."""
    traffic = traffic or {}
    steps = len(res["step_ms"])
    a = res["acct"]
    ms = res["ms_per_step"]
    hbm, tf = peaks["hbm_gbs"], peaks["bf16_tflops_sustained"]
    hbm_time_ms = (a["weight_bytes"] + a["kv_bytes"]) / (hbm * 1e9) * 1e3
    tensor_time_ms = (a["gemm_flops"] + a["attn_flops"]) / (tf * 1e12) * 1e3

    def tensor_bound(v):
        return v["flops"] / (tf * 1e12) >= v["bytes"] / (hbm * 1e9)

    def group(prefix, want=None):
        """Launches of one GEMM kernel (by profile-label prefix), all of them or only those on one side of the ridge."""
        vs = {n: v for n, v in res["prof"].items() if n.startswith(prefix) and (want is None or tensor_bound(v) == want)}
        t = sum(v["ms"] for v in vs.values()) / steps
        return dict(ms=t, flops=sum(v["flops"] for v in vs.values()) / steps, bytes=sum(v["bytes"] for v in vs.values()) / steps,
                    io_bytes=sum(v["io_bytes"] for v in vs.values()) / steps, launches=sum(v["n"] for v in vs.values()) // steps,
                    labels=sorted(n.split(":", 1)[1] for n in vs))
    g1, g2 = group("gemm:"), group("gemm2:")          # one-CTA kernel (few rows), 2-CTA persistent kernel (many rows)
    gemm_ms, gemm_flops, gemm_bytes = g1["ms"] + g2["ms"], g1["flops"] + g2["flops"], g1["bytes"] + g2["bytes"]
    att = res["prof"].get("attn_partial")
    n_attn = max(1, sum(res["cfg"]["has_attn"]))
    att_ms = att["ms"] / steps if att else 0.0
    att_gbs = a["kv_bytes"] / (att_ms * 1e-3) / 1e9 if att_ms > 0 else 0.0
    gemm_tfs = gemm_flops / (gemm_ms * 1e-3) / 1e12 if gemm_ms > 0 else 0.0
    gemm_gbs = gemm_bytes / (gemm_ms * 1e-3) / 1e9 if gemm_ms > 0 else 0.0
    sm_mhz = res.get("sm_mhz")

    def dram_traffic(kernel, algorithmic_bytes_per_launch):
        """DRAM bytes per launch = the ratio a profiler capture of this kernel measured (small case, scaled by the
        algorithmic bytes: every byte is read once, so traffic grows in proportion) x this launch's algorithmic bytes."""
        t = traffic.get(kernel)
        if not t:
            return None, "no profiler capture on record for this kernel"
        return round(t["ratio"] * algorithmic_bytes_per_launch), \
            f"{t['ratio']:.3f} x algorithmic bytes per launch (ncu dram__bytes_read+write on {t['case']})"

    def gemm_roof(kernel, grp, is_tensor):
        """Roofline of one GEMM kernel over those of its launches in a step that sit on one side of the ridge (a launch
        is tensor-bound when its flops at the tensor peak take longer than its weight bytes at the HBM peak)."""
        if grp["ms"] <= 0:
            return None
        tfs, gbs = grp["flops"] / (grp["ms"] * 1e-3) / 1e12, grp["bytes"] / (grp["ms"] * 1e-3) / 1e9
        # (captures on record: the pair kernel on a tensor-bound case and on a streaming case, the one-CTA kernel streaming)
        bound = "tensor" if is_tensor else "hbm"
        key = kernel + ":" + bound if kernel + ":" + bound in traffic else kernel
        tr, tr_note = dram_traffic(key, (grp["bytes"] + grp["io_bytes"]) / max(1, grp["launches"]))
        base = dict(kernel=kernel, launches=grp["labels"], traffic=tr, traffic_note=tr_note, ms_per_step=round(grp["ms"], 4),
                    launches_per_step=grp["launches"],
                    algorithmic_bytes_per_launch=round((grp["bytes"] + grp["io_bytes"]) / max(1, grp["launches"])))
        if is_tensor:
            r = dict(base, bound="tensor", achieved=round(tfs, 1), peak=tf, unit="TFLOP/s", frac=round(tfs / tf, 4),
                     note=f"sum over its launches per step: 2*M*N*K flops / CUDA-event time; peak = cuBLAS bf16 sustained, "
                          f"of {peaks['source']} (fp16 has the same nominal rate)")
            if sm_mhz and peaks.get("sustained_sm_mhz"):
                # the sustained peak was measured at its own (lower) clock: compare flops per clock as well
                r["per_clock"] = dict(achieved_tflops_per_ghz=round(tfs / (sm_mhz * 1e-3), 1),
                                      peak_tflops_per_ghz=round(tf / (peaks["sustained_sm_mhz"] * 1e-3), 1),
                                      frac=round((tfs / sm_mhz) / (tf / peaks["sustained_sm_mhz"]), 4),
                                      sm_mhz=sm_mhz, peak_sm_mhz=peaks["sustained_sm_mhz"])
            return r
        return dict(base, bound="hbm", achieved=round(gbs, 1), peak=hbm, unit="GB/s", frac=round(gbs / hbm, 4),
                    note=f"sum over its launches per step: weight bytes / CUDA-event time; peak = copy bandwidth, of "
                         f"{peaks['source']}")
    roofs = [r for r in (gemm_roof(kern, group(prefix, want), want)
                         for kern, prefix in (("gemm_2sm_kernel", "gemm2:"), ("gemm_tcgen05_kernel", "gemm:"))
                         for want in (True, False)) if r]
    if att_ms > 0:
        tr, tr_note = dram_traffic("attn_tc_kernel", a["kv_bytes"] / n_attn)
        roofs.append(dict(kernel="attn_tc_kernel", bound="hbm", achieved=round(att_gbs, 1), peak=hbm, unit="GB/s",
                          frac=round(att_gbs / hbm, 4), traffic=tr, traffic_note=tr_note, ms_per_step=round(att_ms, 4),
                          launches_per_step=n_attn, algorithmic_bytes_per_launch=round(a["kv_bytes"] / n_attn),
                          note=f"visible target-KV bytes / CUDA-event time over its launches per step, of {peaks['source']}"))
    roof = max(roofs, key=lambda r: r["ms_per_step"])            # the dominant kernel of this workload
    serial_ms = serial_roofline_ms([(n, v["flops"] / steps, v["bytes"] / steps) for n, v in res["prof"].items()],
                                   a["kv_bytes"], peaks)
    return dict(
        ms_per_step=round(ms, 4), draft_tokens_per_s=round(res["B"] * res["k"] / (ms * 1e-3), 1),
        hbm_roofline_ms=round(hbm_time_ms, 4), hbm_roofline_frac=round(hbm_time_ms / ms, 4),
        tensor_roofline_ms=round(tensor_time_ms, 4),
        max_roofline_frac=round(max(hbm_time_ms, tensor_time_ms) / ms, 4),
        serial_roofline_ms=round(serial_ms, 4), serial_roofline_frac=round(serial_ms / ms, 4),
        weight_GB=round(a["weight_bytes"] / 1e9, 3), kv_GB=round(a["kv_bytes"] / 1e9, 3),
        attention=dict(ms_per_step=round(att_ms, 4), achieved_GBs=round(att_gbs, 1), frac_of_hbm=round(att_gbs / hbm, 4),
                       launches_per_step=n_attn),
        gemm=dict(ms_per_step=round(gemm_ms, 4), achieved_TFs=round(gemm_tfs, 1), frac_of_tensor=round(gemm_tfs / tf, 4),
                  achieved_weight_GBs=round(gemm_gbs, 1), frac_of_hbm=round(gemm_gbs / hbm, 4)),
        roofline=roof, rooflines=roofs, drafter_kv_GB_avoided=round(a["drafter_kv_bytes_avoided"] / 1e9, 3),
        launches_per_step=res["launches_per_step"],
        ms_per_step_profiled=round(res["ms_per_step_profiled"], 4),
        graph_replay_ms_per_step=(round(res["graph_replay_ms_per_step"], 4)
                                  if res.get("graph_replay_ms_per_step") is not None else None),
    )


def brief(s, r=None):
    """The few figures of a summarised workload that the side tables of the bench line carry."""
    out = dict(draft_tokens_per_s=s["draft_tokens_per_s"], ms_per_step=s["ms_per_step"],
               hbm_roofline_frac=s["hbm_roofline_frac"], max_roofline_frac=s["max_roofline_frac"],
               serial_roofline_frac=s["serial_roofline_frac"],
               attention_frac_of_hbm=s["attention"]["frac_of_hbm"], weight_GB=s["weight_GB"], kv_GB=s["kv_GB"],
               graph_replay_ms_per_step=s["graph_replay_ms_per_step"])
    if r is not None:
        out["sm_mhz"] = r.get("sm_mhz")
    return out


def run_sweep(steps, warmup, peaks, rank=0):
    """The concurrency x block-size sweep on the 8B-class drafter: B in {1, 8, 32, 64, 128, 256} x k in {8, 16, 32},
    contexts uniform in [1024, 16384].  One handle (made for B <= 256, k <= 32) and one weight set serve all cells; per
    cell: warm-up, `steps` timed steps between one pair of events, then two profiled steps for the attention kernel's
    share.  Also per cell: the bytes a drafter-side KV cache over the same contexts would hold (K and V of the two
    attention layers, 8 KiB per context token; and the figure the sweep's own description spells out, one tensor of
    2 layers x 8 heads x 128 x 2 B = 4 KiB per token) against zero for in-place reuse of the target's cache."""
    import paper_2609_24197_b200 as hs
    dev = torch.device("cuda", torch.cuda.current_device())
    Bs, ks = (1, 8, 32, 64, 128, 256), (8, 16, 32)
    cfg_max = synth.get_config(f"sweep_8b_B{max(Bs)}_k{max(ks)}")
    weights = synth.make_weights(cfg_max, device=dev)
    drafter = hs.Drafter(cfg_max, weights, max(Bs), max(ks), cfg_max["ctx"][2])
    del weights
    torch.cuda.empty_cache()
    stream = torch.cuda.current_stream()
    cells = []
    for B in Bs:
        cfg = synth.get_config(f"sweep_8b_B{B}_k8")
        batch = synth.make_request_batch(cfg, device=dev, seed_offset=1000 * rank)
        ctx = batch["ctx_lens_host"]
        max_ctx = max(ctx)
        for k in ks:
            ids = torch.empty((B, k), dtype=torch.int32, device=dev)

            def step():
                hs.hspec_draft_block(drafter.handle, batch["page_table"], batch["ctx_lens"], batch["last_hidden"],
                                     batch["last_token"], k, batch["k_pools"], batch["v_pools"], drafter.workspace, ids,
                                     max_ctx=max_ctx)
            for _ in range(max(warmup, 3)):
                step()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record(stream)
            for _ in range(steps):
                step()
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / steps
            hs.hspec_set_profiling(drafter.handle, True)
            att_ms, n_prof = 0.0, 2
            for _ in range(n_prof):
                step()
                prof = hs.hspec_get_profile(drafter.handle)
                att_ms += sum(e["ms"] for e in prof if e["name"] == "attn_partial")
            hs.hspec_set_profiling(drafter.handle, False)
            att_ms /= n_prof
            a = workload_accounting(dict(cfg, k=k), ctx, B, k)
            hbm_ms = (a["weight_bytes"] + a["kv_bytes"]) / (peaks["hbm_gbs"] * 1e9) * 1e3
            tensor_ms = (a["gemm_flops"] + a["attn_flops"]) / (peaks["bf16_tflops_sustained"] * 1e12) * 1e3
            cells.append(dict(
                B=B, k=k, ms_per_step=round(ms, 4), draft_tokens_per_s=round(B * k / (ms * 1e-3), 1),
                hbm_roofline_frac=round(hbm_ms / ms, 4), max_roofline_frac=round(max(hbm_ms, tensor_ms) / ms, 4),
                serial_roofline_frac=round(serial_roofline_ms([(e["name"], e["flops"], e["bytes"]) for e in prof],
                                                              a["kv_bytes"], peaks) / ms, 4),
                attention_frac_of_hbm=round(a["kv_bytes"] / (att_ms * 1e-3) / 1e9 / peaks["hbm_gbs"], 4) if att_ms > 0 else None,
                kv_GB_read=round(a["kv_bytes"] / 1e9, 3),
                drafter_kv_GB_avoided=round(a["drafter_kv_bytes_avoided"] / 1e9, 3),
                drafter_kv_GB_avoided_single_tensor=round(a["drafter_kv_bytes_avoided"] / 2e9, 3)))
        stats = drafter.stats()
        assert stats["rc"] == 0, f"device status block not clean: {stats}"
        del batch
        torch.cuda.empty_cache()
    drafter.close()
    torch.cuda.empty_cache()
    return dict(workload="sweep_8b_B<B>_k<k>: 8B-class drafter, contexts uniform in [1024, 16384], full context",
                steps_per_cell=steps, weight_GB=round(a["weight_bytes"] / 1e9, 3),
                drafter_kv_note="bytes a drafter-side KV cache over the same contexts would hold (K and V, 2 layers: 8 KiB per "
                                "token; single_tensor = 2 layers x 8 heads x 128 x 2 B = 4 KiB per token) vs 0 for in-place reuse",
                cells=cells)


# ----------------------------------------------------------------------------- single-kernel cases (profiler captures)

def _randn(shape, seed, std, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)


def case_attention(reps, Hq=32, Hkv=8, B=32, lo=512, hi=8192, k=16, window=0, dist="uniform"):
    """One attention layer of the serving shapes: dh = 128, contexts drawn from [lo, hi]."""
    import paper_2609_24197_b200 as hs
    dh = 128
    cfg = dict(page_size=16, Hkv=Hkv, dh=dh, n_slots=1, n_fuse=1, D=8, V=16, B=B, ctx=(dist, lo, hi))
    ctx = synth.make_ctx_lens(cfg)
    batch = synth.make_request_batch(cfg, ctx_lens=ctx, device="cuda")
    M = B * k
    q, kb, vb = (_randn((M, h, dh), s, 1.0, torch.bfloat16) for h, s in ((Hq, 1), (Hkv, 2), (Hkv, 3)))
    o = torch.empty((M, Hq * dh), dtype=torch.float16, device="cuda")
    mc = max(ctx)
    ws = torch.empty(hs.hspec_attention_workspace_bytes(B, k, Hq, Hkv, dh, mc, window, 0), dtype=torch.uint8, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(reps + 1)]
    ev[0].record()
    for i in range(reps):
        hs.hspec_op_attention(q, kb, vb, batch["k_pools"][0], batch["v_pools"][0], batch["page_table"],
                              batch["ctx_lens"], mc, o, B, k, Hq, Hkv, dh, 16, window, 0, ws)
        ev[i + 1].record()
    torch.cuda.synchronize()
    kv_bytes = sum(min(c, window - 1) if window > 0 else c for c in ctx) * Hkv * dh * 2 * 2
    us = [ev[i].elapsed_time(ev[i + 1]) * 1e3 for i in range(reps)]
    print(f"attention: B={B} k={k} Hq={Hq} Hkv={Hkv} window={window} sum ctx={sum(ctx)} target-KV bytes per launch={kv_bytes} "
          f"us per call={[round(u, 1) for u in us]} -> {kv_bytes / (min(us) * 1e-6) / 1e12:.2f} TB/s")


def case_gemm(reps, M=2048, n_out=25600, K=5120):
    import paper_2609_24197_b200 as hs
    x, W = _randn((M, K), 4, 1.0, torch.float16), _randn((n_out, K), 5, 0.02, torch.float16)
    y = torch.empty((M, n_out), dtype=torch.float32, device="cuda")
    ws = torch.empty(hs.hspec_gemm_workspace_bytes(M, n_out, K), dtype=torch.uint8, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(reps + 1)]
    ev[0].record()
    for i in range(reps):
        hs.hspec_op_gemm(x, W, y, workspace=ws)
        ev[i + 1].record()
    torch.cuda.synchronize()
    us = [ev[i].elapsed_time(ev[i + 1]) * 1e3 for i in range(reps)]
    print(f"gemm: M={M} n_out={n_out} K={K} flops per launch={2 * M * n_out * K} weight bytes={2 * n_out * K} "
          f"x bytes={2 * M * K} y bytes={4 * M * n_out} us per call={[round(u, 1) for u in us]} -> "
          f"{2 * n_out * K / (min(us) * 1e-6) / 1e12:.2f} TB/s of weights, {2 * M * n_out * K / (min(us) * 1e-6) / 1e12:.0f} TFLOP/s")


def case_scan(reps, B=32, Di=8192):
    import paper_2609_24197_b200 as hs
    k, P, N, G = 16, 64, 128, 4
    H = Di // P
    ld = 2 * Di + 2 * G * N + H
    zx = _randn((B * k, ld), 6, 1.0, torch.float32)
    s0 = _randn((B, H, P, N), 7, 1.0, torch.float16)
    cw, cb = _randn((Di + 2 * G * N, 4), 8, 0.3, torch.float32), _randn((Di + 2 * G * N,), 9, 0.02, torch.float32)
    dtb, Al, Ds = _randn((H,), 10, 1.0, torch.float32) - 4, torch.rand(H, device="cuda") * 2, torch.ones(H, device="cuda")
    y = torch.empty((B * k, Di), dtype=torch.float32, device="cuda")
    ws = torch.empty(hs.hspec_scan_workspace_bytes(B, k, Di, N, G), dtype=torch.uint8, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(reps + 1)]
    ev[0].record()
    for i in range(reps):
        hs.hspec_op_mamba_scan(zx, None, s0, cw, cb, dtb, Al, Ds, y, B, k, Di, P, N, G, 4, ws)
        ev[i + 1].record()
    torch.cuda.synchronize()
    us = [round(ev[i].elapsed_time(ev[i + 1]) * 1e3, 1) for i in range(reps)]
    print(f"scan: B={B} H={H} S_init bytes per launch={B * H * P * N * 2} activation bytes (z, xBC, dt in; y out)="
          f"{B * k * (ld + Di) * 4} us per call (both kernels)={us}")


def case_rowwise(reps, M=2048, D=5120, Hq=64, Hkv=8, dh=128, k=16):
    """The row-wise kernels of a layer at the 32B-class shapes: RMSNorm over D, and per-head norm + RoPE of q, k, v."""
    import paper_2609_24197_b200 as hs
    x, w = _randn((M, D), 31, 1.0, torch.float32), 1 + _randn((D,), 32, 0.02, torch.float32)
    y = torch.empty((M, D), dtype=torch.float16, device="cuda")
    qkv = _randn((M, (Hq + 2 * Hkv) * dh), 33, 1.0, torch.float32)
    qw, kw = 1 + _randn((dh,), 34, 0.1, torch.float32), 1 + _randn((dh,), 35, 0.1, torch.float32)
    B = M // k
    ctx = torch.randint(0, 32000, (B,), dtype=torch.int32, device="cuda")
    q = torch.empty((M, Hq, dh), dtype=torch.bfloat16, device="cuda")
    kb, vb = (torch.empty((M, Hkv, dh), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * reps + 1)]
    ev[0].record()
    for i in range(reps):
        hs.hspec_op_rmsnorm(x, w, y, 1e-6)
        ev[2 * i + 1].record()
        hs.hspec_op_qk_norm_rope(qkv, qw, kw, ctx, q, kb, vb, B, k, Hq, Hkv, dh, 1e6, 1e-6, 1)
        ev[2 * i + 2].record()
    torch.cuda.synchronize()
    us = [round(ev[i].elapsed_time(ev[i + 1]) * 1e3, 1) for i in range(2 * reps)]
    print(f"rowwise: rmsnorm [{M} x {D}] fp32 -> fp16 ({M * D * 6} bytes) us={us[0::2]}; qk_norm_rope [{M} x {(Hq + 2 * Hkv) * dh}] "
          f"fp32 -> bf16 ({M * (Hq + 2 * Hkv) * dh * 6} bytes) us={us[1::2]}")


def case_overlap(reps):
    """Does the weight-streaming state projection (HBM-bound) overlap with a tensor-bound GEMM when both are in flight?
    Proj_dS of the 32B-class drafter at 128 rows (a fifth of it) on one stream, the layer's in-projection at 2048 rows
    on another: serial time vs the time with both streams fed at once."""
    import paper_2609_24197_b200 as hs
    xs, Ws = _randn((128, 5120), 11, 1.0, torch.float16), _randn((262144, 5120), 12, 0.02, torch.float16)
    ys = torch.empty((128, 262144), dtype=torch.float16, device="cuda")
    xg, Wg = _randn((2048, 5120), 13, 1.0, torch.float16), _randn((21664, 5120), 14, 0.02, torch.float16)
    yg = torch.empty((2048, 21664), dtype=torch.float32, device="cuda")
    ws_s = torch.empty(hs.hspec_gemm_workspace_bytes(128, 262144, 5120), dtype=torch.uint8, device="cuda")
    ws_g = torch.empty(hs.hspec_gemm_workspace_bytes(2048, 21664, 5120), dtype=torch.uint8, device="cuda")
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream(priority=-1)
    n_g = 5                                         # five in-projections ~ the tensor-bound work next to one projection

    def run(parallel):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        s1.wait_stream(torch.cuda.current_stream())
        s2.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s1):
            hs.hspec_op_gemm(xs, Ws, ys, workspace=ws_s)
        if not parallel:
            s2.wait_stream(s1)
        with torch.cuda.stream(s2):
            for _ in range(n_g):
                hs.hspec_op_gemm(xg, Wg, yg, workspace=ws_g)
        torch.cuda.current_stream().wait_stream(s1)
        torch.cuda.current_stream().wait_stream(s2)
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) * 1e3
    for _ in range(2):
        run(False), run(True)
    ser = [round(run(False), 1) for _ in range(reps)]
    par = [round(run(True), 1) for _ in range(reps)]
    print(f"overlap: state projection (128 x 262144 x 5120) + {n_g} x in-projection (2048 x 21664 x 5120): one after the other "
          f"{ser} us, both streams at once {par} us")


CASES = {
    # name: (function, keyword arguments) - each runs ONE kernel family a few times on inputs larger than L2
    "attention": (case_attention, {}),                                             # 8B-class, 64 query rows per KV head
    "attention32b": (case_attention, dict(Hq=64, Hkv=8, B=16, lo=2048, hi=16384)),  # 32B-class, 128 rows per KV head
    "attention32b_full": (case_attention, dict(Hq=64, Hkv=8, B=128, lo=1024, hi=32768, dist="loguniform")),  # conc128_32b's layer
    "attention8b_full": (case_attention, dict(Hq=32, Hkv=8, B=128, lo=1024, hi=16384)),                       # sweep B = 128, k = 16
    "attention32b_w2048": (case_attention, dict(Hq=64, Hkv=8, B=128, lo=2048, hi=16384, window=2048)),   # the paper's window
    "gemm": (case_gemm, {}),                                                       # the 2-SM kernel, M = 2048
    "gemm_skinny": (case_gemm, dict(M=32, n_out=65536, K=4096)),                   # weight streaming, Proj_dS class
    "gemm_skinny64": (case_gemm, dict(M=64, n_out=262144, K=5120)),                # Proj_dS at concurrency 64 (a fifth of it)
    "gemm_skinny128": (case_gemm, dict(M=128, n_out=262144, K=5120)),              # Proj_dS at concurrency 128 (a fifth of it; the 2-SM kernel)
    "scan": (case_scan, {}),
    "scan32b": (case_scan, dict(B=128, Di=10240)),                                 # conc128_32b's layer
    "rowwise": (case_rowwise, {}),
    "overlap": (case_overlap, {}),
}


def main_case(args):
    if not torch.cuda.is_available():
        raise SystemExit("bench.py --case needs a CUDA device")
    from paper_2609_24197_b200 import build
    build.build()
    fn, kw = CASES[args.case]
    fn(args.reps, **kw)


# ----------------------------------------------------------------------------- entry points

# What is measured beside the headline, in the order in which it is printed.
TABLES = ("dtype_note", "timing", "peaks", "step", "rooflines", "attention", "gemm", "kernels", "kv_injection_counterexample",
          "by_concurrency", "window_2048", "bf16_operands", "sweep")


def print_result(line):
    """The tables, a line of their own each (not JSON lines: "[bench] name: {...}"), then the ONE JSON line with the headline."""
    for name in TABLES:
        if name in line:
            print(f"[bench] {name}: {json.dumps(line[name])}")
    head = {k: v for k, v in line.items() if k not in TABLES}
    if "roofline" in head:                         # (its notes are in the rooflines table)
        head["roofline"] = {k: v for k, v in head["roofline"].items() if "note" not in k and not isinstance(v, dict)}
    print(json.dumps(head), flush=True)


def main_ours(args):
    rank, local_rank, world = dist_info()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the draft step has no CPU path")
    torch.cuda.set_device(local_rank % torch.cuda.device_count())
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", torch.cuda.current_device()))
    from paper_2609_24197_b200 import build
    if rank == 0:
        build.build()
    barrier()
    peaks = load_peaks()
    traffic = load_traffic()
    if args.sweep:                                 # only the sweep, as a line of its own
        sw = run_sweep(args.steps, args.warmup, peaks, rank)
        if rank == 0:
            head = next(c for c in sw["cells"] if c["B"] == 128 and c["k"] == 16)
            print_result({"metric": METRIC, "value": head["draft_tokens_per_s"], "unit": "draft tokens/s", "n_gpus": world,
                          "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": head["ms_per_step"],
                          "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f16",
                          "data": "synthetic", "config": {"workload": "sweep_8b_B128_k16", "note": "value = the B = 128, "
                                                          "k = 16 cell; every cell under `sweep`"},
                          "sweep": sw, "peaks": peaks})
        return
    head = run_workload(args.workload, args.steps, args.warmup, rank, clock_gpu=torch.cuda.current_device(),
                        lean=args.lean, repeats=args.repeats, settle_s=args.settle_s)
    s = summarize(head, peaks, traffic)
    e2e_ms = head["e2e"]["ms_per_step"]
    units = head["B"] * head["k"] * world
    reg = sorted(r["ms_per_step"] for r in head["regions"])
    line = {
        "metric": METRIC, "value": round(units / (head["ms_per_step"] * 1e-3), 1), "unit": "draft tokens/s",
        "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": s["ms_per_step"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f16",
        "dtype_note": "f16 tensor-core operands (bf16 weights widened exactly at load), f32 accumulate, f32 residual / scan / "
                      "softmax; the target KV is read as bf16",
        "data": "synthetic",
        "config": {"workload": args.workload, "B": head["B"], "k": head["k"], "ctx_sum": head["ctx_sum"],
                   "ctx_max": head["ctx_max"], "window": head["cfg"]["window"],
                   "parallelism": "replicas only" if world > 1 else "1 GPU",
                   "l2": f"inputs larger than L2: {s['weight_GB'] + s['kv_GB']:.1f} GB touched per step, no flush"},
        "timing": {"regions": head["regions"], "region_steps": args.steps, "ms_per_step_min": round(reg[0], 4),
                   "ms_per_step_median": s["ms_per_step"], "ms_per_step_max": round(reg[-1], 4),
                   "settle_steps_untimed": head["settle_steps"],
                   "note": "value = the median region; every region is exactly `steps` steps between one pair of CUDA events"},
        "e2e": {"value": round(units / (e2e_ms * 1e-3), 1), "unit": "draft tokens/s",
                "h2d_bytes_per_step": head["e2e"]["h2d_bytes_per_step"],
                "d2h_bytes_per_step": head["e2e"]["d2h_bytes_per_step"], "ms_per_step": round(e2e_ms, 4)},
        "gpu_launches": head["launches_per_step"] * args.steps,
        "clocks": head["clocks"],
        "roofline": s["roofline"], "rooflines": s["rooflines"],
        "step": {k: s[k] for k in ("hbm_roofline_ms", "hbm_roofline_frac", "tensor_roofline_ms", "max_roofline_frac",
                                   "serial_roofline_ms", "serial_roofline_frac",
                                   "weight_GB", "kv_GB", "drafter_kv_GB_avoided", "ms_per_step_profiled",
                                   "graph_replay_ms_per_step")},
        "attention": s["attention"], "gemm": s["gemm"], "kernels": kernel_table(head),
        "peaks": peaks,
    }
    del head["_keep"]
    torch.cuda.empty_cache()
    if world == 1 and not args.lean:
        try:
            line["kv_injection_counterexample"] = kv_injection_counterexample(head["cfg"])
        except Exception as exc:                   # a side measurement must not cost the bench line
            print(f"[bench] KV-injection counter-example skipped: {exc}", file=sys.stderr)
        torch.cuda.empty_cache()
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cb, _ = cpu_baseline(args.workload)
        cb.pop("ids")
        line["cpu_baseline"] = {k: (round(v, 3) if isinstance(v, float) else v) for k, v in cb.items()}
        torch.cuda.empty_cache()
    if world == 1 and not args.headline_only:
        byc = {}
        for conc, name in BY_CONCURRENCY.items():
            if name == args.workload:
                byc[conc] = dict(brief(s, head), workload=name)
                continue
            r = run_workload(name, args.steps, args.warmup, rank, clock_gpu=torch.cuda.current_device(), want_e2e=False,
                             settle_s=min(args.settle_s, 1.0))
            t = summarize(r, peaks, traffic)
            byc[conc] = dict(brief(t, r), workload=name, gemm=t["gemm"], rooflines=t["rooflines"], kernels=kernel_table(r))
            del r
            torch.cuda.empty_cache()
        line["by_concurrency"] = byc
        # the paper's 2048-token sliding window (App. B.1) on the two serving workloads, beside the full-context rows
        win = {}
        for name in ("serving_8b", "conc128_32b"):
            try:
                r = run_workload(name, args.steps, args.warmup, rank, clock_gpu=torch.cuda.current_device(), want_e2e=False,
                                 settle_s=min(args.settle_s, 1.0), want_graph=False, window=2048)
                t = summarize(r, peaks, traffic)
                win[name] = dict(brief(t, r), window=2048, attention=t["attention"])
                del r
            except Exception as exc:
                print(f"[bench] window row of {name} skipped: {exc}", file=sys.stderr)
            torch.cuda.empty_cache()
        line["window_2048"] = win
        # the same headline workload with bf16 tensor-core operands (act_bf16 = 1: the caller's bf16 matrices used in place,
        # bf16 activations) beside the default fp16 operands
        try:
            r = run_workload(args.workload, args.steps, args.warmup, rank, clock_gpu=torch.cuda.current_device(),
                             want_e2e=False, settle_s=min(args.settle_s, 1.0), want_graph=False, act_bf16=1)
            t = summarize(r, peaks, traffic)
            line["bf16_operands"] = dict(brief(t, r), workload=args.workload, gemm=t["gemm"],
                                         note="act_bf16 = 1; parity bound 5e-2 of the output RMS instead of 2e-2 (8-bit operands)")
            del r
        except Exception as exc:
            print(f"[bench] bf16-operand row skipped: {exc}", file=sys.stderr)
        torch.cuda.empty_cache()
        if not args.no_sweep:
            try:
                line["sweep"] = run_sweep(args.sweep_steps, args.warmup, peaks, rank)
            except Exception as exc:
                print(f"[bench] sweep skipped: {exc}", file=sys.stderr)
            torch.cuda.empty_cache()
    if rank == 0:
        print_result(line)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def main_reference(args):
    """The reference arm is the CPU oracle, timed as it stands on a bounded sample of the same workload."""
    rank, _, world = dist_info()
    if rank != 0:
        return
    cfg = synth.get_config(args.workload)
    k = cfg["k"]
    first, state = cpu_baseline(args.workload, k)
    # keep the whole run within a few minutes: shrink the sample to the first k' block rows (causal prefix property)
    n_runs = args.steps + args.warmup
    budget_s = 240.0
    if first["seconds"] * n_runs > budget_s and k > 1:
        k = max(1, int(k * budget_s / (first["seconds"] * n_runs)))
    from oracle import hspec_oracle as O
    cfg, weights, batch = state
    pools = [to_np(t) for t in batch["k_pools"]], [to_np(t) for t in batch["v_pools"]]
    times = []
    for i in range(n_runs):
        t0 = time.time()
        O.draft_block(cfg, weights, pools[0], pools[1], to_np(batch["page_table"]), batch["ctx_lens_host"],
                      to_np(batch["last_hidden"]), to_np(batch["last_token"]), k, dtype=np.float32)
        if i >= args.warmup:
            times.append(time.time() - t0)
    sec = sum(times) / len(times)
    value = k / sec
    cores = len(os.sched_getaffinity(0))
    sample = f"1 request of {args.workload} (context {batch['ctx_lens_host'][0]}), first {k} of {cfg['k']} block rows per step"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": round(value, 3), "unit": "draft tokens/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(sec * 1e3, 2), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "dtype_note": "numpy oracle on the host cores", "data": "synthetic",
        "config": {"workload": args.workload, "sample": sample},
        "cpu_baseline": {"value": round(value, 3), "unit": "draft tokens/s", "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(value, 3), "unit": "draft tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--repeats", type=int, default=5, help="timed regions of --steps steps each; value = the median one")
    ap.add_argument("--settle-s", type=float, default=2.0,
                    help="seconds of untimed steps after the warm-up, so the clocks have settled under the power cap")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default=HEADLINE,
                    help="one of %s, or a sweep cell sweep_8b_B<B>_k<k>" % ", ".join(sorted(synth.CONFIGS)))
    ap.add_argument("--headline-only", action="store_true",
                    help="skip the concurrency-1 / -32 workloads, the window rows and the sweep")
    ap.add_argument("--no-sweep", action="store_true")
    ap.add_argument("--sweep", action="store_true", help="run only the concurrency x block-size sweep (--steps per cell)")
    ap.add_argument("--sweep-steps", type=int, default=10, help="timed steps per sweep cell inside the default run")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--lean", action="store_true", help="only warm-up + timed steps (for profiler launch lists)")
    ap.add_argument("--case", choices=sorted(CASES), help="run one kernel on a small case (for profiler captures) and exit")
    ap.add_argument("--reps", type=int, default=3, help="launches of --case")
    args = ap.parse_args()
    if args.lean:
        args.repeats, args.settle_s = 1, 0.0
    if args.case:
        main_case(args)
    elif args.impl == "reference":
        main_reference(args)
    else:
        main_ours(args)


if __name__ == "__main__":
    main()
