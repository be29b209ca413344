#!/usr/bin/env python3
"""Benchmark of the selective-scan layer core on one GB300 (or N replicas).

One step = one pass of every entry point of the hot path over seeded,
synthetic inputs resident in HBM:
  1. mb_scan_prefill  MambaByte-353M-shaped layer: batch 8, L 8192, d_inner 2048,
                      d_state 16, bf16 x/z/dt/B/C, fp32 state (h0 = 0)
  2. mb_scan_verify   32 streams resuming from cached fp32 states, a drafted
                      span of k = 16 bytes, d_inner 2048, all 16 states kept
  3. mb_rollback      keep the state at each stream's seeded accept count
  4. mb_step x 48     batched decode step, batch 256, d_inner 4608 (1.6B-shaped),
                      48 layers with distinct state buffers (fp32, in place)

value = algorithmic HBM bytes of the step (each tensor counted once, read +
write) / device time, in GB/s. Per-entry-point figures, the decode rate in
generated bytes/s at batch 256, the roofline of the dominant kernel, an
end-to-end figure with host buffers, and the fp64 oracle's rate on all host
cores and on one core are added to the same JSON line, with the legs beyond the step: one
speculative-decoding iteration (verify, top-beta accept, corrector steps),
the training pass of the prefill layer (checkpointed forward, backward), the
prefill with the Delta projection fused against the unfused layer, a
single-prompt prefill (batch 1: the span split over L vs unsplit), a
whole 48-layer MambaByte decoder (kernels plus cuBLAS projections), and the
MambaByte-972M-shaped layer prefill (batch 4, d_inner 3584, given h0) timed on
its own (per_kernel.prefill_972m, not part of the step). The oracle leg also
checks the timed launches' outputs against the oracle ("parity").

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl mine|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "selective-scan HBM GB/s (% of GB300 peak); decode-step bytes/sec at batch 256"
N_STATE = 16
STEP_LAYERS = 48
PEAK_FALLBACK_GBS = 6800.0

PREFILL = dict(batch=8, seqlen=8192, d_inner=2048)
VERIFY = dict(batch=32, seqlen=16, d_inner=2048)
# MambaByte-972M-shaped layer prefill from a given h0: timed on its own, outside the step
PREFILL_972M = dict(batch=4, seqlen=8192, d_inner=3584)
STEP = dict(batch=256, seqlen=1, d_inner=4608)
WORKLOAD_NAME = ("mambabyte353m-prefill-b8-L8192-D2048 + verify-s32-k16-D2048 + rollback"
                 " + decode-step-b256-D4608-x48layers")


# ----------------------------------------------------------------------------- bytes
def bytes_prefill(batch, seqlen, d_inner, s_in=2, h0=False, h_last=True):
    rd = 3 * batch * seqlen * d_inner * s_in + 2 * batch * seqlen * N_STATE * s_in
    rd += d_inner * N_STATE * 4 + 2 * d_inner * 4 + (batch * d_inner * N_STATE * 4 if h0 else 0)
    wr = batch * seqlen * d_inner * s_in + (batch * d_inner * N_STATE * 4 if h_last else 0)
    return rd, wr


# SFU issue cost in SM clocks, measured on GB300: ex2.approx 32 / clk / SM,
# lg2.approx and rcp.approx 16 / clk / SM.
SFU_CLK_EX2, SFU_CLK_LG2_RCP = 1.0 / 32, 1.0 / 16


def sfu_clocks_per_element():
    """SM clocks of SFU work per (b, t, d, n) element of the scan: one ex2 for
    Abar, plus per (b, t, d) the softplus (ex2 + lg2) and silu (ex2 + rcp)
    shared by the 16 states."""
    per_channel_step = 2 * SFU_CLK_EX2 + 2 * SFU_CLK_LG2_RCP
    return SFU_CLK_EX2 + per_channel_step / N_STATE


def sfu_clocks_per_element_backward():
    """The backward recomputes Abar twice (state recompute and reverse sweep)
    and per (b, t, d) evaluates softplus (ex2 + lg2), silu (ex2 + rcp),
    sigmoid(dt + bias) (ex2 + rcp) and sigmoid(z) (ex2 + rcp)."""
    per_channel_step = 4 * SFU_CLK_EX2 + 4 * SFU_CLK_LG2_RCP
    return 2 * SFU_CLK_EX2 + per_channel_step / N_STATE


def sfu_roofline(elements, seconds, sms, sm_mhz, clocks_per_element=None):
    """Compute roofline of a scan kernel: elements / s against the SFU-bound
    rate sms * clock / clocks_per_element (default: the forward scan's)."""
    cpe = clocks_per_element or sfu_clocks_per_element()
    peak = sms * sm_mhz * 1e6 / cpe
    achieved = elements / seconds
    return {"bound": "sfu", "unit": "elements/s", "elements_per_launch": elements,
            "achieved": round(achieved, 1), "peak": round(peak, 1), "frac": round(achieved / peak, 4),
            "peak_basis": f"{sms} SMs x {sm_mhz:.0f} MHz / {cpe:.5f} SFU clocks"
                          " per element (measured ex2 32/clk/SM, lg2 and rcp 16/clk/SM)"}


def bytes_backward(batch, seqlen, d_inner, s_in=2, h0=False, dh_last=True):
    """Training backward: reads x, z, dt, dout, B, C, the parameters, the state
    checkpoints (one per 16 steps), [h0], [dh_last]; writes dx, ddt, dz,
    dB, dC (fp32), dA, dD, ddt_bias and dh0."""
    nch = (seqlen + 15) // 16
    st = batch * d_inner * N_STATE * 4
    rd = 4 * batch * seqlen * d_inner * s_in + 2 * batch * seqlen * N_STATE * s_in
    rd += d_inner * N_STATE * 4 + 2 * d_inner * 4 + nch * st + (st if h0 else 0) + (st if dh_last else 0)
    wr = 3 * batch * seqlen * d_inner * s_in + 2 * batch * seqlen * N_STATE * 4
    wr += d_inner * N_STATE * 4 + 2 * d_inner * 4 + st
    return rd, wr


def bytes_verify(batch, seqlen, d_inner, s_in=2):
    rd, _ = bytes_prefill(batch, seqlen, d_inner, s_in, h0=True, h_last=False)
    wr = batch * seqlen * d_inner * s_in + batch * seqlen * d_inner * N_STATE * 4
    return rd, wr


def bytes_rollback(batch, d_inner):
    per = batch * d_inner * N_STATE * 4
    return per + batch * 4, per


def bytes_step(batch, d_inner, s_in=2):
    st = batch * d_inner * N_STATE * 4
    rd = st + 3 * batch * d_inner * s_in + 2 * batch * N_STATE * s_in + d_inner * N_STATE * 4 + 2 * d_inner * 4
    wr = st + batch * d_inner * s_in
    return rd, wr


def step_bytes():
    parts = {
        "prefill": sum(bytes_prefill(**PREFILL)),
        "verify": sum(bytes_verify(**VERIFY)),
        "rollback": sum(bytes_rollback(VERIFY["batch"], VERIFY["d_inner"])),
        "step": STEP_LAYERS * sum(bytes_step(STEP["batch"], STEP["d_inner"])),
    }
    return parts


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return PEAK_FALLBACK_GBS, "fallback"


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi clock / throttle samples every 200 ms while running."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap,uuid")

    def __init__(self, uuid=None):
        self.uuid = uuid
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return self

        def reader():
            for line in self.proc.stdout:
                self.rows.append([c.strip() for c in line.split(",")])
        self.thread = threading.Thread(target=reader, daemon=True)
        self.thread.start()
        return self

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        rows = [r for r in self.rows if len(r) >= 9 and (self.uuid is None or r[8] == self.uuid)]
        if not rows:
            return None
        sm = [float(r[0]) for r in rows if r[0].replace(".", "").isdigit()]
        smax = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[4 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": reasons,
                "samples": len(rows)}


# ----------------------------------------------------------------------------- GPU arm
def source_sha(sources):
    """First 16 hex digits of the SHA-256 of the concatenated csrc files named
    in `sources` (comma-separated: a kernel's .cu and the headers it includes);
    None if one is missing."""
    h = hashlib.sha256()
    for name in sources.split(","):
        src = os.path.join(ROOT, "paper_2401_13660_gb300", "csrc", name)
        if not name or not os.path.exists(src):
            return None
        h.update(open(src, "rb").read())
    return h.hexdigest()[:16]


def traffic_from_profiles(kernel_key):
    """DRAM bytes per launch from the committed ncu summary, if the kernel source
    is unchanged since it was taken (else None)."""
    path = os.path.join(ROOT, "profiles", "ncu_traffic.txt")
    if not os.path.exists(path):
        return None
    for line in open(path):
        kv = dict(p.split("=", 1) for p in line.split() if "=" in p)
        if kv.get("kernel") != kernel_key:
            continue
        if source_sha(kv.get("source", "")) != kv.get("sha"):
            return None
        return float(kv["bytes_per_launch"]) * float(kv.get("scale", 1.0))
    return None


def kernel_name(group, prefill_ws_bytes):
    """The kernel (csrc/) that a group of the step launches. The prefill runs in even shares where the library asked
    for scratch beyond the 256-byte status block on this GPU, else as one CTA per channel tile."""
    prefill = "forward_shares_kernel" if prefill_ws_bytes > 256 else "forward_kernel"
    return {"prefill": prefill, "verify": "prefill_kernel", "rollback": "rollback_kernel", "step": "step_kernel"}[group]


def reduce_max(value, dist, device="cpu"):
    """Max of a float over all ranks (the slowest rank sets the job time)."""
    if not dist:
        return float(value)
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def build_gpu_state(dev):
    import torch

    from paper_2401_13660_gb300 import mbscan as mb
    from paper_2401_13660_gb300.inputs import make_inputs

    def alloc(inp, h_last=False, h_all=False, seed_accept=False):
        x = inp["x"]
        out = dict(inp)
        out["y"] = torch.empty_like(x)
        out["ws"] = torch.zeros(256, dtype=torch.uint8, device=dev)
        if "dt" in inp and x.shape[1] > 1:   # the scratch that the library asks for (a decode step needs none)
            out["ws"] = mb.new_workspace(mb.make_args(x, inp["dt"], inp["B"], inp["C"], inp["A"], out["y"],
                                                      z=inp["z"]), dev)
        if h_last:
            out["h_last"] = torch.empty(x.shape[0], x.shape[2], N_STATE, device=dev)
        if h_all:
            out["h_all"] = torch.empty(x.shape[0], x.shape[1], x.shape[2], N_STATE, device=dev)
            out["h_keep"] = torch.empty(x.shape[0], x.shape[2], N_STATE, device=dev)
        return out

    P = alloc(make_inputs(**PREFILL, d_state=N_STATE, dtype="bf16", h0="zeros", seed=1,
                          device=dev), h_last=True)
    V = alloc(make_inputs(**VERIFY, d_state=N_STATE, dtype="bf16", h0="normal", seed=3,
                          device=dev, accept=True), h_all=True)
    S = []
    for layer in range(STEP_LAYERS):
        inp = make_inputs(**STEP, d_state=N_STATE, dtype="bf16", h0="normal", seed=4000 + layer,
                          device=dev)
        inp["state"] = inp.pop("h0")
        S.append(alloc(inp))
    return P, V, S


def run_step(mb, P, V, S, stream, events=None):
    """Launch one whole step on `stream`; record an event after each group."""
    ev = iter(events) if events is not None else None
    mb.mb_scan_prefill(P["x"], P["dt"], P["B"], P["C"], P["A"], P["y"], z=P["z"], D=P["D"],
                       dt_bias=P["dt_bias"], h0=P["h0"], h_last=P["h_last"], ws=P["ws"], stream=stream)
    if ev:
        next(ev).record(stream)
    mb.mb_scan_verify(V["x"], V["dt"], V["B"], V["C"], V["A"], V["y"], V["h_all"], z=V["z"],
                      D=V["D"], dt_bias=V["dt_bias"], h0=V["h0"], ws=V["ws"], stream=stream)
    if ev:
        next(ev).record(stream)
    mb.mb_rollback(V["h0"], V["h_all"], V["accept"], V["h_keep"], ws=V["ws"], stream=stream)
    if ev:
        next(ev).record(stream)
    for L in S:
        mb.mb_step(L["x"], L["dt"], L["B"], L["C"], L["A"], L["y"], L["state"], z=L["z"], D=L["D"],
                   dt_bias=L["dt_bias"], ws=L["ws"], stream=stream)
    if ev:
        next(ev).record(stream)


LAUNCHES_PER_STEP = 3 + STEP_LAYERS


def step_groups(mb, P, V, S, stream):
    """The step's launch groups (prefill, verify, rollback, the 48 decode steps)."""
    return [
        lambda: mb.mb_scan_prefill(P["x"], P["dt"], P["B"], P["C"], P["A"], P["y"], z=P["z"], D=P["D"],
                                   dt_bias=P["dt_bias"], h0=P["h0"], h_last=P["h_last"], ws=P["ws"],
                                   stream=stream),
        lambda: mb.mb_scan_verify(V["x"], V["dt"], V["B"], V["C"], V["A"], V["y"], V["h_all"], z=V["z"],
                                  D=V["D"], dt_bias=V["dt_bias"], h0=V["h0"], ws=V["ws"], stream=stream),
        lambda: mb.mb_rollback(V["h0"], V["h_all"], V["accept"], V["h_keep"], ws=V["ws"], stream=stream),
        lambda: [mb.mb_step(L["x"], L["dt"], L["B"], L["C"], L["A"], L["y"], L["state"], z=L["z"],
                            D=L["D"], dt_bias=L["dt_bias"], ws=L["ws"], stream=stream) for L in S],
    ]


def capture_timed_graph(mb, P, V, S, stream, K):
    """All K timed steps in one CUDA graph, with timing events recorded inside
    it (external event nodes) at the start and after every launch group, so one
    replay runs the timed region with no host launches or gaps between graphs.
    Returns (graph, start event, [K][4] end events), or None where this
    PyTorch has no external events."""
    import torch

    try:
        start = torch.cuda.Event(enable_timing=True, external=True)
        ends = [[torch.cuda.Event(enable_timing=True, external=True) for _ in range(4)] for _ in range(K)]
    except TypeError:
        return None
    groups = step_groups(mb, P, V, S, stream)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        start.record(stream)
        for k in range(K):
            for gi, fn in enumerate(groups):
                fn()
                ends[k][gi].record(stream)
    return g, start, ends


def capture_step_graphs(mb, P, V, S, stream):
    """One CUDA graph per launch group of the step (prefill, verify, rollback,
    the 48 decode steps), captured on `stream` after warm-up. Replaying them
    times the device work without the Python/ctypes cost of 51 launches per
    step starving the GPU between the short decode kernels."""
    import torch

    groups = step_groups(mb, P, V, S, stream)
    graphs = []
    for fn in groups:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            fn()
        graphs.append(g)
    return graphs


def gpu_arm(args, rank, world, dist):
    import torch

    from paper_2401_13660_gb300 import mbscan as mb

    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", 0)))
    torch.cuda.set_device(dev)
    mb.load_library()
    P, V, S = build_gpu_state(dev)
    stream = torch.cuda.Stream(dev)
    parts = step_bytes()
    total_bytes = sum(parts.values())

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            run_step(mb, P, V, S, stream)
    stream.synchronize()
    for ws in [P["ws"], V["ws"]] + [L["ws"] for L in S]:
        st, det = mb.mb_check(ws, stream)
        if st != mb.MB_OK:
            raise RuntimeError(f"device-side status {mb.mb_status_string(st)} ({det})")

    uuid = None
    try:
        uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    clocks = ClockSampler(uuid).start() if rank == 0 else None

    K = args.steps
    # preferred: the K timed steps in one graph with timing events inside it;
    # else one graph per launch group replayed per step; --eager: no graphs
    timed = None if args.eager else capture_timed_graph(mb, P, V, S, stream, K)
    graphs = None if (args.eager or timed) else capture_step_graphs(mb, P, V, S, stream)
    with torch.cuda.stream(stream):
        if timed:
            timed[0].replay()   # one untimed replay (K steps)
        for g in graphs or []:
            g.replay()          # one untimed replay of each graph
    stream.synchronize()

    if timed:
        _, start, ends = timed
    else:
        start = torch.cuda.Event(enable_timing=True)
        ends = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(K)]
    if dist:
        dist.barrier()
    torch.cuda.synchronize(dev)
    with torch.cuda.stream(stream):
        if timed:
            timed[0].replay()
        else:
            start.record(stream)
            for k in range(K):
                if graphs:
                    for gi, g in enumerate(graphs):
                        g.replay()
                        ends[k][gi].record(stream)
                else:
                    run_step(mb, P, V, S, stream, ends[k])
    stream.synchronize()
    torch.cuda.synchronize(dev)
    if dist:
        dist.barrier()
    clock_rec = clocks.stop() if clocks else None
    snap = snapshot_outputs(P, V)   # the timed launches' outputs, for the parity check

    # per-group device time
    groups = ["prefill", "verify", "rollback", "step"]
    tot = {g: 0.0 for g in groups}
    prev = start
    for k in range(K):
        for gi, g in enumerate(groups):
            tot[g] += prev.elapsed_time(ends[k][gi])
            prev = ends[k][gi]
    elapsed_ms = reduce_max(start.elapsed_time(ends[K - 1][3]), dist, dev)

    peak, peak_kind = load_peaks()
    per_kernel = {}
    launches = {"prefill": 1, "verify": 1, "rollback": 1, "step": STEP_LAYERS}
    for g in groups:
        ms = tot[g] / K
        gbs = parts[g] / (ms * 1e-3) / 1e9 if ms > 0 else None
        per_kernel[g] = {"ms_per_step": round(ms, 5), "us_per_launch": round(1e3 * ms / launches[g], 3),
                         "bytes_per_step": parts[g], "GB/s": round(gbs, 1) if gbs else None,
                         "frac_of_peak": round(gbs / peak, 4) if gbs else None,
                         "share": round(tot[g] / sum(tot.values()), 4)}
    props = torch.cuda.get_device_properties(dev)
    sm_mhz = (clock_rec or {}).get("sm_mhz") or (clock_rec or {}).get("sm_max_mhz") or 2070.0
    pf = PREFILL
    per_kernel["prefill"]["compute_roofline"] = sfu_roofline(
        pf["batch"] * pf["seqlen"] * pf["d_inner"] * N_STATE, tot["prefill"] / K * 1e-3,
        props.multi_processor_count, float(sm_mhz))
    dom = max(groups, key=lambda g: tot[g])
    dom_launch_ms = tot[dom] / (K * launches[dom])
    dom_bytes = parts[dom] / launches[dom]
    achieved = dom_bytes / (dom_launch_ms * 1e-3) / 1e9
    kernel_key = kernel_name(dom, P["ws"].numel())
    roofline = {"kernel": kernel_key, "bound": "hbm", "achieved": round(achieved, 1),
                "peak": peak, "peak_kind": f"{peak_kind} (hbm_gbs)", "unit": "GB/s",
                "frac": round(achieved / peak, 4), "traffic": traffic_from_profiles(kernel_key),
                "algorithmic_bytes_per_launch": dom_bytes}

    value = world * total_bytes * K / (elapsed_ms * 1e-3) / 1e9
    step_ms = tot["step"] / K
    line = {
        "metric": METRIC, "value": round(value, 1), "unit": "GB/s", "n_gpus": world,
        "steps": K, "warmup": args.warmup, "ms_per_step": round(elapsed_ms / K, 5),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "io_dtype": "bf16", "data": "synthetic (seeded; shapes of MambaByte layers)",
        "config": {"workload": WORKLOAD_NAME, "prefill": PREFILL, "verify": VERIFY,
                   "decode_step": dict(STEP, layers=STEP_LAYERS), "d_state": N_STATE,
                   "l2": "no explicit flush: every step streams > 8 GB (> 129 MB L2) and the 48 "
                         "decode layers rotate distinct buffers, so each kernel starts cold",
                   "parallelism": f"replicas x{world}",
                   "launch": "eager (one binding call per kernel)" if args.eager else
                             ("one CUDA graph holding the K timed steps (captured after warm-up, replayed "
                              "once untimed, then once timed), CUDA timing events recorded inside it "
                              "after each launch group" if timed else
                              "CUDA graphs: one per launch group (prefill, verify, rollback, 48 decode "
                              "steps), captured after warm-up and replayed per step")},
        "frac_of_peak": round(value / world / peak, 4),
        "decode_step": {"batch": STEP["batch"], "layers": STEP_LAYERS,
                        "generated_bytes_per_s": round(world * STEP["batch"] / (step_ms * 1e-3), 1),
                        "ms_per_48_layers": round(step_ms, 5),
                        "GB/s": per_kernel["step"]["GB/s"]},
        "per_kernel": per_kernel, "roofline": roofline, "gpu_launches": LAUNCHES_PER_STEP * K,
        "clocks": clock_rec,
    }
    pk972, snap972 = prefill_972m_leg(args, mb, stream, dev, dist, peak)
    per_kernel["prefill_972m"] = pk972
    if not args.no_e2e:
        line["e2e"] = e2e_leg(args, mb, P, V, S, stream, dev, total_bytes, world, dist)
    line["speculative_iteration"] = spec_iteration_leg(args, mb, V, stream, dev, dist)
    if not args.no_training:
        line["training"] = training_leg(args, mb, P, stream, dev, dist)
    if not args.no_fused_delta:
        line["fused_delta"] = fused_delta_leg(args, mb, stream, dev, dist)
    if not args.no_prompt_prefill:
        line["prompt_prefill"] = prompt_prefill_leg(args, mb, stream, dev, dist)
    if not args.no_decode_model:
        line["decode_model"] = decode_model_leg(args, dev, dist, peak)
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(P, V, S, args.cpu_fraction)
        line["parity"] = oracle_parity(mb, P, V, S, snap, snap972, stream)
    return line


# channels sampled for the parity check of the full-size prefills (as in the
# full-size GPU parity test): 2 batch rows x 64 random channels + the first
# and last channel, over the whole 8192-byte span
def prefill_sample(batch, d_inner, seed=7):
    import torch

    g = torch.Generator().manual_seed(seed)
    rows = sorted(torch.randperm(batch, generator=g)[:2].tolist())
    chans = sorted(set(torch.randperm(d_inner, generator=g)[:64].tolist()) | {0, d_inner - 1})
    return rows, chans


def _sample_prefill_outputs(inp, rows, chans):
    import torch

    dev = inp["x"].device
    r_t, c_t = torch.tensor(rows, device=dev), torch.tensor(chans, device=dev)
    return {"rows": rows, "chans": chans, "y": inp["y"].index_select(0, r_t)[:, :, c_t].cpu(),
            "h_last": inp["h_last"].index_select(0, r_t)[:, c_t].cpu()}


def snapshot_outputs(P, V):
    """Copies of the outputs of the timed launches (the inputs never change, so
    the last timed launch's outputs are every timed launch's): the sampled
    channels of the prefill, all of verify (y, h_all) and of the rollback."""
    rows, chans = prefill_sample(PREFILL["batch"], PREFILL["d_inner"])
    return {"prefill": _sample_prefill_outputs(P, rows, chans),
            "verify_y": V["y"].cpu(), "verify_h_all": V["h_all"].cpu(), "rollback": V["h_keep"].cpu()}


def prefill_972m_leg(args, mb, stream, dev, dist, peak):
    """The MambaByte-972M-shaped layer prefill (batch 4, L 8192, d_inner 3584,
    bf16, h0 ~ N(0, 0.1^2)) timed on its own: one CUDA graph of the launch,
    replayed K times between CUDA events on the launching stream (0.94 GB of
    inputs and outputs per launch, > 129 MB L2). Not part of the step's value."""
    import torch

    from paper_2401_13660_gb300.inputs import make_inputs

    c = PREFILL_972M
    inp = make_inputs(**c, d_state=N_STATE, dtype="bf16", h0="normal", seed=2, device=dev)
    inp["y"] = torch.empty_like(inp["x"])
    inp["h_last"] = torch.empty(c["batch"], c["d_inner"], N_STATE, device=dev)
    ws = mb.new_workspace(mb.make_args(inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"], inp["y"], z=inp["z"]), dev)

    def fn():
        mb.mb_scan_prefill(inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"], inp["y"], z=inp["z"], D=inp["D"],
                           dt_bias=inp["dt_bias"], h0=inp["h0"], h_last=inp["h_last"], ws=ws, stream=stream)

    K = max(3, min(args.steps, 30))
    with torch.cuda.stream(stream):
        for _ in range(3):
            fn()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            fn()
        graph.replay()
        stream.synchronize()
        st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        st.record(stream)
        for _ in range(K):
            graph.replay()
        en.record(stream)
        en.synchronize()
    us = reduce_max(1e3 * st.elapsed_time(en) / K, dist, dev)
    st_, md = mb.mb_check(ws, stream)
    if st_ != mb.MB_OK:
        raise RuntimeError(f"device-side status {mb.mb_status_string(st_)} ({md})")
    nb = sum(bytes_prefill(**c, h0=True))
    gbs = nb / (us * 1e-6) / 1e9
    props = torch.cuda.get_device_properties(dev)
    out = {"config": "MambaByte-972M-shaped layer: batch 4, L 8192, d_inner 3584, bf16, h0 ~ N(0, 0.1^2)",
           "in_step": False, "us_per_launch": round(us, 3), "bytes_per_launch": nb, "GB/s": round(gbs, 1),
           "frac_of_peak": round(gbs / peak, 4), "timed_launches": K,
           "compute_roofline": sfu_roofline(c["batch"] * c["seqlen"] * c["d_inner"] * N_STATE, us * 1e-6,
                                            props.multi_processor_count, 2070.0)}
    rows, chans = prefill_sample(c["batch"], c["d_inner"])
    snap = _sample_prefill_outputs(inp, rows, chans)
    snap["inputs"] = {k: (None if v is None else v.cpu()) for k, v in inp.items() if k not in ("y", "h_last")}
    del inp
    torch.cuda.empty_cache()
    return out, snap


SPEC_CORRECT_STEPS = 4   # corrector bytes per iteration (one subword's worth)


def spec_iteration_leg(args, mb, V, stream, dev, dist):
    """One speculative-decoding iteration of Algorithm 1 on the verify workload
    (32 streams, 16 drafted bytes, d_inner 2048), entirely on the device:
    verify from the cached state -> top-beta accept counts from (synthetic)
    verifier scores -> SPEC_CORRECT_STEPS corrector decode steps, the first of
    which resumes from the accepted prefix (mb_step_resume: rollback fused
    into the step). The unfused form (mb_rollback, then plain steps) is timed
    alongside."""
    import torch

    from paper_2401_13660_gb300.inputs import make_inputs

    b, k, Dn = VERIFY["batch"], VERIFY["seqlen"], VERIFY["d_inner"]
    g = torch.Generator(device=dev).manual_seed(11)
    logits = torch.randn(b, k, 256, device=dev, generator=g).to(torch.bfloat16)
    drafted = torch.where(torch.rand(b, k, device=dev, generator=g) < 0.15,
                          torch.randint(0, 256, (b, k), device=dev, generator=g),
                          logits.float().argmax(dim=2)).to(torch.uint8)
    accept = torch.empty(b, dtype=torch.int32, device=dev)
    cache = V["h0"].clone()
    corr = [make_inputs(b, 1, Dn, N_STATE, "bf16", "zeros", seed=900 + i, device=dev) for i in
            range(SPEC_CORRECT_STEPS)]
    ycorr = [torch.empty_like(c["x"]) for c in corr]

    def verify_accept():
        mb.mb_scan_verify(V["x"], V["dt"], V["B"], V["C"], V["A"], V["y"], V["h_all"], z=V["z"],
                          D=V["D"], dt_bias=V["dt_bias"], h0=cache, ws=V["ws"], stream=stream)
        mb.mb_accept_topk(logits, drafted, 3, accept, stream=stream)

    def step(c, yc):
        mb.mb_step(c["x"], c["dt"], c["B"], c["C"], V["A"], yc, cache, z=c["z"], D=V["D"],
                   dt_bias=V["dt_bias"], ws=V["ws"], stream=stream)

    def fused():
        verify_accept()
        c, yc = corr[0], ycorr[0]
        mb.mb_step_resume(c["x"], c["dt"], c["B"], c["C"], V["A"], yc, V["h_all"], accept, cache,
                          z=c["z"], D=V["D"], dt_bias=V["dt_bias"], h0=cache, ws=V["ws"], stream=stream)
        for c, yc in zip(corr[1:], ycorr[1:]):
            step(c, yc)

    def unfused():
        verify_accept()
        mb.mb_rollback(cache, V["h_all"], accept, cache, ws=V["ws"], stream=stream)
        for c, yc in zip(corr, ycorr):
            step(c, yc)

    def timed(fn):
        with torch.cuda.stream(stream):
            for _ in range(3):
                fn()
            stream.synchronize()
        run = fn
        if not args.eager:   # replay one graph per iteration (6 short launches)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                fn()
            run = graph.replay
        with torch.cuda.stream(stream):
            run()
            stream.synchronize()
            K = max(10, args.steps)
            st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.record(stream)
            for _ in range(K):
                run()
            en.record(stream)
            en.synchronize()
        return reduce_max(1e3 * st.elapsed_time(en) / K, dist, dev)

    # rounds whose corrector loop adds no byte: the next verify starts from the
    # state kept at the bifurcation (h_all of the previous round, ping-pong)
    h_all_b = torch.empty_like(V["h_all"])
    accept_b = torch.empty_like(accept)
    kept = torch.empty_like(cache)
    vkw = dict(z=V["z"], D=V["D"], dt_bias=V["dt_bias"], ws=V["ws"], stream=stream)

    def rounds_fused():
        for src, dst, a_in, a_out in ((V["h_all"], h_all_b, accept, accept_b), (h_all_b, V["h_all"], accept_b, accept)):
            mb.mb_scan_verify_resume(V["x"], V["dt"], V["B"], V["C"], V["A"], V["y"], dst, src, a_in, h0=cache, **vkw)
            mb.mb_accept_topk(logits, drafted, 3, a_out, stream=stream)

    def rounds_unfused():
        for src, dst, a_in, a_out in ((V["h_all"], h_all_b, accept, accept_b), (h_all_b, V["h_all"], accept_b, accept)):
            mb.mb_rollback(cache, src, a_in, kept, ws=V["ws"], stream=stream)
            mb.mb_scan_verify(V["x"], V["dt"], V["B"], V["C"], V["A"], V["y"], dst, h0=kept, **vkw)
            mb.mb_accept_topk(logits, drafted, 3, a_out, stream=stream)

    us_unfused = timed(unfused)
    us = timed(fused)
    us_rounds_unfused = timed(rounds_unfused) / 2
    us_rounds = timed(rounds_fused) / 2
    mean_acc = float(accept.float().mean().item())
    return {"streams": b, "drafted_bytes": k, "d_inner": Dn, "beta": 3,
            "corrector_steps": SPEC_CORRECT_STEPS, "us_per_iteration": round(us, 3),
            "launches_per_iteration": 2 + SPEC_CORRECT_STEPS,
            "us_per_iteration_unfused_rollback": round(us_unfused, 3),
            "us_per_round_no_corrector": round(us_rounds, 3),
            "us_per_round_no_corrector_unfused_rollback": round(us_rounds_unfused, 3),
            "mean_accepted_bytes": round(mean_acc, 2),
            "note": "verify + accept + corrector steps (first one resumes from h_all: rollback "
                    "fused) on one layer; rounds with no corrector byte: the next verify resumes "
                    "from the previous h_all (mb_scan_verify_resume) vs mb_rollback + mb_scan_verify; "
                    "scores synthetic"}


def training_leg(args, mb, P, stream, dev, dist):
    """Training pass of the 353M-shaped layer on its prefill inputs: the
    forward with state checkpoints, then the backward from seeded dJ/dout and
    dJ/dh_last. Each is replayed from a CUDA graph and timed with CUDA events."""
    import torch

    b, L, Dn = PREFILL["batch"], PREFILL["seqlen"], PREFILL["d_inner"]
    g = torch.Generator(device=dev).manual_seed(21)
    dout = torch.randn(b, L, Dn, device=dev, generator=g).to(torch.bfloat16)
    dh_last = torch.randn(b, Dn, N_STATE, device=dev, generator=g)
    h_ckpt = torch.empty(b, (L + 15) // 16, Dn, N_STATE, device=dev)
    grads = {}

    def fwd():
        mb.mb_scan_prefill_ckpt(P["x"], P["dt"], P["B"], P["C"], P["A"], P["y"], h_ckpt, z=P["z"], D=P["D"],
                                dt_bias=P["dt_bias"], h0=P["h0"], h_last=P["h_last"], ws=P["ws"], stream=stream)

    def bwd():
        mb.mb_scan_backward(P["x"], P["dt"], P["B"], P["C"], P["A"], h_ckpt, dout, z=P["z"], D=P["D"],
                            dt_bias=P["dt_bias"], h0=P["h0"], dh_last=dh_last, grads=grads, ws=P["ws"],
                            stream=stream)

    with torch.cuda.stream(stream):
        fwd()
        grads.update(mb.mb_scan_backward(P["x"], P["dt"], P["B"], P["C"], P["A"], h_ckpt, dout, z=P["z"],
                                         D=P["D"], dt_bias=P["dt_bias"], h0=P["h0"], dh_last=dh_last,
                                         ws=P["ws"], stream=stream))
    stream.synchronize()
    K = max(3, min(args.steps, 20))
    out = {}
    for name, fn in (("forward_ckpt", fwd), ("backward", bwd)):
        with torch.cuda.stream(stream):
            for _ in range(2):
                fn()
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                fn()
            graph.replay()
            stream.synchronize()
            st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.record(stream)
            for _ in range(K):
                graph.replay()
            en.record(stream)
            en.synchronize()
        out[name] = reduce_max(1e3 * st.elapsed_time(en) / K, dist, dev)
    st_, md = mb.mb_check(P["ws"], stream)
    if st_ != mb.MB_OK:
        raise RuntimeError(f"device-side status {mb.mb_status_string(st_)} ({md})")
    props = torch.cuda.get_device_properties(dev)
    elements = b * L * Dn * N_STATE
    bwd_bytes = sum(bytes_backward(b, L, Dn))
    fwd_bytes = sum(bytes_prefill(b, L, Dn)) + b * ((L + 15) // 16) * Dn * N_STATE * 4
    return {"config": "353M-shaped layer: batch 8, L 8192, d_inner 2048, bf16; dJ/dout, dJ/dh_last seeded",
            "forward_ckpt_us": round(out["forward_ckpt"], 2), "backward_us": round(out["backward"], 2),
            "forward_ckpt_GB/s": round(fwd_bytes / (out["forward_ckpt"] * 1e-6) / 1e9, 1),
            "backward_GB/s": round(bwd_bytes / (out["backward"] * 1e-6) / 1e9, 1),
            "backward_algorithmic_bytes": bwd_bytes,
            "backward_compute_roofline": sfu_roofline(elements, out["backward"] * 1e-6,
                                                      props.multi_processor_count, 2070.0,
                                                      sfu_clocks_per_element_backward()),
            "timed_launches": K}


def fused_delta_leg(args, mb, stream, dev, dist):
    """The low-rank Delta projection of Eq. 3 (dt = W_Delta (W_R x), r = 64 for
    the 353M layer) two ways on the same seeded inputs: unfused, a cuBLAS bf16
    GEMM writing dt [b, L, d_inner] followed by the prefill kernel; fused, the
    prefill kernel forming dt tile by tile on the tensor cores from dt_low and
    W_dt. Each is replayed from a CUDA graph and timed with CUDA events."""
    import torch

    from paper_2401_13660_gb300.inputs import WORKLOADS, workload_inputs

    w = WORKLOADS["mambabyte353m_prefill_fused_r64_b8_L8192"]
    inp = workload_inputs(w, dev)
    b, L, Dn, r = w.batch, w.seqlen, w.d_inner, w.dt_rank
    y = torch.empty_like(inp["x"])
    hl = torch.empty(b, Dn, N_STATE, device=dev)
    dt = torch.empty(b, L, Dn, device=dev, dtype=torch.bfloat16)
    ws = torch.zeros(256, dtype=torch.uint8, device=dev)
    common = dict(z=inp["z"], D=inp["D"], dt_bias=inp["dt_bias"], h0=inp["h0"], h_last=hl, ws=ws, stream=stream)

    def unfused():
        torch.matmul(inp["dt_low"], inp["W_dt"].t(), out=dt)
        mb.mb_scan_prefill(inp["x"], dt, inp["B"], inp["C"], inp["A"], y, **common)

    def fused():
        mb.mb_scan_prefill(inp["x"], None, inp["B"], inp["C"], inp["A"], y, dt_low=inp["dt_low"], W_dt=inp["W_dt"],
                           **common)

    K = max(3, min(args.steps, 10))
    out = {}
    for name, fn in (("unfused_gemm_then_prefill", unfused), ("fused", fused)):
        with torch.cuda.stream(stream):
            for _ in range(2):
                fn()
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                fn()
            graph.replay()
            stream.synchronize()
            st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.record(stream)
            for _ in range(K):
                graph.replay()
            en.record(stream)
            en.synchronize()
        out[name] = reduce_max(1e3 * st.elapsed_time(en) / K, dist, dev)
    st_, md = mb.mb_check(ws, stream)
    if st_ != mb.MB_OK:
        raise RuntimeError(f"device-side status {mb.mb_status_string(st_)} ({md})")
    return {"config": f"353M-shaped layer: batch {b}, L {L}, d_inner {Dn}, dt_rank {r}, bf16",
            "unfused_us": round(out["unfused_gemm_then_prefill"], 2), "fused_us": round(out["fused"], 2),
            "dt_bytes_saved": b * L * Dn * 2, "timed_launches": K,
            "note": "unfused = cuBLAS GEMM dt_low W_dt^T (bf16 out) + prefill kernel; fused = prefill kernel "
                    "forming dt on the tensor cores (dt kept in fp32, never stored)"}


def prompt_prefill_leg(args, mb, stream, dev, dist):
    """Prefill of a single prompt (batch 1, 8192 bytes, d_inner 2048: 64 channel
    tiles for 152 SMs) with the workspace mb_workspace_size asks for (the span
    is split over L: summaries, then every segment from its folded start
    state) against a 256-byte workspace (unsplit). CUDA graphs, CUDA events."""
    import torch

    from paper_2401_13660_gb300.inputs import make_inputs

    b, L, Dn = 1, 8192, 2048
    inp = make_inputs(b, L, Dn, N_STATE, "bf16", "zeros", seed=12, device=dev)
    y = torch.empty_like(inp["x"])
    hl = torch.empty(b, Dn, N_STATE, device=dev)
    a = mb.make_args(inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"], y, z=inp["z"])
    out = {}
    K = max(3, min(args.steps, 20))
    for name, nbytes in (("unsplit", 256), ("split", mb.mb_workspace_size(a))):
        ws = torch.zeros(max(nbytes, 256), dtype=torch.uint8, device=dev)

        def fn():
            mb.mb_scan_prefill(inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"], y, z=inp["z"], D=inp["D"],
                               dt_bias=inp["dt_bias"], h_last=hl, ws=ws, stream=stream)
        with torch.cuda.stream(stream):
            for _ in range(2):
                fn()
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                fn()
            graph.replay()
            stream.synchronize()
            st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.record(stream)
            for _ in range(K):
                graph.replay()
            en.record(stream)
            en.synchronize()
        out[name] = reduce_max(1e3 * st.elapsed_time(en) / K, dist, dev)
        st_, md = mb.mb_check(ws, stream)
        if st_ != mb.MB_OK:
            raise RuntimeError(f"device-side status {mb.mb_status_string(st_)} ({md})")
    nb = sum(bytes_prefill(b, L, Dn))
    return {"config": f"batch {b}, L {L}, d_inner {Dn}, bf16 (one prompt)",
            "unsplit_us": round(out["unsplit"], 2), "split_us": round(out["split"], 2),
            "split_GB/s": round(nb / (out["split"] * 1e-6) / 1e9, 1), "timed_launches": K}


def decode_model_leg(args, dev, dist, peak):
    """Whole-model recurrent decoding: 48 MambaByte blocks (d_model 2304,
    d_inner 4608) at batch 256, one generated byte per stream per step, replayed
    from one CUDA graph. Bytes per step = every weight once + SSM states and
    convolution windows read and written."""
    import torch

    from paper_2401_13660_gb300.decoder import CONFIGS, Decoder

    name = "mambabyte_48x2304"
    dec = Decoder(CONFIGS[name], batch=STEP["batch"], device=dev, seed=1)
    dec.capture()
    g = torch.Generator(device=dev).manual_seed(8)
    tok = torch.randint(0, 256, (STEP["batch"],), device=dev, generator=g)
    for _ in range(3):
        dec.step(tok)
    torch.cuda.synchronize(dev)
    K = max(5, min(args.steps, 30))
    st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    st.record()
    for _ in range(K):
        dec.step(tok)
    en.record()
    en.synchronize()
    ms = reduce_max(st.elapsed_time(en) / K, dist, dev)
    dec.check()
    nb = dec.bytes_per_step()
    gbs = nb / (ms * 1e-3) / 1e9
    del dec
    torch.cuda.empty_cache()
    return {"model": name, "layers": 48, "d_model": 2304, "d_inner": 4608, "batch": STEP["batch"],
            "ms_per_step": round(ms, 4), "generated_bytes_per_s": round(STEP["batch"] / (ms * 1e-3), 1),
            "bytes_per_step": nb, "GB/s": round(gbs, 1), "frac_of_peak": round(gbs / peak, 4),
            "note": "per layer: mb_rmsnorm, one batched input GEMM (x and z), mb_conv_xproj (convolution "
                    "step fused with the [dt_low | B | C] projection, split over K), the Delta GEMM, mb_step "
                    "(B and C read in place), the output GEMM (GEMMs: cuBLAS bf16); one CUDA graph per step; "
                    "random seeded weights"}


def e2e_leg(args, mb, P, V, S, stream, dev, total_bytes, world, dist):
    """Same step through the public API with every step's inputs copied from
    pinned host memory and its outputs read back, inside the timed region.

    Three streams overlap the transfers with the kernels: step k's inputs are
    copied (host->device stream) into one of two device input sets while step
    k-1 computes on the other; each entry point starts as soon as its own
    inputs have landed, and its outputs go back (device->host stream) as soon
    as it finishes. The 48 decode layers' inputs and outputs are packed into
    one buffer per tensor kind (the layers use views of it), so a step makes a
    few large copies in each direction instead of hundreds of small ones. The
    recurrent states stay on the device (they are the model's cache), as in
    generation.
    """
    import torch

    def pin(t):
        return None if t is None else t.to("cpu").pin_memory()

    toks = ("x", "z", "dt", "B", "C")
    nl = len(S)
    skeys = [k for k in toks if S[0][k] is not None]
    host_P = {k: pin(P[k]) for k in toks}
    host_V = {k: pin(V[k]) for k in toks}
    host_S = {k: torch.stack([L[k] for L in S]).to("cpu").pin_memory() for k in skeys}
    host_acc = pin(V["accept"])
    # two device copies of every per-step input and output
    dev_sets = []
    for j in range(2):
        Pj, Vj = dict(P), dict(V)
        for d, src in ((Pj, P), (Vj, V)):
            for k in toks:
                if src[k] is not None and j == 1:
                    d[k] = torch.empty_like(src[k])
            if j == 1:
                d["y"] = torch.empty_like(src["y"])
        if j == 1:
            Pj["h_last"] = torch.empty_like(P["h_last"])
            Vj["accept"] = torch.empty_like(V["accept"])
        packed = {k: torch.stack([L[k] for L in S]) for k in skeys}      # fresh [nl, ...] buffers
        packed_y = torch.empty((nl,) + tuple(S[0]["y"].shape), dtype=S[0]["y"].dtype, device=dev)
        layers = [dict(L, **{k: packed[k][i] for k in skeys}, y=packed_y[i]) for i, L in enumerate(S)]
        dev_sets.append(dict(P=Pj, V=Vj, S=layers, packed=packed, packed_y=packed_y))
    outs_of = lambda st: [st["P"]["y"], st["P"]["h_last"], st["V"]["y"], st["packed_y"]]
    host_out = [torch.empty(o.shape, dtype=o.dtype, pin_memory=True) for o in outs_of(dev_sets[0])]
    h2d = sum(t.numel() * t.element_size() for h in (host_P, host_V, host_S) for t in h.values() if t is not None)
    h2d += host_acc.numel() * 4
    d2h = sum(o.numel() * o.element_size() for o in host_out)

    s_in, s_out = torch.cuda.Stream(dev), torch.cuda.Stream(dev)
    free = [torch.cuda.Event() for _ in range(2)]       # compute finished with set j
    out_free = [torch.cuda.Event() for _ in range(2)]   # set j's outputs copied back
    for e in free:
        e.record(stream)
    for e in out_free:
        e.record(s_out)

    def one(k):
        j = k % 2
        st = dev_sets[j]
        Pj, Vj, Sj = st["P"], st["V"], st["S"]
        landed = []
        s_in.wait_event(free[j])
        with torch.cuda.stream(s_in):
            for d, h in ((Pj, host_P), (Vj, host_V), (st["packed"], host_S)):
                for key, t in h.items():
                    if t is not None:
                        d[key].copy_(t, non_blocking=True)
                if d is Vj:
                    d["accept"].copy_(host_acc, non_blocking=True)
                ev = torch.cuda.Event()
                ev.record(s_in)
                landed.append(ev)
        done = []
        with torch.cuda.stream(stream):
            stream.wait_event(out_free[j])
            stream.wait_event(landed[0])
            mb.mb_scan_prefill(Pj["x"], Pj["dt"], Pj["B"], Pj["C"], Pj["A"], Pj["y"], z=Pj["z"],
                               D=Pj["D"], dt_bias=Pj["dt_bias"], h0=Pj["h0"], h_last=Pj["h_last"],
                               ws=P["ws"], stream=stream)
            ev = torch.cuda.Event(); ev.record(stream); done.append(ev)
            stream.wait_event(landed[1])
            mb.mb_scan_verify(Vj["x"], Vj["dt"], Vj["B"], Vj["C"], Vj["A"], Vj["y"], V["h_all"],
                              z=Vj["z"], D=Vj["D"], dt_bias=Vj["dt_bias"], h0=V["h0"], ws=V["ws"],
                              stream=stream)
            mb.mb_rollback(V["h0"], V["h_all"], Vj["accept"], V["h_keep"], ws=V["ws"], stream=stream)
            ev = torch.cuda.Event(); ev.record(stream); done.append(ev)
            stream.wait_event(landed[2])
            for Lj, L in zip(Sj, S):
                mb.mb_step(Lj["x"], Lj["dt"], Lj["B"], Lj["C"], L["A"], Lj["y"], L["state"], z=Lj["z"],
                           D=L["D"], dt_bias=L["dt_bias"], ws=L["ws"], stream=stream)
            ev = torch.cuda.Event(); ev.record(stream); done.append(ev)
            free[j].record(stream)
        with torch.cuda.stream(s_out):
            for o, ho, m in zip(outs_of(st), host_out, [0, 0, 1, 2]):   # output -> entry that writes it
                s_out.wait_event(done[m])
                ho.copy_(o, non_blocking=True)
            out_free[j].record(s_out)

    K = max(2, min(args.steps, 6))
    one(0)
    one(1)
    torch.cuda.synchronize(dev)
    if dist:
        dist.barrier()
    st, en = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    st.record(s_in)
    for k in range(K):
        one(k)
    s_in.wait_stream(s_out)
    s_in.wait_stream(stream)
    en.record(s_in)
    en.synchronize()
    ms = reduce_max(st.elapsed_time(en), dist, dev)
    return {"value": round(world * total_bytes * K / (ms * 1e-3) / 1e9, 1), "unit": "GB/s",
            "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h, "steps": K,
            "ms_per_step": round(ms / K, 4),
            "overlap": "double-buffered inputs; H2D, kernels and D2H on three streams; the decode "
                       "layers' inputs and outputs packed into one buffer per tensor kind"}


# ----------------------------------------------------------------------------- oracle
def oracle_sample(P, V, S, fraction, min_seconds=0.0, nthreads=None):
    """The oracle on a bounded sample of one step: the same fraction of the
    channels of every entry point (channels are independent), run repeatedly
    until at least min_seconds have been timed (once when 0), on `nthreads`
    threads (all host cores by default). Returns (seconds, algorithmic bytes
    of the samples, threads, description)."""
    import numpy as np
    import torch

    import oracle

    def np64(t):
        return None if t is None else t.detach().cpu().double().numpy()

    def sub(inp, nchan, rows):
        c = torch.arange(nchan, device=inp["x"].device)
        r = torch.arange(rows, device=inp["x"].device)
        tok = lambda t: None if t is None else np64(t.index_select(0, r)[:, :, c])
        h0 = inp.get("h0", inp.get("state"))
        return dict(x=tok(inp["x"]), z=tok(inp["z"]), dt=tok(inp["dt"]), B=np64(inp["B"].index_select(0, r)),
                    C=np64(inp["C"].index_select(0, r)), A=np64(inp["A"][c]), D=np64(inp["D"][c]),
                    dt_bias=np64(inp["dt_bias"][c]),
                    h0=None if h0 is None else np64(h0.index_select(0, r)[:, c]))

    nthreads = nthreads or os.cpu_count() or 1
    f = fraction
    pc = max(8, int(PREFILL["d_inner"] * PREFILL["batch"] * f))
    vc = max(8, int(VERIFY["d_inner"] * f))
    sc = max(8, int(STEP["d_inner"] * f))
    jobs = [("prefill", sub(P, min(pc, PREFILL["d_inner"]), 1), False),
            ("verify", sub(V, vc, VERIFY["batch"]), True)]
    layers = [sub(L, sc, STEP["batch"]) for L in S]
    secs, repeats = 0.0, 0
    while repeats == 0 or (secs < min_seconds and repeats < 200):
        t0 = time.perf_counter()
        for _, a, want_all in jobs:
            oracle.scan(a["x"], a["dt"], a["B"], a["C"], a["A"], z=a["z"], D=a["D"], dt_bias=a["dt_bias"],
                        h0=a["h0"], want_h_all=want_all, nthreads=nthreads)
        for a in layers:
            oracle.scan(a["x"], a["dt"], a["B"], a["C"], a["A"], z=a["z"], D=a["D"], dt_bias=a["dt_bias"],
                        h0=a["h0"], nthreads=nthreads)
        secs += time.perf_counter() - t0
        repeats += 1
    pch = min(pc, PREFILL["d_inner"])
    nbytes = repeats * (sum(bytes_prefill(**PREFILL)) * pch / (PREFILL["batch"] * PREFILL["d_inner"])
                        + sum(bytes_verify(**VERIFY)) * vc / VERIFY["d_inner"]
                        + STEP_LAYERS * sum(bytes_step(STEP["batch"], STEP["d_inner"])) * sc / STEP["d_inner"])
    desc = (f"fp64 C oracle, {nthreads} threads: prefill 1x8192x{pch} channels, verify "
            f"32x16x{vc}, decode step 256x{sc} x {STEP_LAYERS} layers (rollback omitted), "
            f"{repeats} repeat(s); bytes counted as the same fraction of each entry point's "
            f"algorithmic bytes")
    return secs, nbytes, nthreads, desc


def cpu_baseline(P, V, S, fraction, min_seconds=10.0):
    """The oracle on all host cores (repeated for at least min_seconds) and,
    once, on one core."""
    secs, nbytes, nthreads, desc = oracle_sample(P, V, S, fraction, min_seconds)
    secs1, nbytes1, _, _ = oracle_sample(P, V, S, fraction, 0.0, nthreads=1)
    return {"value": round(nbytes / secs / 1e9, 4), "unit": "GB/s", "cores": nthreads,
            "kind": "oracle", "sample": desc, "seconds": round(secs, 3),
            "single_core": {"value": round(nbytes1 / secs1 / 1e9, 4), "unit": "GB/s", "cores": 1,
                            "seconds": round(secs1, 3), "sample": "the same sample, once"}}


def rel_err(got, ref):
    """max_i |g_i - r_i| / max(|r_i|, rms(r)) (the parity metric of the tests)."""
    import numpy as np

    g = got.detach().cpu().double().numpy() if hasattr(got, "detach") else np.asarray(got, dtype=np.float64)
    r = np.asarray(ref, dtype=np.float64)
    rms = float(np.sqrt(np.mean(r * r))) or 1e-30
    return float(np.max(np.abs(g - r) / np.maximum(np.abs(r), rms)))


def oracle_parity(mb, P, V, S, snap, snap972, stream):
    """Part of the oracle leg: the timed launches' outputs against the fp64
    oracle on the same inputs. Prefills (both layers): the sampled channels
    over the whole span; verify: every stream, y and all 16 per-position
    states; rollback: bit-exact against the gather of the GPU's own h_all, and
    against the oracle; decode step: one more launch of layer 0 (same launch
    configuration, after the timed region) from a copy of its state, every
    channel. Bars: y 2e-2 (bf16 inputs), fp32 states 1e-3."""
    import numpy as np
    import torch

    import oracle

    np64 = lambda t: None if t is None else t.detach().cpu().double().numpy()
    tol = {"y": 2e-2, "state": 1e-3}
    out = {}

    def sampled(name, inp, sn):
        rows, chans = sn["rows"], sn["chans"]
        r_t, c_t = torch.tensor(rows), torch.tensor(chans)
        tok = lambda k: None if inp.get(k) is None else np64(inp[k].cpu().index_select(0, r_t)[:, :, c_t])
        h0 = inp.get("h0")
        ry, rh, _ = oracle.scan(tok("x"), tok("dt"), np64(inp["B"].cpu().index_select(0, r_t)),
                                np64(inp["C"].cpu().index_select(0, r_t)), np64(inp["A"].cpu()[c_t]),
                                z=tok("z"), D=np64(inp["D"].cpu()[c_t]), dt_bias=np64(inp["dt_bias"].cpu()[c_t]),
                                h0=None if h0 is None else np64(h0.cpu().index_select(0, r_t)[:, c_t]))
        out[name] = {"err_y": rel_err(sn["y"], ry), "err_h_last": rel_err(sn["h_last"], rh),
                     "sample": f"{len(rows)} batch rows x {len(chans)} channels x all {inp['x'].shape[1]} steps"}

    sampled("prefill", P, snap["prefill"])
    sampled("prefill_972m", snap972["inputs"], snap972)
    ry, _, rall = oracle.scan(np64(V["x"]), np64(V["dt"]), np64(V["B"]), np64(V["C"]), np64(V["A"]), z=np64(V["z"]),
                              D=np64(V["D"]), dt_bias=np64(V["dt_bias"]), h0=np64(V["h0"]), want_h_all=True)
    out["verify"] = {"err_y": rel_err(snap["verify_y"], ry), "err_h_all": rel_err(snap["verify_h_all"], rall),
                     "sample": "every stream, channel and drafted position"}
    acc = V["accept"].cpu().long()
    h_all = snap["verify_h_all"]
    gather = torch.where((acc == 0)[:, None, None], V["h0"].cpu(),
                         h_all[torch.arange(len(acc)), (acc - 1).clamp(min=0)])
    out["rollback"] = {"bit_exact_vs_gather": bool(torch.equal(snap["rollback"], gather)),
                       "err_vs_oracle": rel_err(snap["rollback"], oracle.rollback(np64(V["h0"]), rall,
                                                                                 acc.numpy().astype(np.int32)))}
    L = S[0]
    before = L["state"].clone()
    with torch.cuda.stream(stream):
        mb.mb_step(L["x"], L["dt"], L["B"], L["C"], L["A"], L["y"], L["state"], z=L["z"], D=L["D"],
                   dt_bias=L["dt_bias"], ws=L["ws"], stream=stream)
    stream.synchronize()
    sy, sh, _ = oracle.scan(np64(L["x"]), np64(L["dt"]), np64(L["B"]), np64(L["C"]), np64(L["A"]), z=np64(L["z"]),
                            D=np64(L["D"]), dt_bias=np64(L["dt_bias"]), h0=np64(before))
    out["step"] = {"err_y": rel_err(L["y"], sy), "err_state": rel_err(L["state"], sh),
                   "sample": "layer 0, every batch row and channel, one extra launch after the timed region"}
    errs_y = [out[k]["err_y"] for k in ("prefill", "prefill_972m", "verify", "step")]
    errs_s = [out["prefill"]["err_h_last"], out["prefill_972m"]["err_h_last"], out["verify"]["err_h_all"],
              out["step"]["err_state"], out["rollback"]["err_vs_oracle"]]
    for v in out.values():
        for k in list(v):
            if k.startswith("err"):
                v[k] = float(f"{v[k]:.3e}")
    out["tolerance"] = tol
    out["pass"] = bool(max(errs_y) <= tol["y"] and max(errs_s) <= tol["state"] and out["rollback"]["bit_exact_vs_gather"])
    return out


def reference_arm(args, rank, world, dist):
    """The oracle as it stands on the host cores, on a bounded sample of the
    same workload per step (inputs drawn on the CPU with the same generator)."""
    import torch

    dev = torch.device("cpu")
    P, V, S = build_gpu_state(dev)
    for _ in range(args.warmup):
        oracle_sample(P, V, S, args.ref_fraction)
    secs, nb, nthreads, desc = 0.0, 0.0, 1, ""
    for _ in range(args.steps):
        s, b, nthreads, desc = oracle_sample(P, V, S, args.ref_fraction)
        secs += s
        nb += b
    v = nb / secs / 1e9
    return {"impl": "reference", "metric": METRIC, "value": round(v, 4), "unit": "GB/s",
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(1e3 * secs / args.steps, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD_NAME, "sample_fraction": args.ref_fraction},
            "cpu_baseline": {"value": round(v, 4), "unit": "GB/s", "cores": nthreads,
                             "kind": "oracle", "sample": desc},
            "e2e": {"value": round(v, 4), "unit": "GB/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


def main():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["mine", "reference"], default="mine")
    ap.add_argument("--eager", action="store_true",
                    help="launch through the binding every step instead of replaying CUDA graphs")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-training", action="store_true", help="skip the forward+backward training leg")
    ap.add_argument("--no-fused-delta", action="store_true",
                    help="skip the fused-vs-unfused Delta projection prefill leg")
    ap.add_argument("--no-prompt-prefill", action="store_true",
                    help="skip the batch-1 prompt prefill leg (time split vs unsplit)")
    ap.add_argument("--no-decode-model", action="store_true", help="skip the 48-layer model decode leg")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-fraction", type=float, default=1 / 8,
                    help="fraction of one step's channels the oracle baseline processes")
    ap.add_argument("--ref-fraction", type=float, default=1 / 32,
                    help="per-step sample fraction for --impl reference")
    args = ap.parse_args()
    if args.warmup < 3:
        print("warning: fewer than 3 warm-up steps", file=sys.stderr)

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    dist = None
    if world > 1:
        import torch
        import torch.distributed as tdist
        backend = "nccl" if (args.impl == "mine" and torch.cuda.is_available()) else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", 0)))
        tdist.init_process_group(backend=backend)
        dist = tdist

    if args.impl == "reference":
        if rank == 0:
            line = reference_arm(args, rank, world, None)
            print(json.dumps(line), flush=True)
    else:
        line = gpu_arm(args, rank, world, dist)
        if rank == 0:
            print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
