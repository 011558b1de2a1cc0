"""Benchmark of the NAV verify pass: verified tokens/s and verify-pass latency, 7B shape, k=8.

One step = one speculative round through the public C ABI: pipesd_verify (target forward over the
pending token + k drafts against the cached prefix, accept/correct rule) + pipesd_ctx_sync (the two
result ints come back to the host) + pipesd_kv_rollback.  The cache grows by n_accepted+1 per step.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--workload 7b-k8]

Workload "ragged-7b" is the multi-edge case: 32 requests with seeded prefix lengths ~U[256,4096], draft lengths
~U{1..16} and noise sigma ~U[0.3,2]; one step = ONE batched verify + sync + one rollback call for all requests.

Prints ONE JSON line (rank 0).  Multi-GPU runs are independent replicas (no collective on the path).
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import tempfile
import time
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parent
if str(ROOT) not in sys.path:
    sys.path.insert(0, str(ROOT))

from paper_2605_13319_b200 import synth  # noqa: E402

WORKLOADS = {
    # name: (shape, prefix, k, sigma)
    "7b-k8": ("7b", 2048, 8, 1.0),
    "7b-k4": ("7b", 2048, 4, 1.0),
    "7b-k16": ("7b", 2048, 16, 1.0),
    "1b-k8": ("1b", 512, 8, 1.0),
    "8b-k16": ("8b", 8192, 16, 0.5),
    "tiny-k4": ("tiny", 64, 4, 1.0),
    "7b2l-k8": ("7b2l", 2048, 8, 1.0),   # two layers of the 7b shape: small enough for counter captures
    "ragged-7b": ("7b", None, None, None),      # 32 requests, lengths / k / sigma from synth.ragged_requests(0, 32)
    "ragged-7b2l": ("7b2l", None, None, None),  # the same batch on two layers (counter captures)
}
N_RAGGED = 32
METRIC = "verified tokens/sec (verify-pass latency in ms_per_step), k=8, 7B shape, % of HBM roofline"
NOMINAL_HBM_GBS = 8000.0


def peaks():
    p = ROOT / "MEASURED_PEAKS.json"
    if p.exists():
        return float(json.loads(p.read_text())["hbm_gbs"]), "measured"
    return 6650.0, "fallback"


def tensor_peak():
    """Sustained dense bf16 TFLOP/s (the projections of a large pass run inside a long step)."""
    p = ROOT / "MEASURED_PEAKS.json"
    if p.exists():
        return float(json.loads(p.read_text())["bf16_tflops_sustained"]), "measured"
    return 1400.0, "fallback"


def pass_flops(shape, ks):
    """Tensor-core flops of the projections of one pass as the kernels run them: every activation is a bf16 hi term and
    a bf16 lo term, so each weight element meets two products per row (2 x 2 flops)."""
    M = int(np.atleast_1d(ks).sum() + np.atleast_1d(ks).size)
    d, F, V = shape.d_model, shape.d_ffn, shape.vocab
    per_layer = (shape.q_dim + 2 * shape.kv_dim) * d + d * shape.q_dim + 3 * F * d
    return 4.0 * M * (shape.n_layers * per_layer + V * d)


def pass_bytes(shape, ks, cached_lens):
    """Algorithmic bytes of one verify pass over the requests (k_i drafts against cached_len_i positions): every
    weight once (bf16), embedding rows of the tokens, K/V of each cached prefix read and of the k_i+1 new rows
    written, logits written + read once, q read."""
    ks, cached_lens = np.atleast_1d(ks), np.atleast_1d(cached_lens)
    M = int(ks.sum() + ks.size)
    d, F, V = shape.d_model, shape.d_ffn, shape.vocab
    per_layer = (shape.q_dim + 2 * shape.kv_dim) * d + d * shape.q_dim + 3 * F * d
    weights = 2 * (shape.n_layers * per_layer + V * d) + 4 * d * (2 * shape.n_layers + 1) + 2 * M * d
    kv_tok = 2 * shape.n_layers * shape.kv_dim * 2
    kv = kv_tok * int(cached_lens.sum() + M)
    vocab_io = 4 * M * V * 2 + 4 * int(ks.sum()) * V
    return weights + kv + vocab_io


class ClockSampler:
    """nvidia-smi samples of the SM clock and throttle reasons while the timed regions run."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.uuid = uuid
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.p = None

    def start(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", self.uuid, f"--query-gpu={self.FIELDS}",
                                       "--format=csv,noheader,nounits", "-lms", "50"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is not None:
            self.p.terminate()
            try:
                self.p.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()
        self.f.flush()
        self.f.seek(0)
        sm, mx, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for line in self.f.read().splitlines():
            c = [x.strip() for x in line.split(",")]
            if len(c) < 8:
                continue
            try:
                sm.append(float(c[0])); mx.append(float(c[1]))
            except ValueError:
                continue
            for n, v in zip(names, c[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        self.f.close()
        os.unlink(self.f.name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(mx)), "reasons": sorted(reasons),
                "samples": len(sm)}


def draw_from(q_row, u):
    cdf = np.cumsum(q_row.astype(np.float64))
    return min(int(np.searchsorted(cdf, float(u) * cdf[-1], side="right")), q_row.size - 1)


def softmax64(x):
    x = x.astype(np.float64)
    e = np.exp(x - x.max())
    return e / e.sum()


def record_rounds(ctx, reqs, shape, ks, sigmas, seed, n_rounds, torch):
    """Untimed: produce every round's inputs by running the target one token at a time through the
    library (q_i = softmax(target logits + sigma*noise), draft ~ q_i), then verify + rollback so that
    the next round starts from the committed state.  One entry per request in reqs / ks / sigmas; every
    round is ONE batched verify.  Returns the per-round inputs and outcomes."""
    V = shape.vocab
    rounds = []
    pending = [synth.make_pending(shape, seed, i) for i in range(len(reqs))]
    for r in range(n_rounds):
        items, bases = [], []
        for i, req in enumerate(reqs):
            k = int(ks[i])
            base = ctx.req_len(req)
            noise = synth.normal_f32((k, V), seed, synth.STREAM_NOISE + 100 * i + 7919 * r)
            du = synth.uniform_f32(k, seed, synth.STREAM_DRAFT_U + 100 * i + 7919 * r)
            toks = [int(pending[i])]
            q = np.empty((k, V), np.float32)
            for j in range(k):
                l = ctx.prefill(req, [toks[-1]], want_last_logits=True)
                q[j] = softmax64(l.astype(np.float64) + float(sigmas[i]) * noise[j]).astype(np.float32)
                toks.append(draw_from(q[j], du[j]))
            ctx.debug_set_len(req, base)
            items.append(dict(req=req, tokens=np.array(toks, np.int32), q_dev=torch.from_numpy(q).to(ctx.device),
                              q_pin=torch.from_numpy(q).pin_memory(), u=synth.make_accept_uniforms(k, seed, i, r)))
            bases.append(base)
        got = ctx.verify([dict(req=it["req"], tokens=it["tokens"], q=it["q_dev"], u=it["u"]) for it in items])
        ctx.kv_rollback(reqs, [g[0] for g in got])
        rounds.append(dict(items=items, got=got, bases=bases))
        pending = [g[1] for g in got]
    return rounds


def replay(ctx, reqs, rounds, host_q, torch, timed=True):
    """Run recorded rounds back to back, bracketed by CUDA events on the context's stream when timed.
    Returns (elapsed_ms, verified tokens, results that differ from the recording)."""
    from paper_2605_13319_b200 import binding
    st = ctx.stream
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    tokens = mism = 0
    torch.cuda.synchronize()
    e0.record(st)
    for rd in rounds:
        if host_q:
            got = ctx.verify([dict(req=it["req"], tokens=it["tokens"], q=it["q_pin"].numpy(), u=it["u"])
                              for it in rd["items"]], flags=binding.Q_HOST)
        else:
            got = ctx.verify([dict(req=it["req"], tokens=it["tokens"], q=it["q_dev"], u=it["u"]) for it in rd["items"]])
        ctx.kv_rollback(reqs, [g[0] for g in rd["got"]])   # the recorded decision keeps the trajectory fixed
        mism += sum(g != h for g, h in zip(got, rd["got"]))
        tokens += sum(g[0] + 1 for g in rd["got"])
    e1.record(st)
    torch.cuda.synchronize()
    return (e0.elapsed_time(e1) if timed else 0.0), tokens, mism


def set_oracle_threads(n):
    """Threads of the CPU checker's OpenMP loops (it is built with gcc: libgomp)."""
    import ctypes
    try:
        ctypes.CDLL("libgomp.so.1").omp_set_num_threads(int(n))
        return True
    except OSError:
        return False


def workload_spec(name):
    """(shape, prefix lengths, draft lengths, noise sigmas): one entry per request."""
    sname, P, k, sigma = WORKLOADS[name]
    shape = synth.B7.scaled(name="7b2l", n_layers=2) if sname == "7b2l" else synth.SHAPES[sname]
    if P is None:
        lens, ks, sig = synth.ragged_requests(0, N_RAGGED)
        return shape, [int(x) for x in lens], [int(x) for x in ks], [float(x) for x in sig]
    return shape, [P], [k], [sigma]


def oracle_prepare(shape, weights, lens, ks, sigmas, seed, n_layers=None, requests=None):
    """Untimed set-up of the CPU checker for one round of the workload, request by request (they are independent):
    synthetic seeded K/V prefix (a CPU prefill is out of reach) and the checker's own drafts.
    `requests`: indices of the sample (default all)."""
    import oracle
    if n_layers is not None and n_layers < shape.n_layers:
        shape = shape.scaled(n_layers=n_layers)
        weights = dict(weights, layers=weights["layers"][:n_layers])
    std = 0.02 * np.sqrt(shape.d_model)
    V = shape.vocab
    cases = []
    for i in (range(len(lens)) if requests is None else requests):
        P, k = lens[i], ks[i]
        orc = oracle.Oracle(shape, weights, P + k + 8)
        for l in range(shape.n_layers):
            kk, vv = synth.make_synthetic_kv(shape, P, seed, l, request=i, std_k=std, std_v=std)
            orc.set_synthetic_kv(l, kk, vv)
        orc.set_len(P)
        toks, q, _ = orc.draft_round(synth.make_pending(shape, seed, i), k, sigmas[i],
                                     synth.normal_f32((k, V), seed, synth.STREAM_NOISE + 100 * i),
                                     synth.uniform_f32(k, seed, synth.STREAM_DRAFT_U + 100 * i))
        cases.append((orc, P, toks, q, synth.make_accept_uniforms(k, seed, i)))
    return cases


def oracle_time(cases):
    """The checker's verify call, as it stands, over the prepared requests.  Returns (seconds, verified tokens)."""
    total, tokens = 0.0, 0
    for orc, P, toks, q, u in cases:
        t0 = time.perf_counter()
        r = orc.verify(toks, q, u)
        total += time.perf_counter() - t0
        tokens += r["n_accepted"] + 1
        orc.truncate(P)
    return total, tokens


def run_reference(args, shape, lens, ks, sigmas):
    """--impl reference: the CPU checker timed on the host cores, each step a bounded sample."""
    cores = os.cpu_count() or 1
    steps, warm = args.steps, args.warmup
    budget = 150.0
    # sample: the first requests of the batch (all of a single-request workload), on as many leading layers as fit
    n_req = min(len(lens), 4)
    sample_reqs = list(range(n_req))
    w1 = synth.make_weights(shape.scaled(n_layers=1), 0)
    t1, _ = oracle_time(oracle_prepare(shape.scaled(n_layers=1), w1, lens, ks, sigmas, 0, requests=sample_reqs))
    est_full = t1 * shape.n_layers
    nl = int(max(1, min(shape.n_layers, budget / max(1e-9, (steps + warm) * est_full) * shape.n_layers)))
    sh = shape.scaled(n_layers=nl)
    cases = oracle_prepare(sh, synth.make_weights(sh, 0), lens, ks, sigmas, 0, requests=sample_reqs)
    total, tokens = 0.0, 0
    for s in range(steps + warm):
        dt, tk = oracle_time(cases)
        if s >= warm:
            total += dt
            tokens += tk
    scale = shape.n_layers / nl
    ms = total / steps * scale * 1e3 * (len(lens) / n_req)
    value = tokens / (total * scale)
    sample = (f"oracle verify pass of requests 0..{n_req - 1} of {len(lens)} on {nl} of {shape.n_layers} layers + LM "
              f"head per step (time scaled by {scale:.2f}; ms_per_step scaled to all requests), synthetic seeded K/V "
              f"prefixes, one fixed round of drafts")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "tokens/s", "n_gpus": args.gpus,
            "steps": steps, "warmup": warm, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(args.workload, shape, lens, ks, sigmas),
            "cpu_baseline": {"value": value, "unit": "tokens/s", "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def workload_config(name, shape, lens, ks, sigmas):
    if len(lens) == 1:
        return {"workload": name, "shape": shape.name, "prefix": lens[0], "k": ks[0], "sigma": sigmas[0]}
    return {"workload": name, "shape": shape.name, "requests": len(lens), "prefix": f"U[256,4096] (sum {sum(lens)})",
            "k": f"U{{1..16}} (sum {sum(ks)})", "sigma": "U[0.3,2.0]", "rows_per_pass": sum(ks) + len(ks)}


def kernel_source_hash():
    """Hash of the kernels' source: the stored DRAM-traffic figure is only reported while it matches."""
    import hashlib
    h = hashlib.sha256()
    for f in sorted((ROOT / "paper_2605_13319_b200" / "csrc").glob("*.cu*")):
        h.update(f.read_bytes())
    return h.hexdigest()[:16]


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=64)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="7b-k8", choices=sorted(WORKLOADS))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--quick-inputs", action="store_true",
                    help="profiler runs: seeded synthetic K/V prefix and random drafts instead of a recorded "
                         "trajectory, one timed region only, so that few launches precede the captured ones")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    shape, lens, ks, sigmas = workload_spec(args.workload)
    n_req = len(lens)
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))

    if args.impl == "reference":
        if rank == 0:
            run_reference(args, shape, lens, ks, sigmas)
        return

    import torch
    import torch.distributed as dist
    from paper_2605_13319_b200 import binding, build
    build.build_cuda()
    if world > 1:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    seed = 0
    n_rounds = args.warmup + args.steps
    grow = n_rounds * (max(ks) + 1) + 64
    max_seq = max(lens) + grow
    n_pages = sum((P + grow) // 16 + 2 for P in lens) + 4
    max_rows = max(32, sum(ks) + n_req)
    weights = synth.make_weights(shape, seed)
    mk = dict(n_pages=n_pages, max_seq=max_seq, max_draft=max(max(ks), 16), max_requests=n_req, max_rows=max_rows,
              device=local)
    ctx = binding.Context(shape, weights, **mk)
    prefixes = [synth.make_prefix(shape, P, seed + rank, request=i) for i, P in enumerate(lens)]
    if args.quick_inputs:
        quick_run(args, ctx, shape, lens, ks, seed, torch)
        return

    def fresh():
        reqs = []
        for pf in prefixes:
            reqs.append(ctx.req_open())
            ctx.prefill(reqs[-1], pf)
        return reqs

    def close(reqs):
        for r in reqs:
            ctx.req_close(r)

    reqs = fresh()
    rounds = record_rounds(ctx, reqs, shape, ks, sigmas, seed, n_rounds, torch)
    close(reqs)

    uuid = "GPU-" + str(torch.cuda.get_device_properties(local).uuid)
    sampler = ClockSampler(uuid)

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()

    # -- timed region 1: inputs resident in HBM
    reqs = fresh()
    ctx.profile_enable(False)
    barrier()
    sampler.start()
    replay(ctx, reqs, rounds[:args.warmup], False, torch, timed=False)  # warm-up
    ctx.profile_read()
    ms, tokens, mism = replay(ctx, reqs, rounds[args.warmup:], False, torch)
    prof = ctx.profile_read()
    barrier()
    close(reqs)
    # -- timed region 2: host buffers (q copied H2D inside, results D2H)
    reqs = fresh()
    replay(ctx, reqs, rounds[:args.warmup], True, torch, timed=False)
    barrier()
    ms_e2e, tokens_e2e, mism2 = replay(ctx, reqs, rounds[args.warmup:], True, torch)
    barrier()
    close(reqs)
    # -- region 3: the same steps with every GEMM launch bracketed by CUDA events (a kernel per projection then, also where the
    # timed pass is one kernel)
    reqs = fresh()
    replay(ctx, reqs, rounds[:args.warmup], False, torch, timed=False)
    ctx.profile_enable(True)
    ms_prof, _, _ = replay(ctx, reqs, rounds[args.warmup:], False, torch)
    gprof = ctx.profile_read()
    ctx.profile_enable(False)
    close(reqs)
    clocks = sampler.stop()

    # -- reduce over ranks: max time, summed tokens
    if world > 1:
        from paper_2605_13319_b200 import replicas
        (ms, ms_e2e), (tokens, tokens_e2e) = replicas.reduce_replicas([ms, ms_e2e], [tokens, tokens_e2e], device="cuda")
    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    steps = args.steps
    ms_step = ms / steps
    bytes_pass = float(np.mean([pass_bytes(shape, ks, rd["bases"]) for rd in rounds[args.warmup:]]))
    peak, peak_kind = peaks()
    pass_gbs = bytes_pass / (ms_step * 1e-3) / 1e9
    dense = sum(ks) + n_req > 32
    # a pass of the layer-stack kernel is three launches: the stack, the row statistics, the acceptance
    stacked = prof["kernel_launches"] <= 3 * steps
    projections = "gemm_dense_kernel" if dense else "gemm_wstream_kernel"
    gemm_gbs = gprof["gemm_bytes"] / (gprof["gemm_ms"] * 1e-3) / 1e9 if gprof["gemm_ms"] > 0 else 0.0
    cfg = workload_config(args.workload, shape, lens, ks, sigmas)
    cfg.update({"rounds": steps, "l2": "inputs larger than L2 (weights streamed once per pass)",
                "accepted_per_step": tokens / world / steps - n_req, "replay_mismatches": int(mism + mism2)})
    traffic = TRAFFIC.get(args.workload)
    if traffic is not None and TRAFFIC["kernel_source_hash"] != kernel_source_hash():
        traffic = None       # the kernels have changed since the counters were taken
    line = {
        "metric": METRIC, "value": tokens / (ms * 1e-3), "unit": "tokens/s", "n_gpus": world, "steps": steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "arithmetic": "bf16 weights x split-bf16 (hi + lo) activations on the tensor cores, fp32 accumulate; K/V bf16",
        "data": "synthetic",
        "config": cfg,
        "pass": {"bytes": bytes_pass, "gbs": pass_gbs, "frac_of_nominal_8TBs": pass_gbs / NOMINAL_HBM_GBS,
                 "frac_of_measured_copy": pass_gbs / peak},
        "e2e": {"value": tokens_e2e / (ms_e2e * 1e-3), "unit": "tokens/s", "ms_per_step": ms_e2e / steps,
                "h2d_bytes_per_step": int(4 * sum(ks) * shape.vocab + 4 * (sum(ks) + n_req) * 2),
                "d2h_bytes_per_step": 16 * n_req},
        "gpu_launches": int(prof["kernel_launches"]),
        # The roofline of the timed region itself: algorithmic bytes of the pass / ms_per_step.  A pass of up to 32 rows is
        # one kernel (embedding to logits) and two small ones behind it, a larger one a chain of kernels that overlap by
        # programmatic dependent launch: either way only the whole pass fits inside ms_per_step.
        "roofline": {"bound": "hbm",
                     "kernel": "verify pass (one layer_stack_kernel, then row_stats_kernel and accept_sample_kernel)" if stacked else
                               f"verify pass (chain of {projections} and attn_kernel launches)",
                     "achieved": pass_gbs, "peak": peak, "peak_kind": peak_kind, "unit": "GB/s", "frac": pass_gbs / peak,
                     "algorithmic_bytes_per_step": bytes_pass, "traffic": traffic,
                     # GEMM launches alone, each between two CUDA events, in a separate replay: an event between two launches
                     # undoes their overlap, so these times are the kernels WITHOUT dependent-launch overlap and do not fit
                     # inside ms_per_step.  Where the timed pass is one kernel, they are other kernels than the timed ones
                     "gemm_launches_isolated": {"kernel": projections, "in_timed_pass": not stacked,
                                                "achieved": gemm_gbs, "frac": gemm_gbs / peak, "unit": "GB/s",
                                                "launches": int(gprof["gemm_launches"]),
                                                "algorithmic_bytes_per_launch": gprof["gemm_bytes"] / max(1, gprof["gemm_launches"]),
                                                "ms_per_step_with_events": ms_prof / steps,
                                                "share_of_that_replay": gprof["gemm_ms"] / ms_prof,
                                                "regime": "no dependent-launch overlap (events between launches)"}},
        "clocks": clocks,
    }
    if dense:
        # a pass of more than 32 rows runs its projections on the dense tensor-core kernel: those are bound by the
        # tensor cores, the attention by HBM, so neither roofline alone bounds the pass; both fractions are given
        tp, tp_kind = tensor_peak()
        tfl = pass_flops(shape, ks) / (ms_step * 1e-3) / 1e12
        line["roofline"]["projections_tensor"] = {"bound": "tensor", "achieved": tfl, "peak": tp, "peak_kind": tp_kind,
                                                  "unit": "TFLOP/s", "frac": tfl / tp,
                                                  "note": "projection flops (hi and lo products) over the WHOLE pass time"}
    if world == 1 and not args.no_cpu_baseline:
        sample_reqs = list(range(min(n_req, 4)))
        dt, toks_o = oracle_time(oracle_prepare(shape, weights, lens, ks, sigmas, seed, requests=sample_reqs))
        cores = os.cpu_count()
        what = (f"one verify pass (all {shape.n_layers} layers) of " +
                (f"requests 0..{len(sample_reqs) - 1} of {n_req}" if n_req > 1 else f"the request (k={ks[0]})") +
                ", seeded synthetic K/V prefix, drafts made by the oracle itself")
        line["cpu_baseline"] = {"value": toks_o / dt, "unit": "tokens/s", "cores": cores, "kind": "oracle",
                                "ms_per_pass": dt * 1e3 * n_req / len(sample_reqs), "sample": what}
        # the same checker on one core, on a quarter of the layers (time scaled), first request only
        nl1 = max(1, shape.n_layers // 4)
        cases1 = oracle_prepare(shape, weights, lens, ks, sigmas, seed, n_layers=nl1, requests=[0])
        if set_oracle_threads(1):
            dt1, tk1 = oracle_time(cases1)
            set_oracle_threads(cores)
            dt1 *= shape.n_layers / nl1
            line["cpu_baseline"]["one_core"] = {"value": tk1 / dt1, "unit": "tokens/s", "cores": 1,
                                                "sample": f"request 0 on {nl1} of {shape.n_layers} layers + LM head, time scaled"}
    print(json.dumps(line), flush=True)
    ctx.close()
    if world > 1:
        dist.destroy_process_group()


def quick_run(args, ctx, shape, lens, ks, seed, torch):
    """Profiler-friendly variant: no prefill passes, no recording.  Kernel durations do not depend on the
    values, only on the shapes and lengths, which are those of the workload."""
    V = shape.vocab
    std = 0.02 * np.sqrt(shape.d_model)
    reqs = []
    for i, P in enumerate(lens):
        reqs.append(ctx.req_open())
        for l in range(shape.n_layers):
            kk, vv = synth.make_synthetic_kv(shape, P, seed, l, request=i, std_k=std, std_v=std)
            ctx.debug_write_kv(reqs[-1], l, 0, kk, vv)
    rounds = []
    for r in range(args.warmup + args.steps):
        items = []
        for i, req in enumerate(reqs):
            k = ks[i]
            noise = synth.normal_f32((k, V), seed, synth.STREAM_NOISE + 100 * i + 7919 * r)
            q = np.stack([softmax64(noise[j]) for j in range(k)]).astype(np.float32)
            toks = synth.tokens_i32(k + 1, seed, synth.STREAM_PENDING + 100 * i + r, V)
            items.append(dict(req=req, tokens=toks, q=torch.from_numpy(q).to(ctx.device),
                              u=synth.make_accept_uniforms(k, seed, i, r)))
        rounds.append(items)
    st = ctx.stream
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    tokens = 0
    for i, items in enumerate(rounds):
        if i == args.warmup:
            torch.cuda.synchronize()
            e0.record(st)
        got = ctx.verify(items)
        ctx.kv_rollback(reqs, [g[0] for g in got])
        tokens += sum(g[0] + 1 for g in got) if i >= args.warmup else 0
    e1.record(st)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    print(json.dumps({"mode": "quick-inputs", "workload": args.workload, "steps": args.steps, "warmup": args.warmup,
                      "ms_per_step": ms / args.steps, "tokens": tokens}), flush=True)
    ctx.close()


# dram__bytes_read.sum + dram__bytes_write.sum per step, of all launches of a pass, from the ncu capture summarised under profiles/ (of
# the full workload, caches kept between launches), with the hash of the kernel sources it was taken on: the figure is
# reported only while the sources still hash to that value.
TRAFFIC = {"kernel_source_hash": "0e94f9e562c16ca9", "7b-k8": 14303753728.0}


if __name__ == "__main__":
    main()
