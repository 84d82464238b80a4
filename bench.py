#!/usr/bin/env python
"""Benchmark of one auto-correct decoding step (attention + verify + KV commit).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--config NAME] [--impl ours|reference]

--config lmhead_* times space_lmhead_verify (output projection fused with greedy
verification, one kernel per step) on a projection workload instead.

One step = space_attn_step + space_verify_commit (verification and KV commit in
one call) for the whole batch of one synthetic input set.  Several distinct input sets are rotated so that no
step finds its inputs in L2.  Prints ONE JSON line (rank 0).

--impl ours       the CUDA library.  `value` is steps/s with inputs resident in
                  HBM, the K steps replayed from a CUDA graph.  `roofline` comes
                  from CUDA events recorded around every attention-kernel launch
                  in a second, stream-launched pass over the same steps; `e2e`
                  from space_step_host with pinned host buffers; `cpu_baseline`
                  from the CPU oracle on the host cores.
--impl reference  the CPU oracle alone on the host cores (rank 0 only).
With N > 1 (torchrun) every rank runs an independent replica on its own GPU.
"""
import argparse
import json
import os
import re
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2402_11809_b200 import replicas, workloads  # noqa: E402

L2_BYTES = 126 * 1024 * 1024
# dram__bytes_read.sum + dram__bytes_write.sum per launch of the dominant kernel, from the ncu captures
# summarised under profiles/: (bytes, kernel source file, first 12 hex digits of the sha256 of that file and
# the headers it includes when the capture was taken).  The figure is reported only while the sources still have
# that hash; once the kernel has changed the bench line carries null until the capture is taken again.  (A hash
# moves on without a capture only where what changed since is comments, host code or a build that the case does not run.)
ATTN_TRAFFIC = {"llama7b": (34524672, "attn_tc.cu", "9d3d3e891f87"),
                "gqa70b": (289018368, "attn_rows.cu", "88d7215e03b5")}
LMHEAD_TRAFFIC = {"lmhead_llama7b": (263353088, "lmhead.cu", "56d9407a9aef"),
                  "lmhead_vocab128k": (1087300608, "lmhead.cu", "56d9407a9aef")}
METRIC = "auto-correct steps/sec"
UNIT = "steps/s"


def source_hash(fname, root=ROOT):
    """First 12 hex digits of the sha256 of a kernel source and of every file that it includes by a quoted name,
    directly or through another."""
    import hashlib
    files, todo = [], [os.path.join(root, "paper_2402_11809_b200", "csrc", fname)]
    while todo:
        path = os.path.normpath(todo.pop(0))
        if path not in files:
            files.append(path)
            todo += [os.path.join(os.path.dirname(path), n) for n in re.findall(r'^#include "([^"]+)"', open(path).read(), re.M)]
    h = hashlib.sha256()
    for path in files:
        h.update(open(path, "rb").read())
    return h.hexdigest()[:12]


def measured_traffic(table, name):
    """DRAM bytes per launch from the committed ncu capture, or None when there is no capture of
    the kernel as it stands now."""
    ent = table.get(name)
    if ent is None:
        return None
    nbytes, fname, digest = ent
    return nbytes if source_hash(fname) == digest else None


def timed_region(run_steps, K, stream, barrier):
    """Time K steps with CUDA events on `stream`.  A region shorter than about 50 ms is repeated
    (every repeat is again exactly K steps between two events) and the median is returned, so that
    a short run gives the same per-step figure as a long one.  Returns (ms of K steps, repeats, all ms)."""
    import torch
    def once():
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        run_steps(K)
        e1.record(stream)
        stream.synchronize()
        return e0.elapsed_time(e1)
    first = once()
    reps = [first]
    if first < 50.0:
        n = int(min(200, max(4, np.ceil(50.0 / max(first, 1e-3)))))
        for _ in range(n):
            reps.append(once())
    return float(np.median(reps)), len(reps), reps


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return float(d["hbm_gbs"]), float(d.get("bf16_tflops", 1590.0)), "measured"
    return 6650.0, 1590.0, "fallback"


# ---------------------------------------------------------------- clock sampler
class ClockSampler:
    """Samples SM clock and throttle reasons of one GPU through NVML while running."""

    def __init__(self, index):
        self.samples, self.reasons, self.other, self.max_mhz = [], set(), set(), None
        self._stop = threading.Event()
        self._thread = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByIndex(index)
            self.max_mhz = pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM)
        except Exception:
            self.nv = None

    def _loop(self):
        nv = self.nv
        names = {
            nv.nvmlClocksThrottleReasonHwSlowdown: "hw_slowdown",
            nv.nvmlClocksThrottleReasonHwThermalSlowdown: "hw_thermal_slowdown",
            nv.nvmlClocksThrottleReasonSwThermalSlowdown: "sw_thermal_slowdown",
            nv.nvmlClocksThrottleReasonSwPowerCap: "sw_power_cap",
        }
        # further clock-event reasons, kept apart ("other_reasons"): a clock below the maximum then has a
        # name (a short timed region catches the clocks between idle and load)
        others = {}
        for attr, name in (("nvmlClocksThrottleReasonGpuIdle", "gpu_idle"),
                           ("nvmlClocksThrottleReasonApplicationsClocksSetting", "applications_clocks_setting"),
                           ("nvmlClocksThrottleReasonHwPowerBrakeSlowdown", "hw_power_brake_slowdown"),
                           ("nvmlClocksThrottleReasonSyncBoost", "sync_boost")):
            if hasattr(nv, attr):
                others[getattr(nv, attr)] = name
        while not self._stop.is_set():
            try:
                self.samples.append(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM))
                r = nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.h)
                for bit, name in names.items():
                    if r & bit:
                        self.reasons.add(name)
                for bit, name in others.items():
                    if r & bit:
                        self.other.add(name)
            except Exception:
                pass
            self._stop.wait(0.005)

    def start(self):
        if self.nv is not None:
            self._thread = threading.Thread(target=self._loop, daemon=True)
            self._thread.start()

    def stop(self):
        self._stop.set()
        if self._thread is not None:
            self._thread.join()
        med = float(np.median(self.samples)) if self.samples else None
        return {"sm_mhz": med, "sm_max_mhz": self.max_mhz, "reasons": sorted(self.reasons),
                "other_reasons": sorted(self.other), "samples": len(self.samples)}


# ------------------------------------------------------------------- CPU oracle
def oracle_step(cfg, x):
    """One whole step with the CPU oracle (attention, verify, commit)."""
    from oracle.attention import attention_step
    from oracle.verify import verify_step
    from oracle.commit import commit_step
    k = cfg["k"]
    attention_step(x["q"], x["k_cache"], x["v_cache"], x["kv_len"], k, x["scale"])
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, cfg["mode"],
                    temperature=cfg["temperature"], seed=cfg["seed"], seq_id=x["seq_id"],
                    kv_len=x["kv_len"])
    kc, vc = x["k_cache"].copy(), x["v_cache"].copy()
    commit_step(kc, vc, x["kv_len"], r["n_accept"], k)
    return r


def blas_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [p.get("num_threads", 1) for p in threadpool_info() if p.get("user_api") == "blas"]
        return max(n) if n else 1
    except Exception:
        return os.cpu_count() or 1


def time_oracle(cfg, x, budget_s, min_reps=3, max_reps=None):
    oracle_step(cfg, x)                                   # warm-up (imports, BLAS threads)
    t0 = time.perf_counter()
    reps = 0
    while True:
        oracle_step(cfg, x)
        reps += 1
        el = time.perf_counter() - t0
        if max_reps is not None and reps >= max_reps:
            break
        if max_reps is None and reps >= min_reps and el >= budget_s:
            break
    return reps / el, reps, el


def run_reference(args):
    rank, _, _ = replicas.rank_env()
    if rank != 0:                                         # rank 0 alone times the oracle
        return
    cfg = workloads.resolve(args.config)
    x = workloads.make_step_inputs(cfg)
    for _ in range(args.warmup if args.warmup < 3 else 2):
        oracle_step(cfg, x)
    # bounded: at most ~150 s of timed work; a "step" stays one whole step of the
    # workload and the number of timed repetitions is what is bounded
    t0 = time.perf_counter()
    oracle_step(cfg, x)
    one = time.perf_counter() - t0
    reps = max(1, min(args.steps, int(150.0 / max(one, 1e-6))))
    sps, reps, el = time_oracle(cfg, x, 0.0, max_reps=reps)
    cores = blas_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": sps, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 / sps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": cfg["name"], "timed_steps": reps,
                   "note": "CPU oracle (numpy fp64), whole steps; repetitions bounded to ~150 s"},
        "cpu_baseline": {"value": sps, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{reps} whole step(s) of {cfg['name']} in {el:.1f} s"},
        "e2e": {"value": sps, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------- CUDA arm
def run_ours(args):
    import torch
    from paper_2402_11809_b200 import device as H
    from paper_2402_11809_b200 import build
    build.build()
    from paper_2402_11809_b200 import binding as B

    rank, world, local = replicas.rank_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py --impl ours needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    replicas.init("nccl", local)

    over = {}
    if args.batch:
        over["B"] = args.batch
    if args.k:
        over["k"] = args.k
    cfg = workloads.resolve(args.config, **over)
    if args.batch:
        cfg["name"] = f"{args.config}@batch{args.batch}"   # a reduced copy of the workload (profiler captures)
    if args.k:
        cfg["name"] += f"@k{args.k}"                       # another number of mask tokens (Sec. 4.3: k = 2 beats k = 5 from batch 8)
    if args.top_k and cfg["mode"] == "sample":
        cfg["name"] += f"+top{args.top_k}p{args.top_p:g}"  # filtered target distributions (App. A.4: top-k 10, top-p 0.95)
    if args.paged:
        cfg["name"] += "+paged"                            # (no profiler capture of this form: traffic stays null)
    k, n_q = cfg["k"], workloads.n_block_rows(cfg["k"])
    sample = cfg["mode"] == "sample"
    mode = B.MODE_SAMPLE if sample else B.MODE_GREEDY

    # ---- input sets: enough distinct sets that their footprint is twice L2 ----
    x0 = workloads.make_step_inputs(cfg, set_index=replicas.set_index(rank, 0))
    ab = workloads.algorithmic_bytes(cfg, x0["kv_len"])
    n_sets = max(2, int(np.ceil(2.0 * L2_BYTES / ab["total"])))
    n_sets = min(n_sets, 16)
    sets = [x0] + [workloads.make_step_inputs(cfg, set_index=replicas.set_index(rank, i)) for i in range(1, n_sets)]

    # --paged: the same caches as page pools behind shuffled page tables (the host-buffer leg and the
    # oracle keep the contiguous form: space_step_host has no paged variant)
    dev_sets = [workloads.to_pages(x, seed=i, poison=False) for i, x in enumerate(sets)] if args.paged else sets
    s_cap = max(x["s_cap"] for x in dev_sets + sets)
    ctx = B.Context(device=local, max_batch=cfg["B"], n_q_heads=cfg["H_q"], n_kv_heads=cfg["H_kv"],
                    head_dim=cfg["d"], k_max=k, vocab=cfg["V"], host_staging=1, s_cap=s_cap)
    steps_dev = [H.DeviceStep(cfg, x) for x in dev_sets]
    arg_sets = []
    for ds in steps_dev:
        a = ctx.attn_args(ds.q, ds.k_cache, ds.v_cache, ds.kv_len, ds.out, k, ds.scale, status=ds.status,
                          impl=B.ATTN_TENSOR_ROWS if args.attn_impl == "rows" else B.ATTN_TENSOR,
                          page_table=ds.page_table)
        v = ctx.verify_args(ds.logits, ds.cand, ds.cand_prob, ds.kv_len, ds.n_accept, ds.out_tokens,
                            ds.n_out, ds.next_cand, ds.next_cand_prob, ds.finished, k, mode=mode,
                            temperature=cfg["temperature"], seed=cfg["seed"], seq_id=ds.seq_id,
                            status=ds.status, top_k=args.top_k if sample else 0, top_p=args.top_p)
        c = ctx.commit_args(ds.k_cache, ds.v_cache, ds.n_accept, ds.kv_len, k, kv_len_out=ds.kv_len_out,
                            status=ds.status, page_table=ds.page_table)
        arg_sets.append((a, v, c))

    def step(i):
        a, v, c = arg_sets[i % n_sets]
        ctx.space_attn_step(a)
        if args.separate_commit:
            ctx.space_verify(v)
            ctx.space_kv_commit(c)
        else:
            ctx.space_verify_commit(v, c)

    stream = torch.cuda.Stream()
    K, W = args.steps, max(args.warmup, 3)
    with torch.cuda.stream(stream):
        for i in range(n_sets):                           # first launches, descriptor set-up
            step(i)
        stream.synchronize()
        n0 = ctx.launch_count
        step(0)
        launches_per_step = ctx.launch_count - n0
        # one graph holding n_sets consecutive steps, one holding the remainder
        g_full = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g_full, stream=stream):
            for i in range(n_sets):
                step(i)
        rem = K % n_sets
        g_rem = None
        if rem:
            g_rem = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g_rem, stream=stream):
                for i in range(rem):
                    step(i)

        def run_steps(n):
            for _ in range(n // n_sets):
                g_full.replay()
            if n % n_sets:
                if n % n_sets == rem and g_rem is not None:
                    g_rem.replay()
                else:
                    for i in range(n % n_sets):
                        step(i)

        run_steps(W)
        stream.synchronize()
        sampler = ClockSampler(local)
        replicas.barrier()
        torch.cuda.synchronize()
        sampler.start()
        ms, n_repeats, _ = timed_region(run_steps, K, stream, replicas.barrier)
        torch.cuda.synchronize()
        replicas.barrier()
        # keep the sampler running through the kernel-timing pass as well
        # ---- second pass: per-kernel CUDA events, stream-launched ------------
        n_prof = min(max(K, 256), 2048)
        ctx.space_profile_enable(1)
        for i in range(n_prof):
            step(i)
        stream.synchronize()
        ctx.space_profile_enable(0)
        prof = ctx.space_profile_read()
        clocks = sampler.stop()
        status = sum(int(ds.status.abs().sum()) for ds in steps_dev)

    steps_per_s, sec = replicas.job_throughput(K, ms * 1e-3, device="cuda")
    ms = sec * 1e3

    # ---- end to end from pinned host buffers (space_step_host) ---------------
    import ctypes as C
    x = sets[0]
    pin = {}
    for name in ("q", "k_cache", "v_cache", "logits", "cand", "cand_prob", "kv_len"):
        arr = x[name]
        t = torch.from_numpy(arr.view(np.int16) if arr.dtype == np.uint16 else arr).clone().pin_memory()
        pin[name] = t
    kv_len0 = pin["kv_len"].clone()
    outs = dict(out=torch.empty((cfg["B"], n_q, cfg["H_q"], cfg["d"]), dtype=torch.float32).pin_memory(),
                n_accept=torch.empty(cfg["B"], dtype=torch.int32).pin_memory(),
                out_tokens=torch.empty((cfg["B"], k + 1), dtype=torch.int32).pin_memory(),
                n_out=torch.empty(cfg["B"], dtype=torch.int32).pin_memory(),
                next_cand=torch.empty((cfg["B"], k), dtype=torch.int32).pin_memory(),
                next_cand_prob=torch.empty((cfg["B"], k), dtype=torch.float32).pin_memory(),
                finished=torch.empty(cfg["B"], dtype=torch.uint8).pin_memory(),
                status=torch.empty(cfg["B"], dtype=torch.int32).pin_memory())
    h2d, d2h = C.c_int64(0), C.c_int64(0)
    hs = B.HostStepArgs(batch=cfg["B"], k=k, vocab=cfg["V"],
                        logits_dtype=B.DTYPE_F32 if cfg["logits_dtype"] == "f32" else B.DTYPE_BF16,
                        mode=mode, resample=B.RESAMPLE_RESIDUAL_POINTMASS, eos_id=-1,
                        mask_variant=B.MASK_SAME_GROUP, scale=x["scale"], temperature=cfg["temperature"],
                        seed=cfg["seed"],
                        **{n_: C.c_void_p(t.data_ptr()) for n_, t in pin.items()},
                        **{n_: C.c_void_p(t.data_ptr()) for n_, t in outs.items()},
                        h2d_bytes=C.cast(C.pointer(h2d), C.c_void_p), d2h_bytes=C.cast(C.pointer(d2h), C.c_void_p))
    n_e2e = max(3, min(K, 100))
    with torch.cuda.stream(stream):
        for _ in range(3):
            pin["kv_len"].copy_(kv_len0)
            ctx.space_step_host(hs)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            pin["kv_len"].copy_(kv_len0)
            ctx.space_step_host(hs)
        torch.cuda.synchronize()
        e2e_s = time.perf_counter() - t0
    e2e_val, _ = replicas.job_throughput(n_e2e, e2e_s, device="cuda")
    e2e_ok = bool((outs["status"] == 0).all()) and \
        bool(torch.equal(outs["n_accept"], steps_dev[0].n_accept.cpu()))
    if args.top_k and sample:
        e2e_ok = None          # space_step_host verifies against the unfiltered distributions: nothing to compare
    h2d_full, d2h_full = int(h2d.value), int(d2h.value)

    # The same call as a decoder would make it: the KV cache is state that stays on the device
    # between steps, so a step uploads only the block's own K/V rows (plus q, logits, candidates).
    hs.cache_resident = 1
    n_res = max(3, min(K, 400))
    with torch.cuda.stream(stream):
        for _ in range(3):
            pin["kv_len"].copy_(kv_len0)
            ctx.space_step_host(hs)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(n_res):
            pin["kv_len"].copy_(kv_len0)
            ctx.space_step_host(hs)
        torch.cuda.synchronize()
        res_s = time.perf_counter() - t0
    res_val, _ = replicas.job_throughput(n_res, res_s, device="cuda")
    res_ok = bool((outs["status"] == 0).all()) and \
        bool(torch.equal(outs["n_accept"], steps_dev[0].n_accept.cpu()))
    if args.top_k and sample:
        res_ok = None
    # The call's own count names all rows of logits; from pinned buffers verification reads only what it needs over
    # PCIe: 2k+1 rows, one of them twice in sampling, or all of them in its single launch where the rows it could
    # skip come to 512 KB at most (csrc/verify.cu: launch_verify).
    row_bytes = x["logits"].dtype.itemsize * cfg["V"]
    single = not sample and cfg["B"] * (n_q - 2 * k - 1) * row_bytes <= 512 << 10
    rows_read = n_q if single else 2 * k + (2 if sample else 1)
    h2d_res = int(h2d.value) - cfg["B"] * (n_q - rows_read) * row_bytes

    if rank != 0:
        replicas.shutdown()
        return

    # ---- roofline of the dominant kernel (attention) --------------------------
    peak, peak_tf, peak_src = load_peaks()
    attn_ms, attn_n = prof["attn"]
    attn_bytes = np.mean([workloads.algorithmic_bytes(cfg, s["kv_len"])["kv"] +
                          workloads.algorithmic_bytes(cfg, s["kv_len"])["q_out"] for s in sets])
    attn_us = 1e3 * attn_ms / max(attn_n, 1)
    achieved = attn_bytes / (attn_us * 1e-6) / 1e9 if attn_n else None
    step_bytes = float(np.mean([workloads.algorithmic_bytes(cfg, s["kv_len"],
                                                            steps_dev[i].n_accept.cpu().numpy())["total"]
                                for i, s in enumerate(sets)]))
    per_kernel_us = {name: (1e3 * v[0] / v[1] if v[1] else None) for name, v in prof.items()}
    # Which roof binds the attention launch: the method's two products (Q K^T and P V, 2 flop per
    # multiply-add each: 4 M (L + n_q) d per kv head) against the K, V, Q and output bytes.  The second
    # product the kernels take for the low half of P is an implementation cost and is not counted.
    rows = n_q * (cfg["H_q"] // cfg["H_kv"])
    attn_flops = float(np.mean([sum(4.0 * rows * cfg["d"] * (int(L) + n_q) * cfg["H_kv"] for L in s_["kv_len"])
                                for s_ in sets]))
    tensor_bound = attn_flops / (peak_tf * 1e12) > attn_bytes / (peak * 1e9)
    if tensor_bound and attn_n:
        roof = {"bound": "tensor", "achieved": attn_flops / (attn_us * 1e-6) / 1e12, "peak": peak_tf,
                "unit": "TFLOP/s", "algorithmic_flops_per_launch": attn_flops,
                "peak_source": peak_src + " (burst bf16 GEMM figure)"}
    else:
        roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                "peak_source": peak_src + " (burst copy figure)"}
    roof["frac"] = (roof["achieved"] / roof["peak"]) if roof["achieved"] else None

    # ---- CPU oracle on the host cores (bounded: about 10 s) -------------------
    cpu_sps, cpu_reps, cpu_el = time_oracle(cfg, sets[0], budget_s=10.0)

    line = {
        "metric": METRIC, "value": steps_per_s, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": W,
        "ms_per_step": ms / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16", "data": "synthetic",
        "config": {"workload": cfg["name"], "batch": cfg["B"], "k": k, "heads": [cfg["H_q"], cfg["H_kv"]],
                   "head_dim": cfg["d"], "kv_len": list(cfg["L"]), "vocab": cfg["V"], "mode": cfg["mode"],
                   "cache": "page pools of 128-row pages behind shuffled page tables" if args.paged else "contiguous",
                   "l2": f"{n_sets} distinct input sets rotated ({n_sets * ab['total'] / 1e6:.0f} MB > 2 x L2)",
                   "launch": "CUDA graph replay of the C-ABI calls (" +
                             ("space_attn_step, space_verify, space_kv_commit" if args.separate_commit
                              else "space_attn_step, space_verify_commit") + ")",
                   "timed_region": f"median of {n_repeats} repeats of {K} steps" if n_repeats > 1
                                   else f"one region of {K} steps",
                   "parallelism": "replicas" if world > 1 else "single"},
        "gpu_launches": int(launches_per_step * K),
        "step_algorithmic_bytes": step_bytes,
        "step_hbm_frac": step_bytes / (ms / K * 1e-3) / 1e9 / peak,
        "roofline": {**roof, "kernel": "attn_tc_kernel" if rows <= 64 else "attn_rows_kernel",
                     "traffic": measured_traffic(ATTN_TRAFFIC, cfg["name"]),
                     "algorithmic_bytes_per_launch": float(attn_bytes), "avg_launch_us": attn_us,
                     "launches_timed": int(attn_n),
                     "timing": "CUDA events around every launch, stream-launched pass after the graph-timed region",
                     "kernel_us": per_kernel_us},
        "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": h2d_full,
                "d2h_bytes_per_step": d2h_full, "steps": n_e2e, "matches_device_run": e2e_ok},
        "e2e_resident_cache": {"value": res_val, "unit": UNIT, "h2d_bytes_per_step": h2d_res,
                               "d2h_bytes_per_step": int(d2h.value), "steps": n_res,
                               "matches_device_run": res_ok,
                               "note": "space_step_host with cache_resident=1: only the block's K/V rows, q, the "
                                       "candidates and the rows of logits that verification reads go up; the "
                                       "verified cache stays on the device"},
        "cpu_baseline": {"value": cpu_sps, "unit": UNIT, "cores": blas_threads(), "kind": "oracle",
                         "sample": f"{cpu_reps} whole step(s) of {cfg['name']} in {cpu_el:.1f} s"},
        "clocks": clocks,
        "device_status_bits": status,
    }
    print(json.dumps(line), flush=True)
    replicas.shutdown()


# ------------------------------------------------- projection + verify workloads
def oracle_lmhead_step(cfg, x):
    from oracle.lmhead import lmhead_verify_step
    return lmhead_verify_step(x["hidden"], x["weight"], x["cand"], x["cand_prob"], cfg["k"])


def run_lmhead(args):
    """space_lmhead_verify on a projection workload: one step = one call (one kernel)."""
    import torch
    from paper_2402_11809_b200 import device as H
    from paper_2402_11809_b200 import build
    build.build()
    from paper_2402_11809_b200 import binding as B

    rank, world, local = replicas.rank_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py --impl ours needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    replicas.init("nccl", local)
    cfg = workloads.resolve_lmhead(args.config)
    Bn, k, V, D = cfg["B"], cfg["k"], cfg["V"], cfg["D"]
    n_q = workloads.n_block_rows(k)
    ab = workloads.lmhead_algorithmic_bytes(cfg)
    n_sets = min(8, max(2, int(np.ceil(2.0 * L2_BYTES / ab["total"]))))
    sets = [workloads.make_lmhead_inputs(cfg, set_index=replicas.set_index(rank, i)) for i in range(n_sets)]
    ctx = B.Context(device=local, max_batch=Bn, n_q_heads=8, n_kv_heads=8, head_dim=64, k_max=k, vocab=V, s_cap=256)
    dev = "cuda"
    bufs, arg_sets = [], []
    for x in sets:
        d = dict(hidden=H.to_dev(x["hidden"]), weight=H.to_dev(x["weight"]), cand=H.to_dev(x["cand"]),
                 n_accept=torch.zeros(Bn, dtype=torch.int32, device=dev),
                 out_tokens=torch.zeros((Bn, k + 1), dtype=torch.int32, device=dev),
                 n_out=torch.zeros(Bn, dtype=torch.int32, device=dev),
                 next_cand=torch.zeros((Bn, k), dtype=torch.int32, device=dev),
                 next_cand_prob=torch.zeros((Bn, k), device=dev),
                 finished=torch.zeros(Bn, dtype=torch.uint8, device=dev),
                 status=torch.zeros(Bn, dtype=torch.int32, device=dev))
        bufs.append(d)
        arg_sets.append(ctx.lmhead_args(d["hidden"], d["weight"], d["cand"], d["n_accept"], d["out_tokens"],
                                        d["n_out"], d["next_cand"], d["next_cand_prob"], d["finished"], k,
                                        status=d["status"]))

    def step(i):
        ctx.space_lmhead_verify(arg_sets[i % n_sets])

    stream = torch.cuda.Stream()
    K, W = args.steps, max(args.warmup, 3)
    with torch.cuda.stream(stream):
        for i in range(n_sets):
            step(i)
        stream.synchronize()
        g_full = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g_full, stream=stream):
            for i in range(n_sets):
                step(i)

        def run_steps(n):
            for _ in range(n // n_sets):
                g_full.replay()
            for i in range(n % n_sets):
                step(i)

        run_steps(W)
        stream.synchronize()
        sampler = ClockSampler(local)
        replicas.barrier()
        torch.cuda.synchronize()
        sampler.start()
        ms, n_repeats, _ = timed_region(run_steps, K, stream, replicas.barrier)
        torch.cuda.synchronize()
        replicas.barrier()
        n_prof = min(max(K, 64), 2048)
        ctx.space_profile_enable(1)
        for i in range(n_prof):
            step(i)
        stream.synchronize()
        ctx.space_profile_enable(0)
        prof = ctx.space_profile_read()
        clocks = sampler.stop()
        status = sum(int(d["status"].abs().sum()) for d in bufs)
    steps_per_s, sec = replicas.job_throughput(K, ms * 1e-3, device="cuda")
    ms = sec * 1e3

    # ---- end to end: the step's own inputs (hidden states, candidates) come from pinned host
    # memory every step and its results are read back; the output embedding is model state and
    # stays on the device
    x, d = sets[0], bufs[0]
    pin_h = torch.from_numpy(x["hidden"].view(np.int16)).clone().pin_memory()
    pin_c = torch.from_numpy(x["cand"]).clone().pin_memory()
    res_names = ("n_accept", "out_tokens", "n_out", "next_cand", "next_cand_prob", "finished", "status")
    pin_o = {n_: torch.empty_like(d[n_], device="cpu").pin_memory() for n_ in res_names}
    h2d = pin_h.numel() * 2 + pin_c.numel() * 4
    d2h = sum(t.numel() * t.element_size() for t in pin_o.values())
    n_e2e = max(3, min(K, 1000))
    with torch.cuda.stream(stream):
        def host_step():
            d["hidden"].view(torch.int16).copy_(pin_h, non_blocking=True)
            d["cand"].copy_(pin_c, non_blocking=True)
            ctx.space_lmhead_verify(arg_sets[0])
            for n_ in res_names:
                pin_o[n_].copy_(d[n_], non_blocking=True)
            stream.synchronize()
        for _ in range(3):
            host_step()
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            host_step()
        e2e_s = time.perf_counter() - t0
    e2e_val, _ = replicas.job_throughput(n_e2e, e2e_s, device="cuda")
    if rank != 0:
        replicas.shutdown()
        return
    peak, peak_tf, peak_src = load_peaks()
    k_ms, k_n = prof["lmhead"]
    k_us = 1e3 * k_ms / max(k_n, 1)
    achieved = ab["total"] / (k_us * 1e-6) / 1e9 if k_n else None
    ref = oracle_lmhead_step(cfg, sets[0])
    matches = bool(np.array_equal(pin_o["n_accept"].numpy(), ref["n_accept"]) and
                   np.array_equal(pin_o["out_tokens"].numpy(), ref["out_tokens"]) and
                   np.array_equal(pin_o["next_cand"].numpy(), ref["next_cand"]))
    t0 = time.perf_counter()
    reps = 0
    while reps < 2 or time.perf_counter() - t0 < 10.0:
        oracle_lmhead_step(cfg, sets[0])
        reps += 1
    cpu_el = time.perf_counter() - t0
    line = {
        "metric": "projection+verify steps/sec", "value": steps_per_s, "unit": UNIT, "n_gpus": world, "steps": K,
        "warmup": W, "ms_per_step": ms / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16", "data": "synthetic",
        "config": {"workload": cfg["name"], "batch": Bn, "k": k, "vocab": V, "hidden_dim": D,
                   "l2": f"{n_sets} distinct weight sets rotated ({n_sets * ab['total'] / 1e6:.0f} MB > 2 x L2)",
                   "launch": "CUDA graph replay of the C-ABI call",
                   "parallelism": "replicas" if world > 1 else "single"},
        "gpu_launches": int(K),
        "step_algorithmic_bytes": float(ab["total"]),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "peak_source": peak_src + " (burst copy figure)",
                     "frac": (achieved / peak) if achieved else None, "kernel": "lmhead_verify_kernel",
                     "traffic": measured_traffic(LMHEAD_TRAFFIC, cfg["name"]),
                     "algorithmic_bytes_per_launch": float(ab["total"]), "avg_launch_us": k_us,
                     "launches_timed": int(k_n),
                     "timing": "CUDA events around every launch, stream-launched pass after the graph-timed region"},
        "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
                "steps": n_e2e, "matches_oracle": matches,
                "note": "hidden states and candidates uploaded from pinned host memory and results read back "
                        "every step; the output embedding is model state resident on the device"},
        "cpu_baseline": {"value": reps / cpu_el, "unit": UNIT, "cores": blas_threads(), "kind": "oracle",
                         "sample": f"{reps} whole step(s) of {cfg['name']} in {cpu_el:.1f} s"},
        "clocks": clocks,
        "device_status_bits": status,
    }
    print(json.dumps(line), flush=True)
    replicas.shutdown()


def run_lmhead_reference(args):
    rank, _, _ = replicas.rank_env()
    if rank != 0:
        return
    cfg = workloads.resolve_lmhead(args.config)
    x = workloads.make_lmhead_inputs(cfg)
    oracle_lmhead_step(cfg, x)
    t0 = time.perf_counter()
    oracle_lmhead_step(cfg, x)
    one = time.perf_counter() - t0
    reps = max(1, min(args.steps, int(150.0 / max(one, 1e-6))))
    t0 = time.perf_counter()
    for _ in range(reps):
        oracle_lmhead_step(cfg, x)
    el = time.perf_counter() - t0
    sps = reps / el
    print(json.dumps({
        "impl": "reference", "metric": "projection+verify steps/sec", "value": sps, "unit": UNIT,
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 / sps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": cfg["name"], "timed_steps": reps,
                   "note": "CPU oracle (numpy fp64), whole steps; repetitions bounded to ~150 s"},
        "cpu_baseline": {"value": sps, "unit": UNIT, "cores": blas_threads(), "kind": "oracle",
                         "sample": f"{reps} whole step(s) of {cfg['name']} in {el:.1f} s"},
        "e2e": {"value": sps, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20000)
    ap.add_argument("--warmup", type=int, default=50)
    ap.add_argument("--config", default="llama7b",
                    choices=sorted(workloads.CONFIGS) + sorted(workloads.LMHEAD_CONFIGS))
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--batch", type=int, default=0,
                    help="override the workload's batch size (a smaller copy of a large workload for profiler "
                         "captures; the bench line then names the workload NAME@batchN)")
    ap.add_argument("--separate-commit", action="store_true",
                    help="three calls per step (space_verify, then space_kv_commit) instead of space_verify_commit")
    ap.add_argument("--top-k", type=int, default=0, dest="top_k",
                    help="sampling workloads: verify against top-k / top-p filtered distributions (0 = unfiltered)")
    ap.add_argument("--top-p", type=float, default=1.0, dest="top_p")
    ap.add_argument("--k", type=int, default=0, help="number of mask tokens k instead of the workload's own")
    ap.add_argument("--paged", action="store_true",
                    help="keep the KV caches as page pools behind page tables (attention and commit through the table)")
    ap.add_argument("--attn-impl", default="tensor", choices=["tensor", "rows"],
                    help="tensor: keys on the MMA M extent (default); rows: query rows on M")
    args = ap.parse_args()
    if args.config in workloads.LMHEAD_CONFIGS:
        if args.steps == 20000:
            args.steps = 4000
        (run_lmhead_reference if args.impl == "reference" else run_lmhead)(args)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
