"""Benchmark: full-inventory Wide & Deep scoring + top-K of single requests.

Workload (default): 2,000,000 ads, d = 64 FP32 embeddings, 16 user x 16 ad
fields, 64 cross pairs, hashed 2^24 cross-weight table, K = 500 (the plain FP32
single-request path at inventory scale).  A step is one request through the
whole hot path: query expansion, the wide term via the compressed inverted list
(Algorithm 2), the streaming inner product with the fused wide add and top-K,
and the final selection.

Prints one JSON line.  `value` is ads scored per second with inputs resident in
device memory; `e2e` is the same metric through the C ABI with host buffers
(host->device copy of the request and device->host copy of the K results inside
the timed region).  Between timed steps the L2 cache is flushed by writing a
256 MiB buffer (outside the per-step events).

--impl reference times the FP64 CPU oracle on the host cores instead.
--gpus N (under torchrun): N independent replicas, one per GPU; the path has no
cross-GPU exchange, so `value` sums the replicas' throughput (weak scaling).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2511_22460_gb300.datagen import make_workload  # noqa: E402

WORKLOAD = "single_fp32_2m"
METRIC = "ads scored/s"
UNIT = "ads/s"


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def _config(w, extra=None, batch=1):
    r = w.recipe
    emb_mb = r.n_ads * r.d * {"f32": 4, "bf16": 2, "fp8e4m3": 1}[r.emb_dtype] / 2**20
    cfg = {"workload": r.name, "n_ads": r.n_ads, "d": r.d, "emb_dtype": r.emb_dtype,
           "user_fields": r.f_u, "ad_fields": r.f_a, "cross_pairs": int(len(w.pairs)),
           "weights": "hashed 2^24 FP32" if r.weights == "hashed" else "dense per pair",
           "k": int(w.ks[0]), "n_keys": w.n_keys, "postings": w.nnz,
           "l2": "flushed between steps (256 MiB write); embedding table %.0f MiB" % emb_mb}
    if batch > 1:
        cfg.update({"batch": batch, "k_per_user": sorted(set(int(x) for x in w.ks[:batch])),
                    "rescore_mult": r.rescore_mult})
    elif r.rescore_mult:
        cfg["rescore_mult"] = r.rescore_mult
    if extra:
        cfg.update(extra)
    return cfg


def max_over_ranks(x, device):
    """Largest value of x over the ranks of the default process group (x itself
    when there is none): the job is as slow as its slowest replica."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank, world, total_ms):
    """Units per second of the whole job: every rank processed units_per_rank
    in at most total_ms (the max over ranks)."""
    return units_per_rank * world / (total_ms / 1e3)


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.Q,
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def run_gpu(args, rank, world, local_rank):
    import torch

    torch.cuda.set_device(local_rank)
    w = _workload(args)
    if w.bench_batch > 1:
        return run_gpu_batched(args, w, rank, world, local_rank)
    out = run_single(args, w, rank, world, local_rank, workload=args.workload)
    del w
    if world == 1 and not args.no_extras and args.workload == WORKLOAD and not args.sparse_query:
        # the other workloads of the method, one object each on the same line
        t0 = time.perf_counter()
        wb = make_workload("batch256_bf16_5m", seed=args.seed)
        out["batched_bf16_5m_b256"] = run_gpu_batched(args, wb, rank, world, local_rank,
                                                      steps=args.extra_steps, cpu_users=2)
        del wb
        w8 = make_workload("fp8_10m", seed=args.seed, batch=64)
        out["fp8_10m_single"] = run_single(args, w8, rank, world, local_rank, workload="fp8_10m",
                                           steps=args.extra_steps, n_req=8, cpu_requests=2)
        out["fp8_10m_b64"] = run_gpu_batched(args, w8, rank, world, local_rank,
                                             steps=args.extra_steps, cpu_users=0)
        del w8
        out["extras_s"] = round(time.perf_counter() - t0, 1)
    if world == 1 and not args.no_serve and args.workload == WORKLOAD and not args.sparse_query:
        out["serving"] = run_serving(args, device=local_rank)
    return out


def run_single(args, w, rank, world, local_rank, workload, steps=None, n_req=16,
               cpu_requests=64):
    """A step is one request (a different user each step, round robin over
    n_req users) through the single-request path."""
    import torch

    from paper_2511_22460_gb300 import ebr

    dev = torch.device("cuda", local_rank)
    st = torch.cuda.current_stream()
    steps = steps or args.steps
    pk, pa = w.postings()
    ix = ebr.build_index(w.n_ads, w.n_keys, pk, pa, w.emb, dtype=w.recipe.emb_dtype,
                         device=local_rank)
    del pk, pa
    cross = ebr.cross_from_workload(w, device=local_rank)
    info = ix.info()
    k = int(w.ks[0])
    nreq = min(w.users.shape[0], n_req)
    h_u = torch.from_numpy(w.h_u).to(dev)
    users = torch.from_numpy(w.users).to(dev)
    ids = torch.empty(k, dtype=torch.int32, device=dev)
    sc = torch.empty(k, dtype=torch.float32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)

    # a sparse query (--sparse-query N): N keys carry the weights, so the
    # key-major traversal (Algorithm 2) serves it; else the user's fields
    # expand to a dense w^ and the fused window-major scan serves it
    sparse = args.sparse_query > 0
    if sparse:
        from paper_2511_22460_gb300.datagen import sparse_query
        sq = [sparse_query(w, args.sparse_query, seed=b) for b in range(nreq)]
        sq_d = [(torch.from_numpy(qk).to(dev), torch.from_numpy(qw).to(dev)) for qk, qw in sq]

    def query(b, host=False):
        if sparse:
            qk, qw = sq[b] if host else sq_d[b]
            return ebr.Query(h_u=(w.h_u[b].copy() if host else h_u[b]), k=k, q_key=qk, q_w=qw,
                             flags={"auto": 0, "key": ebr.QF_KEY_MAJOR,
                                    "window": ebr.QF_WINDOW_MAJOR}[args.sparse_route])
        if host:
            return ebr.Query(h_u=w.h_u[b].copy(), k=k, user_vals=w.users[b].copy())
        return ebr.Query(h_u=h_u[b], k=k, user_vals=users[b])

    def step(i):
        ebr.score_topk(ix, cross, [query(i % nreq)], ids, sc, stream=st)

    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    launches0 = ix.profile_read().launches
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(steps)]
    clocks = ClockSampler(local_rank)
    clocks.start()
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    for i in range(steps):
        flush.zero_()
        evs[i][0].record(st)
        step(i)
        evs[i][1].record(st)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    clk = clocks.stop()
    times = [a.elapsed_time(b) for a, b in evs]
    launches = ix.profile_read().launches - launches0
    total_ms = max_over_ranks(float(sum(times)), dev)
    ms_step = total_ms / steps
    value = whole_job_rate(w.n_ads * steps, world, total_ms)
    # Per-stage device time from a separate pass of the same steps: the stage
    # events sit between the kernels, which keeps a kernel from starting while
    # the one before it ends, so they stay out of the timed steps above.
    ix.profile_enable(True)
    for i in range(steps):
        flush.zero_()
        step(i)
    torch.cuda.synchronize()
    prof = ix.profile_read()
    ix.profile_enable(False)

    # End to end through the C ABI with host buffers (request in, K results out).
    hk_ids = np.empty(k, np.uint32)
    hk_sc = np.empty(k, np.float32)
    hqs = [query(b, host=True) for b in range(nreq)]
    e2e_t = []
    for i in range(args.warmup + steps):
        b = i % nreq
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ebr.score_topk(ix, cross, [hqs[b]], hk_ids, hk_sc, io=ebr.IO_HOST, stream=st)
        t1 = time.perf_counter()
        if i >= args.warmup:
            e2e_t.append(t1 - t0)
    e2e_val = w.n_ads * len(e2e_t) / sum(e2e_t)

    peak, peak_kind = _peaks()
    scan_ms = prof.ms_scan / max(prof.calls, 1)
    emb_bytes = info.emb_bytes
    # the scan must read the embedding table and the forward key table: every
    # posting's key id (16 or 24 bits) and the offsets of its runs of 32 ads
    key_id_bytes = 2 if w.n_keys < 65536 else 3
    kern_bytes = emb_bytes + key_id_bytes * info.nnz_unique + 4 * (w.n_ads // 32 + 1)
    if w.recipe.emb_dtype != "f32":
        kern_bytes += 4 * w.n_ads  # the FP32 wide term, written for the rescoring
    kernel = "k_forward"
    bytes_note = ("embedding table (+ FP8 row scales) + forward key table (a key id per posting, "
                  "run offsets) (+ FP32 wide term out when the table is quantised), per launch")
    routes = None
    if sparse:
        # per launch, the scan either reads the wide term Algorithm 2 scattered
        # or the forward key table
        if args.sparse_route == "auto":
            n_win_r = int(prof.window_routed)
            n_key_r = int(prof.auto_routed - prof.window_routed)
        else:
            n_win_r = steps if args.sparse_route == "window" else 0
            n_key_r = steps - n_win_r
        routes = {"window_major": n_win_r, "key_major": n_key_r}
        key_bytes = emb_bytes + 4 * w.n_ads
        kern_bytes = ((n_win_r * kern_bytes + n_key_r * key_bytes) /
                      max(n_win_r + n_key_r, 1))
        bytes_note = ("embedding table (+ FP8 row scales) + per launch either the FP32 wide "
                      "term read (Algorithm 2 scattered it) or the forward key table (+ FP32 "
                      "wide term out when the table is quantised), averaged over the routes "
                      "the requests took")
    achieved = kern_bytes / (scan_ms / 1e3) / 1e9
    step_bytes = kern_bytes
    traffic = None
    tr_path = os.path.join(ROOT, "profiles", "scan_traffic.json")
    if os.path.exists(tr_path) and not sparse:
        with open(tr_path) as f:
            records = json.load(f)
        for tr in records if isinstance(records, list) else [records]:
            if tr.get("workload") == workload and tr.get("kernel_rev") == KERNEL_REV:
                traffic = tr.get("bytes_per_launch")
    launches_per_step = launches / max(steps, 1)
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": w.recipe.emb_dtype,
        "data": "synthetic",
        "config": _config(w, {"replicas": world, "build_ms": round(info.build_ms, 3),
                              "query": ("sparse: %d keys with weights, %s-major" %
                                        (args.sparse_query, args.sparse_route)
                                        if sparse else "user fields, dense w^"),
                              "window_view_ms": round(info.window_view_ms, 3),
                              "index_bytes": info.index_bytes,
                              "window_view_bytes": info.window_view_bytes}),
        "latency_us": {"p50": 1e3 * float(np.percentile(times, 50)),
                       "p99": 1e3 * float(np.percentile(times, 99))},
        "req_per_s": 1e3 / ms_step * world,
        "step_hbm_gbs": step_bytes / (ms_step / 1e3) / 1e9,
        "stage_ms": {"expand": prof.ms_expand / prof.calls, "wide": prof.ms_wide / prof.calls,
                     "scan_topk": scan_ms, "final": prof.ms_final / prof.calls},
        **({"sparse_routes": routes} if routes else {}),
        "roofline": {"kernel": kernel, "bound": "hbm", "achieved": achieved,
                     "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "peak_kind": peak_kind, "traffic": traffic,
                     "algorithmic_bytes": kern_bytes,
                     "bytes_note": bytes_note},
        "e2e": {"value": e2e_val, "unit": UNIT,
                "h2d_bytes_per_step": int(w.recipe.d * 4 + (8 * args.sparse_query if sparse
                                                            else w.recipe.f_u * 4)),
                "d2h_bytes_per_step": int(k * 8)},
        "gpu_launches": int(round(launches_per_step * steps)),
        "gpu_launches_per_step": launches_per_step,
        "clocks": clk,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline and cpu_requests:
        out["cpu_baseline"] = cpu_baseline(w, budget_s=args.cpu_budget, max_req=cpu_requests)
    del ix, h_u, users, flush
    return out


KERNEL_REV = "forward-v3"

# FP32 add throughput of the CUDA cores: 152 SMs x 128 FP32 lanes x 2.07 GHz
ALU_ADD_PEAK_T = 152 * 128 * 2.07e9 / 1e12


def _workload(args):
    """The workload's arrays; a single-request run draws 16 users (one per
    step, round robin), a batched run the batch's users."""
    from paper_2511_22460_gb300.datagen import RECIPES
    kw = {}
    if args.n_ads:
        kw["n_ads"] = args.n_ads
    batch = args.batch or RECIPES[args.workload].batch
    kw["batch"] = batch if batch > 1 else 16
    w = make_workload(args.workload, seed=args.seed, **kw)
    w.bench_batch = batch
    return w


def run_gpu_batched(args, w, rank, world, local_rank, steps=None, cpu_users=None):
    """A step is one batched call: every user of the batch against the whole
    inventory (tensor-core deep term, wide term from the compressed lists,
    per-user top-K with FP32 rescoring)."""
    import torch

    from paper_2511_22460_gb300 import ebr

    steps = steps or args.steps

    dev = torch.device("cuda", local_rank)
    st = torch.cuda.current_stream()
    pk, pa = w.postings()
    ix = ebr.build_index(w.n_ads, w.n_keys, pk, pa, w.emb, dtype=w.recipe.emb_dtype,
                         device=local_rank)
    del pk, pa
    cross = ebr.cross_from_workload(w, device=local_rank)
    info = ix.info()
    B = getattr(w, "bench_batch", w.recipe.batch)
    ks = [int(x) for x in w.ks[:B]]
    kmax = max(ks)
    h_u = torch.from_numpy(w.h_u).to(dev)
    users = torch.from_numpy(w.users).to(dev)
    filt = None if w.filters is None else torch.from_numpy(w.filters.view(np.int64)).to(dev)
    qs = [ebr.Query(h_u=h_u[b], k=ks[b], user_vals=users[b],
                    filter=None if filt is None else filt[b]) for b in range(B)]
    ids = torch.empty((B, kmax), dtype=torch.int32, device=dev)
    sc = torch.empty((B, kmax), dtype=torch.float32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)

    def step():
        ebr.score_topk(ix, cross, qs, ids, sc, stream=st)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    ix.profile_enable(True)
    p0 = ix.profile_read()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(steps)]
    clocks = ClockSampler(local_rank)
    clocks.start()
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    for i in range(steps):
        flush.zero_()
        evs[i][0].record(st)
        step()
        evs[i][1].record(st)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    clk = clocks.stop()
    times = [a.elapsed_time(b) for a, b in evs]
    prof = ix.profile_read()
    ix.profile_enable(False)
    total_ms = max_over_ranks(float(sum(times)), dev)
    ms_step = total_ms / steps
    value = whole_job_rate(w.n_ads * B * steps, world, total_ms)
    # end to end with host buffers: requests in, B x K results out
    hq = [ebr.Query(h_u=np.ascontiguousarray(w.h_u[b]), k=ks[b],
                    user_vals=np.ascontiguousarray(w.users[b]),
                    filter=None if w.filters is None else np.ascontiguousarray(w.filters[b]))
          for b in range(B)]
    hids = np.empty((B, kmax), np.uint32)
    hsc = np.empty((B, kmax), np.float32)
    e2e_t = []
    for i in range(args.warmup + steps):
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ebr.score_topk(ix, cross, hq, hids, hsc, io=ebr.IO_HOST, stream=st)
        if i >= args.warmup:
            e2e_t.append(time.perf_counter() - t0)
    e2e_val = w.n_ads * B * len(e2e_t) / sum(e2e_t)
    h2d = B * (w.recipe.d * 4 + w.recipe.f_u * 4) + (0 if w.filters is None else w.filters.nbytes)
    calls = max(prof.batch_calls, 1)
    scan_ms = prof.ms_batch_scan / calls
    adds = B * info.nnz_unique  # the wide term's FP32 adds of one batched scan
    achieved = adds / (scan_ms / 1e3) / 1e12
    gemm_flop = 2.0 * B * w.n_ads * w.recipe.d  # the deep term on the tensor cores
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": w.recipe.emb_dtype, "data": "synthetic",
        "config": _config(w, {"replicas": world, "units": "user x ad pairs scored"}, batch=B),
        "req_per_s": B * 1e3 / ms_step * world,
        "latency_ms": {"p50": float(np.percentile(times, 50)),
                       "p99": float(np.percentile(times, 99))},
        "stage_ms": {"stage_expand": prof.ms_batch_stage / calls, "scan": scan_ms,
                     "merge_rescore": prof.ms_batch_merge / calls},
        "recomputed_users": int(prof.recomputed - p0.recomputed),
        "tensor_tflops": gemm_flop / (scan_ms / 1e3) / 1e12,
        "roofline": {"kernel": "k_batch_window", "bound": "alu", "achieved": achieved,
                     "peak": ALU_ADD_PEAK_T, "unit": "Tadd/s", "frac": achieved / ALU_ADD_PEAK_T,
                     "peak_kind": "derived: 152 SMs x 128 FP32 lanes x 2.07 GHz",
                     "traffic": None, "algorithmic_ops": adds,
                     "ops_note": "B x distinct (key, ad) postings FP32 adds of the wide term"},
        "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(B * kmax * 8)},
        "gpu_launches": int(prof.launches - p0.launches),
        "gpu_launches_per_step": (prof.launches - p0.launches) / max(steps, 1),
        "clocks": clk,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline and cpu_users != 0:
        out["cpu_baseline"] = cpu_baseline(w, budget_s=args.cpu_budget, max_req=cpu_users or 64)
    del ix
    return out


MODE_NAMES = {False: "device-resident loop (one graph launch; a WHILE node running waves)",
              True: "host-driven pipelines (a host launch per batch, two in flight)"}


def run_serving(args, device=0):
    """Serving form (the 5,000,000-ad BF16 d=64 serving workload): open-loop
    Poisson arrivals through ebr_submit/ebr_poll at each offered rate, each
    request with its own user, K in {100, 500, 1000} and targeting bitmap;
    p50/p99 from submit to result visible; then the plain per-request FP32 path
    on the same inventory through ebr_score_topk with host buffers."""
    import torch

    from paper_2511_22460_gb300 import ebr
    from paper_2511_22460_gb300.datagen import poisson_arrivals

    t_gen = time.perf_counter()
    pool = args.serve_pool
    w = make_workload("serve_bf16_5m", seed=args.seed, batch=pool)
    pk, pa = w.postings()
    gen_s = time.perf_counter() - t_gen
    ix = ebr.build_index(w.n_ads, w.n_keys, pk, pa, w.emb, dtype="bf16", device=device)
    cross = ebr.cross_from_workload(w, device=device)
    ks = [int(x) for x in w.ks]
    reqs = [(np.ascontiguousarray(w.h_u[b]), np.ascontiguousarray(w.users[b]), ks[b],
             np.ascontiguousarray(w.filters[b])) for b in range(pool)]
    def drive(srv, rate, duration, keep=None):
        # one thread: submit every request whose arrival time has passed, then
        # retire whatever the server reports finished (no lock, no GIL contention);
        # `keep` collects (user, K, ids) of the first results of distinct users
        arr = poisson_arrivals(rate, duration, seed=args.seed + int(rate))
        outstanding = {}
        n_done = rejected = failed = 0
        last = 0.0
        i = 0
        t0 = time.perf_counter()
        while i < len(arr) or outstanding:
            now = time.perf_counter() - t0
            busy = False
            while i < len(arr) and arr[i] <= now:
                b = i % pool
                h, u, k, f = reqs[b]
                t = srv.submit(h, u, k, f)
                if t is None:
                    rejected += 1
                else:
                    outstanding[t] = b
                i += 1
                busy = True
            for t in srv.completed():
                b = outstanding.pop(int(t))
                busy = True
                try:
                    res = srv.poll(int(t), ks[b])
                except ebr.EbrError:
                    failed += 1
                    continue
                if keep is not None and len(keep) < args.serve_check and \
                        all(kb != b for kb, _, _ in keep):
                    keep.append((b, ks[b], res[0].copy()))
                n_done += 1
                last = time.perf_counter()
            if not busy:
                time.sleep(2e-5)
        span = max(last, t0 + duration) - t0
        return len(arr), n_done, rejected + failed, span

    def serve(host_driven, rates, seconds, checks=None):
        srv = ebr.Server(ix, cross, max_batch=args.serve_batch, max_slots=4096, k_max=1000,
                         host_driven=host_driven)
        drive(srv, 2000.0, 0.3)  # warm-up
        rows = []
        launches = srv.stats().loop_launches
        for rate in rates:
            srv.reset_stats()
            keep = [] if checks is not None else None
            offered, n_done, rejected, span = drive(srv, rate, seconds, keep)
            st = srv.stats()
            launches += st.loop_launches
            rows.append({"offered_req_s": rate, "submitted": offered, "completed": n_done,
                         "rejected": rejected, "req_per_s": n_done / span,
                         "p50_ms": st.p50_ms, "p99_ms": st.p99_ms, "mean_ms": st.mean_ms,
                         "mean_batch": st.batched_requests / max(st.batches, 1)})
            if checks is not None:
                checks.append(keep)
        mb = srv.stats().max_batch
        srv.close()
        return rows, launches, mb

    checks = []
    rows, loop_launches, max_batch = serve(args.serve_host_driven, args.serve_rates,
                                           args.serve_seconds, checks)
    other = None
    if not args.no_serve_compare:  # the other form, fewer rates, for comparison
        orows, olaunch, _ = serve(not args.serve_host_driven, (2000.0, 10000.0, 20000.0),
                                  max(2.0, args.serve_seconds / 2))
        other = {"mode": MODE_NAMES[not args.serve_host_driven], "loop_launches": int(olaunch),
                 "rates": orows, "max_req_per_s": max(r["req_per_s"] for r in orows)}
    # the plain per-request FP32 path on the same inventory, host buffers
    del ix
    ix32 = ebr.build_index(w.n_ads, w.n_keys, pk, pa, w.emb, dtype="f32", device=device)
    ids = np.empty(1000, np.uint32)
    sc = np.empty(1000, np.float32)
    for i in range(3):
        h, u, k, f = reqs[i]
        ebr.score_topk(ix32, cross, [ebr.Query(h_u=h, k=k, user_vals=u, filter=f)], ids, sc,
                       io=ebr.IO_HOST)
    n32 = args.serve_fp32_requests
    t0 = time.perf_counter()
    for i in range(n32):
        h, u, k, f = reqs[i % pool]
        ebr.score_topk(ix32, cross, [ebr.Query(h_u=h, k=k, user_vals=u, filter=f)], ids, sc,
                       io=ebr.IO_HOST)
    fp32_rps = n32 / (time.perf_counter() - t0)
    del ix32
    torch.cuda.synchronize()
    # recall@K of the served results against the FP64 oracle (after the timed
    # region; the oracle runs on every host core)
    t_chk = time.perf_counter()
    rec = served_recall(w, [x for keep in checks for x in keep], pk, pa)
    i = 0
    for row, keep in zip(rows, checks):
        r = rec[i:i + len(keep)]
        i += len(keep)
        row["recall_checked"] = len(keep)
        row["recall_min"] = float(min(r)) if r else None
        row["recall_mean"] = float(np.mean(r)) if r else None
    best = max(rows, key=lambda r: r["req_per_s"])
    return {"workload": "serve_bf16_5m", "n_ads": w.n_ads, "d": w.recipe.d,
            "emb_dtype": "bf16 + FP32 rescoring (R=4)", "ad_fields": w.recipe.f_a,
            "cross_pairs": int(len(w.pairs)), "k_choices": [100, 500, 1000],
            "filter_fraction": "U[0.01, 1] per request", "request_pool": pool,
            "max_batch": max_batch, "rates": rows,
            "mode": MODE_NAMES[bool(args.serve_host_driven)],
            "loop_launches": int(loop_launches), "other_mode": other,
            "max_req_per_s": best["req_per_s"],
            "recall": {"checked": len(rec), "min": float(min(rec)) if rec else None,
                       "definition": "|S_gpu & S_oracle| / K against the FP64 oracle, ids "
                                     "within the 1e-5 condition-scale tolerance of the K-th "
                                     "score counted as hits; the first results of distinct "
                                     "users at each rate",
                       "check_s": round(time.perf_counter() - t_chk, 1)},
            "seconds_per_rate": args.serve_seconds,
            "fp32_per_request_req_per_s": fp32_rps,
            "speedup_vs_fp32_per_request": best["req_per_s"] / fp32_rps,
            "datagen_s": round(gen_s, 1)}


def served_recall(w, samples, pk, pa):
    """recall@K of each (user, K, ids) against the FP64 oracle (Z8 tolerance
    for ties at the K-th score), one oracle call per thread."""
    import concurrent.futures as cf

    import oracle
    if not samples:
        return []
    cr = oracle.Cross.from_workload(w)
    cr_abs = oracle.Cross(w.vocab_u, w.vocab_a, w.pairs, np.abs(w.w_table), w.w_off,
                          hashed=cr.hashed, hash_bits=cr.hash_bits)
    emb_abs = np.abs(w.emb)

    def one(item):
        b, k, ids = item
        wh = oracle.expand(cr, w.users[b])
        keys = np.nonzero(wh)[0].astype(np.uint32)
        s = oracle.scores_postings(w.h_u[b], w.emb, w.n_keys, pk, pa, keys, wh[keys],
                                   assume_unique=True)
        wa = oracle.expand(cr_abs, w.users[b])
        ka = np.nonzero(wa)[0].astype(np.uint32)
        cond = oracle.scores_postings(np.abs(w.h_u[b]), emb_abs, w.n_keys, pk, pa, ka, wa[ka],
                                      assume_unique=True)
        tol = 1e-5 * np.maximum(np.abs(s), cond)
        elig = np.ones(w.n_ads, bool)
        if w.filters is not None:
            elig = np.unpackbits(w.filters[b].view(np.uint8), bitorder="little")[:w.n_ads] > 0
        r = np.where(elig, s, -np.inf)
        take = min(k, int(elig.sum()))
        if take == 0:
            return 1.0
        kth = np.partition(r, r.size - take)[r.size - take]
        got = np.asarray(ids[:take]).astype(np.int64)
        ok = (got >= 0) & (got < w.n_ads)
        got = got[ok]
        hit = int(np.sum(elig[got] & (s[got] >= kth - tol[got])))
        return hit / take

    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
        return list(ex.map(one, samples))


def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo), or 'unknown'."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    try:
        with open("/proc/cpuinfo") as f:
            for line in f:
                if line.lower().startswith(("model name", "cpu part")):
                    return line.split(":", 1)[1].strip()
    except Exception:
        pass
    return "unknown"


def cpu_baseline(w, budget_s=15.0, max_req=64):
    """FP64 oracle (expansion + postings walk + dot + full sort) on the host:
    one thread, then every core (one request per thread at a time; the C
    oracle releases the GIL)."""
    import concurrent.futures as cf

    import oracle
    cross = oracle.Cross.from_workload(w)
    pk, pa = w.postings()
    k = int(w.ks[0])
    nu = w.users.shape[0]

    def one(b):
        s = oracle.score_query(w, b, cross, (pk, pa))
        oracle.topk(s, k)

    t_total, n = 0.0, 0
    while t_total < budget_s and n < max_req:
        t0 = time.perf_counter()
        one(n % nu)
        t_total += time.perf_counter() - t0
        n += 1
    single = w.n_ads * n / t_total
    cores = os.cpu_count() or 1
    n_all = min(max(cores, 2 * n), 4 * max(cores, 1))
    t0 = time.perf_counter()
    with cf.ThreadPoolExecutor(max_workers=cores) as ex:
        list(ex.map(one, [i % nu for i in range(n_all)]))
    allc = w.n_ads * n_all / (time.perf_counter() - t0)
    return {"value": allc, "unit": UNIT, "cores": cores, "kind": "oracle",
            "single_thread_value": single, "cpu_model": cpu_model(),
            "sample": "%d full requests of the %s workload (%d ads each) on one thread, then %d "
                      "on %d threads" % (n, w.recipe.name, w.n_ads, n_all, cores)}


def run_reference(args):
    w = _workload(args)
    import oracle
    cross = oracle.Cross.from_workload(w)
    pk, pa = w.postings()
    k = int(w.ks[0])
    for i in range(args.warmup):
        s = oracle.score_query(w, i % w.users.shape[0], cross, (pk, pa))
        oracle.topk(s, k)
    t = []
    for i in range(args.steps):
        t0 = time.perf_counter()
        s = oracle.score_query(w, i % w.users.shape[0], cross, (pk, pa))
        oracle.topk(s, k)
        t.append(time.perf_counter() - t0)
    value = w.n_ads * len(t) / sum(t)
    return {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * sum(t) / len(t),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "impl": "reference", "config": _config(w),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": "%d full requests, single thread" % len(t)},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default=WORKLOAD)
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--cpu-budget", type=float, default=15.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-serve", action="store_true", help="skip the serving measurement")
    ap.add_argument("--serve-host-driven", action="store_true",
                    help="serve with the host-driven pipelines instead of the device-resident loop")
    ap.add_argument("--no-serve-compare", action="store_true",
                    help="skip the shorter run of the other serving form")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the batched BF16, FP8 single and FP8 batched lines")
    ap.add_argument("--extra-steps", type=int, default=10,
                    help="timed steps of each extra line")
    ap.add_argument("--n-ads", type=int, default=0, help="override the workload's inventory size")
    ap.add_argument("--batch", type=int, default=0, help="override the workload's users per step")
    ap.add_argument("--sparse-query", type=int, default=0,
                    help="requests carry this many (key, w) pairs instead of user fields")
    ap.add_argument("--sparse-route", choices=["auto", "key", "window"], default="auto",
                    help="traversal for sparse requests: chosen on the device by the list's "
                         "work (auto), Algorithm 2's key-major scatter, or the window-major "
                         "decode inside the fused scan")
    ap.add_argument("--serve-rates", type=float, nargs="+", default=[2000, 5000, 10000, 20000])
    ap.add_argument("--serve-seconds", type=float, default=10.0)
    ap.add_argument("--serve-batch", type=int, default=128)
    ap.add_argument("--serve-pool", type=int, default=256)
    ap.add_argument("--serve-check", type=int, default=16,
                    help="served results per rate checked against the FP64 oracle")
    ap.add_argument("--serve-fp32-requests", type=int, default=200)
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        if rank == 0:
            print(json.dumps(run_reference(args)))
        return
    if world > 1:
        import torch
        torch.cuda.set_device(local_rank)
        torch.distributed.init_process_group("nccl")
    out = run_gpu(args, rank, world, local_rank)
    if rank == 0:
        print(json.dumps(out))
    if world > 1:
        import torch
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
