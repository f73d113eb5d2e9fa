"""Benchmark: budgeted KV-cache repair on the Llama-3-8B-shaped workload.

Workload: random-init bf16 Llama-3-8B-shaped model (32 layers, d 4096,
32/8 heads, FFN 14336, vocab 128256), a cached document of 5000 uniform
random tokens, an 8-token same-length edit at position 2500, EditLocal
K = 32, so P = 40 rows recomputed through all 32 layers.

One step = the hot path once: kvr_select (EditLocal) + kvr_repair (edit
apply, then the 40 rows through every layer, K/V written back in place).
The full re-prefill of the edited 5000-token document is timed separately
as the baseline the speedup is quoted against.

Prints one JSON line (rank 0).  --impl reference times the CPU oracle on a
bounded sample of the same workload instead.
"""
from __future__ import annotations

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

WORKLOAD = "llama8b"
N_CTX, EDIT_START, EDIT_LEN, K_BUDGET = 5000, 2500, 8, 32
METRIC = "repair latency ms & positions/s at K=32, 5k ctx; speedup vs full re-prefill"


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def load_tensor_peak():
    """Dense bf16 TFLOP/s sustained over seconds (the prefill is a long run)."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["bf16_tflops_sustained"]), "measured"
    except Exception:
        return 1700.0, "fallback"


def prefill_flops(cfg, n: int) -> float:
    """Dense FLOPs of a prefill of n tokens as the library runs it: every
    layer's QKV projection; the O projection, MLP and causal attention of all
    layers but the last (their outputs feed no K/V of the cache)."""
    d, F, L = cfg["d_model"], cfg["ffn"], cfg["n_layers"]
    H, G, dh = cfg["n_heads"], cfg["n_kv_heads"], cfg["head_dim"]
    qkv = 2.0 * n * d * (H + 2 * G) * dh
    rest = 2.0 * n * (H * dh * d + 2 * F * d + F * d)
    attn = 4.0 * H * dh * n * (n + 1) / 2  # QK^T and PV over the causal triangle
    return L * qkv + (L - 1) * (rest + attn)


class Clocks:
    """Samples nvidia-smi clocks and throttle reasons while running."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "20"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
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
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            try:
                sm.append(float(r[1]))
                mx = float(r[2])
                for i, nm in enumerate(names):
                    if r[5 + i].lower() == "active":
                        reasons.add(nm)
            except (ValueError, IndexError):
                continue
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def edit_inputs(cfg):
    from paper_2609_17983_gb300 import synth
    doc = synth.document(1, N_CTX, cfg["vocab"], cfg["delim_id"])
    new = synth.edit_tokens(2, doc[EDIT_START:EDIT_START + EDIT_LEN], cfg["vocab"],
                            cfg["delim_id"])
    return doc, new


# ------------------------------------------------------------- CPU oracle

# CPU seconds the reference arm's W + K timed steps may take in all, and the
# GPU arm's one-step oracle sample (cpu_baseline)
REF_BUDGET_S = 150.0
CPU_BASELINE_S = 10.0
# seed of the synthetic stale cache (the one the full-depth parity test starts from)
STALE_SEED = 11


def oracle_setup(cfg, layers: int):
    """Inputs of the oracle's timed step: the workload's 40 rows (the span and
    its EditLocal window) of the edited document through the model's first
    `layers` decoder layers, each with its own seeded weights, over the seeded
    synthetic stale cache of the document's length restricted to those
    layers."""
    import oracle
    from paper_2609_17983_gb300 import synth
    doc, new = edit_inputs(cfg)
    edited = doc.copy()
    edited[EDIT_START:EDIT_START + EDIT_LEN] = new
    P = np.arange(EDIT_START, EDIT_START + EDIT_LEN + K_BUDGET)
    used = np.unique(edited[P])
    remap = {int(t): i for i, t in enumerate(used)}
    W = dict(embed=synth.rows(0, synth.TID_EMBED, used, cfg["d_model"], cfg["dtype"]),
             final_norm=synth.ones(cfg["d_model"], cfg["dtype"]), lm_head=None,
             layers=[synth.layer_weights(cfg, 0, l) for l in range(layers)])
    ocfg = dict(cfg, n_layers=layers, vocab=len(used))
    toks = np.zeros(N_CTX, np.int32)
    toks[P] = [remap[int(t)] for t in edited[P]]
    k, v = synth.kv_rows(STALE_SEED, N_CTX, cfg["n_layers"], cfg["n_kv_heads"],
                         cfg["head_dim"], cfg["dtype"])
    f32 = synth.bf16_bits_to_f32 if cfg["dtype"] == "bf16" else np.asarray
    cache = oracle.Cache(np.ascontiguousarray(f32(k[:, :layers]).transpose(1, 0, 2, 3)),
                         np.ascontiguousarray(f32(v[:, :layers]).transpose(1, 0, 2, 3)), toks)
    return dict(cfg=ocfg, W=W, cache=cache, toks=toks, P=P, layers=layers)


def oracle_time(sample) -> float:
    """Seconds of one oracle step: operator R on the sample's rows through its
    layers (R writes the same rows each time, so a sample can be rerun)."""
    import oracle
    t0 = time.perf_counter()
    oracle.recompute(sample["cfg"], sample["W"], sample["cache"], sample["toks"], sample["P"])
    return time.perf_counter() - t0


def oracle_value(cfg, layers: int, seconds: float) -> float:
    """positions/s of an oracle step that took `seconds` for the 40 rows through
    `layers` of the model's layers (a position is repaired by all of them)."""
    return (EDIT_LEN + K_BUDGET) * layers / cfg["n_layers"] / seconds


def run_reference(args, cfg, rank):
    """The oracle timed on the host cores as the reference arm.  Every step is
    the same bounded sample of the workload: the 40 rows through the model's
    first `layers` layers, as many (at most --oracle-layers) as let the W
    warm-up and K timed steps fit REF_BUDGET_S by a one-layer probe.
    ms_per_step is the step as it ran; value counts a position once per full
    depth (positions x layers_per_step / layers_per_position per second)."""
    import oracle
    if rank != 0:
        return None
    M = EDIT_LEN + K_BUDGET
    L = cfg["n_layers"]
    threads = oracle.set_threads(os.cpu_count() or 1)
    probe = oracle_setup(cfg, 1)
    t_layer = oracle_time(probe)
    runs = args.warmup + args.steps
    cap = args.oracle_layers or L
    layers = max(1, min(cap, L, int(REF_BUDGET_S / (runs * t_layer))))
    sample = probe if layers == 1 else oracle_setup(cfg, layers)
    for _ in range(args.warmup):
        oracle_time(sample)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle_time(sample)
    t = (time.perf_counter() - t0) / args.steps
    val = oracle_value(cfg, layers, t)
    desc = (f"oracle operator R on the {M} rows through the first {layers} of {L} layers "
            f"per step (each layer its own seeded weights, seeded synthetic stale cache)")
    return {"metric": METRIC, "value": val, "unit": "positions/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": t * 1e3,
            "layers_per_step": layers, "layers_per_position": L,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "impl": "reference",
            "config": workload_config(cfg, args.gpus),
            "cpu_baseline": {"value": val, "unit": "positions/s", "cores": threads,
                             "kind": "oracle", "sample": desc},
            "e2e": {"value": val, "unit": "positions/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


# ------------------------------------------------------------- GPU arm

# DRAM bytes (read + write) of one gate/up GEMM launch at this workload's shape
# (40 x 28672 x 4096), from one ncu capture of that launch; reported only while the
# GEMM kernel's source is the one the capture was taken on.
GU_TRAFFIC_BYTES = 235304192 + 4485632
GU_TRAFFIC_SOURCE_SHA256 = "8a82d2ea095f53a99fd92f52bb020d014fb94fe84da815b8e662963f02d3821b"


def workload_config(cfg: dict, world: int) -> dict:
    """The `config` of both arms' JSON lines: one workload, named the same."""
    return {"workload": f"{WORKLOAD}: Llama-3-8B shape, n={N_CTX}, "
                        f"edit {EDIT_LEN}@{EDIT_START}, editlocal K={K_BUDGET}",
            "rows": EDIT_LEN + K_BUDGET, "layers": cfg["n_layers"],
            "parallelism": "replicas" if world > 1 else "single",
            "l2": "inputs larger than L2 (14 GB of weights streamed per step)"}


def max_over_ranks(x: float, device) -> float:
    """The largest of every rank's x: a replicated job's step ends with its
    slowest rank.  Identity without an initialised process group."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(rows_per_rank: int, world: int, seconds: float) -> float:
    """Whole-job positions/s: the rows every rank repaired per step over the
    slowest rank's step time."""
    return world * rows_per_rank / seconds


def gemm_source_sha256() -> str:
    import hashlib
    h = hashlib.sha256()
    here = os.path.join(os.path.dirname(os.path.abspath(__file__)), "paper_2609_17983_gb300",
                        "csrc")
    for f in ("k_gemm_tc.cu", "kvr_internal.cuh", "tc_ptx.cuh"):
        with open(os.path.join(here, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def time_ms(fn, stream, reps: int = 3, warm: int = 1) -> float:
    """Median device time (CUDA events on `stream`) of fn over reps calls
    after warm untimed ones."""
    import torch
    t = []
    for i in range(warm + reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fn()
        b.record(stream)
        torch.cuda.synchronize()
        if i >= warm:
            t.append(a.elapsed_time(b))
    return statistics.median(t)


def pass_flops(cfg, positions) -> float:
    """Dense FLOPs of a K/V-only pass over rows at `positions` (as the library
    runs it: every layer's QKV projection, the O projection, MLP and causal
    attention over keys 0..p of all layers but the last)."""
    d, F, L = cfg["d_model"], cfg["ffn"], cfg["n_layers"]
    H, G, dh = cfg["n_heads"], cfg["n_kv_heads"], cfg["head_dim"]
    rows = len(positions)
    qkv = 2.0 * rows * d * (H + 2 * G) * dh
    rest = 2.0 * rows * (H * dh * d + 3 * F * d)
    attn = 4.0 * H * dh * float(np.sum(np.asarray(positions, np.float64) + 1))
    return L * qkv + (L - 1) * (rest + attn)


def other_workloads(kv, stream, llama) -> dict:
    """The other paper-shaped workloads, timed on the device (CUDA events,
    median of 3 after one warm-up call, repairs after three):
    - Qwen2.5-7B shape: select and repair for K in 8..128 under EditLocal,
      Random and Attention (selector time apart from the repair, as the paper
      reports it);
    - Mistral-7B shape: the Structural and CacheBlend selectors at K = 32;
    - 16 Llama-3-8B-shaped documents of 8192 tokens, 4 edits each with an
      EditLocal window of 32 after every span, in one batched repair call,
      against the 16 full re-prefills."""
    from paper_2609_17983_gb300 import synth
    out = {}
    tpeak, _ = load_tensor_peak()
    for name, pols in (("qwen7b", ("editlocal", "random", "attention")),
                       ("mistral7b", ("structural", "cacheblend"))):
        cfg = synth.preset(name)
        w = synth.workload(name)
        doc, s, new = w["doc"], w["edit_start"], w["new_tokens"]
        m = kv.Model(cfg, None, seed=0, max_context=8192, max_rows=4096)
        m.set_stream(stream.cuda_stream)
        cache = m.prefill(doc)
        res = {"edit": f"{len(new)}@{s}", "n": len(doc), "layers": cfg["n_layers"]}
        for pol in pols:
            res[pol] = {}
            for K in w["Ks"]:
                A = m.select(cache, pol, K, s, new, 0)
                sel = time_ms(lambda: m.select(cache, pol, K, s, new, 0), stream)
                # the first call launches kernel by kernel, the second captures the
                # pass as a graph: both belong to the warm-up
                rep = time_ms(lambda: cache.repair(new, s, A), stream, warm=3)
                rows = len(new) + len(A)
                res[pol][str(K)] = {"select_ms": sel, "repair_ms": rep, "rows": rows,
                                    "positions_per_s": rows / (rep / 1e3)}
        cache.close()
        m.close()
        out[name] = res
    # batched repair: 16 x 8192, 64 edits (span U[2, 16], window of 32 each)
    cfg = synth.preset(WORKLOAD)
    docs, reqs, P_all = [], [], []
    for d in range(16):
        doc = synth.document(100 + d, 8192, cfg["vocab"], cfg["delim_id"])
        edits, A, P = [], [], set()
        for (st, ln) in synth.batch_edits(200 + d, 8192, 4, (2, 16), K_BUDGET):
            new = synth.edit_tokens(300 + d * 7 + st, doc[st:st + ln], cfg["vocab"])
            edits.append((st, new))
            A += list(range(st + ln, st + ln + K_BUDGET))
            P |= set(range(st, st + ln + K_BUDGET))
        docs.append(doc)
        reqs.append((edits, np.array(sorted(set(A)))))
        P_all += sorted(P)
    caches = [llama.prefill(doc) for doc in docs]
    batch = [(c, e, A) for c, (e, A) in zip(caches, reqs)]
    b_ms = time_ms(lambda: llama.repair_batch(batch), stream)
    for c in caches:
        c.close()
    edited = []
    for doc, (edits, _) in zip(docs, reqs):
        t = doc.copy()
        for st, new in edits:
            t[st:st + len(new)] = new
        edited.append(t)
    p_ms = time_ms(lambda: [llama.prefill(t).close() for t in edited], stream, reps=1)
    fl = pass_flops(cfg, P_all)
    out["batch_16x8192"] = {"docs": 16, "n": 8192, "edits": 64, "rows": len(P_all),
                            "repair_ms": b_ms, "positions_per_s": len(P_all) / (b_ms / 1e3),
                            "prefill_16_ms": p_ms, "speedup_vs_prefill": p_ms / b_ms,
                            "flops": fl, "tflops": fl / (b_ms / 1e3) / 1e12,
                            "frac_of_bf16_sustained": fl / (b_ms / 1e3) / 1e12 / tpeak}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="kvrepair", choices=["kvrepair", "reference"])
    ap.add_argument("--prefill-steps", type=int, default=3)
    ap.add_argument("--oracle-layers", type=int, default=None,
                    help="most layers per oracle step of the reference arm")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-other-workloads", action="store_true",
                    help="skip the Qwen/Mistral/batched workloads (profiling runs)")
    ap.add_argument("--layers", type=int, default=None,
                    help="decoder layers (default: the model's 32); fewer only for profiling")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)

    from paper_2609_17983_gb300 import synth
    cfg = synth.preset(WORKLOAD)
    if args.layers:
        cfg["n_layers"] = args.layers
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))

    if args.impl == "reference":
        out = run_reference(args, cfg, rank)
        if out is not None:
            print(json.dumps(out), flush=True)
        return

    # the CPU baseline runs before any GPU work (no forked workers after CUDA init)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import oracle
        threads = oracle.set_threads(os.cpu_count() or 1)
        t_layer = oracle_time(oracle_setup(cfg, 1))
        # one step through as many of the model's first layers as take about
        # CPU_BASELINE_S
        layers = max(1, min(cfg["n_layers"], round(CPU_BASELINE_S / t_layer)))
        t = oracle_time(oracle_setup(cfg, layers)) if layers > 1 else t_layer
        M = EDIT_LEN + K_BUDGET
        cpu = {"value": oracle_value(cfg, layers, t), "unit": "positions/s",
               "cores": threads, "kind": "oracle", "step_s": t, "layers_per_step": layers,
               "sample": f"oracle operator R on the {M} rows through the first {layers} of "
                         f"{cfg['n_layers']} layers (one step; each layer its own seeded "
                         f"weights, seeded synthetic stale cache)"}

    import torch
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2609_17983_gb300 import kvrepair as kv

    # a stream of our own: the library captures the repair pass as a CUDA graph
    # (the legacy default stream cannot be captured)
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    # device memory from PyTorch's caching allocator, work on PyTorch's stream
    kv.use_torch_allocator()
    model = kv.Model(cfg, None, seed=0, max_context=8192, max_rows=4096)
    model.set_stream(stream.cuda_stream)
    doc, new = edit_inputs(cfg)
    cache = model.prefill(doc)
    model.synchronize()
    M = EDIT_LEN + K_BUDGET

    def step():
        A = model.select(cache, "editlocal", K_BUDGET, EDIT_START, new)
        cache.repair(new, EDIT_START, A)

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    for _ in range(args.warmup):
        step()
    barrier()
    l0 = model.launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with Clocks(local) as clk:
        ev0.record(stream)
        for _ in range(args.steps):
            step()
        ev1.record(stream)
        barrier()
    ms = max_over_ranks(ev0.elapsed_time(ev1) / args.steps, "cuda")
    launches = model.launches() - l0
    value = job_value(M, world, ms / 1e3)

    # per-kernel-class device time over the same steps (CUDA events on the stream)
    kv.kvr_profile_reset(model.h)
    kv.kvr_profile_enable(model.h, True)
    for _ in range(args.steps):
        step()
    model.synchronize()
    prof = kv.kvr_profile_read(model.h)
    kv.kvr_profile_enable(model.h, False)
    gemms = {k: v for k, v in prof.items() if k.startswith("gemm") and v["launches"]}
    dom = max(gemms, key=lambda k: gemms[k]["ms"])
    d = gemms[dom]
    peak, peak_kind = load_peaks()
    achieved = d["bytes"] / d["launches"] / (d["ms"] / d["launches"] / 1e3) / 1e9
    all_w = sum(v["bytes"] for v in gemms.values())
    traffic = (GU_TRAFFIC_BYTES if dom == "gemm_gu" and cfg["n_layers"] == 32
               and gemm_source_sha256() == GU_TRAFFIC_SOURCE_SHA256 else None)
    # the whole step against the HBM floor: the weights R needs once -- every
    # layer's QKV projection; attention output, O and MLP of all layers but
    # the last, whose outputs feed no K/V -- the keys and values of positions
    # 0 .. s_end + K - 1 read once per attending layer (the causal range),
    # the K/V of the |S| + K rows written at every layer
    es = 2
    d, F, L = cfg["d_model"], cfg["ffn"], cfg["n_layers"]
    H, G, dh = cfg["n_heads"], cfg["n_kv_heads"], cfg["head_dim"]
    qkv_w = (H + 2 * G) * dh * d * es
    rest_w = (d * H * dh + 2 * F * d + d * F) * es
    kv_read = (EDIT_START + EDIT_LEN + K_BUDGET) * (L - 1) * 2 * G * dh * es
    kv_write = M * L * 2 * G * dh * es
    pass_bytes = L * qkv_w + (L - 1) * rest_w + kv_read + kv_write
    pass_gbs = pass_bytes / (ms / 1e3) / 1e9
    all_ms = sum(v["ms"] for v in gemms.values())

    # e2e through the public API: host inputs in, the repaired rows' K/V out as
    # stored (bf16) into page-locked host buffers allocated once; the rows of
    # each layer group are copied out while the pass computes the next ones
    shape = (M, cfg["n_layers"], cfg["n_kv_heads"], cfg["head_dim"])
    k_rows = torch.empty(shape, dtype=torch.int16, pin_memory=True).numpy().view(np.uint16)
    v_rows = torch.empty(shape, dtype=torch.int16, pin_memory=True).numpy().view(np.uint16)
    barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        A = model.select(cache, "editlocal", K_BUDGET, EDIT_START, new)
        cache.repair_read(new, EDIT_START, A, k_out=k_rows, v_out=v_rows)
    barrier()
    e2e_s = max_over_ranks((time.perf_counter() - t0) / args.steps, "cuda")
    # what the two calls copy: kvr_select the new tokens in, the count, the
    # device flag and the K positions out; kvr_repair_read the new tokens and
    # the M positions of P in, the rows' K and V and the device flag out
    h2d = int(2 * new.nbytes + 4 * M)
    d2h = int(4 * (K_BUDGET + 2) + k_rows.nbytes + v_rows.nbytes + 4)

    # selector time, reported apart from the repair (the paper's protocol): each
    # policy on this cache, median of 3 after one warm-up; and the repair alone
    A_fixed = model.select(cache, "editlocal", K_BUDGET, EDIT_START, new)
    sel_ms = {}
    for pol in ("editlocal", "editlocal_boundary", "structural", "random", "attention",
                "cacheblend"):
        t = []
        for i in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            model.select(cache, pol, K_BUDGET, EDIT_START, new, 0)
            b.record(stream)
            torch.cuda.synchronize()
            if i:
                t.append(a.elapsed_time(b))
        sel_ms[pol] = statistics.median(t)
    t = []
    for i in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        cache.repair(new, EDIT_START, A_fixed)
        b.record(stream)
        torch.cuda.synchronize()
        if i:
            t.append(a.elapsed_time(b))
    repair_only_ms = statistics.median(t)

    # the baseline: full re-prefill of the edited document
    edited = doc.copy()
    edited[EDIT_START:EDIT_START + EDIT_LEN] = new
    pre = []
    for i in range(1 + args.prefill_steps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        c2 = model.prefill(edited)
        b.record(stream)
        torch.cuda.synchronize()
        c2.close()
        if i:
            pre.append(a.elapsed_time(b))
    prefill_ms = statistics.median(pre)
    tpeak, tpeak_kind = load_tensor_peak()
    pf_tflops = prefill_flops(cfg, N_CTX) / (prefill_ms / 1e3) / 1e12
    others = None
    if not args.no_other_workloads and cfg["n_layers"] == 32:
        others = other_workloads(kv, stream, model)

    if rank == 0:
        out = {"metric": METRIC, "value": value, "unit": "positions/s", "n_gpus": world,
               "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
               "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
               "dtype": "bf16", "data": "synthetic (seeded random-init weights and tokens)",
               "config": workload_config(cfg, world),
               "repair_ms": ms, "repair_only_ms": repair_only_ms, "select_ms": sel_ms,
               "prefill_ms": prefill_ms, "speedup_vs_prefill": prefill_ms / ms,
               "prefill_roofline": {"bound": "tensor", "flops": prefill_flops(cfg, N_CTX),
                                    "achieved": pf_tflops, "peak": tpeak, "unit": "TFLOP/s",
                                    "frac": pf_tflops / tpeak, "peak_kind": tpeak_kind + " sustained"},
               "token_layers_per_s": value * cfg["n_layers"],
               "gpu_launches": launches,
               "e2e": {"value": job_value(M, world, e2e_s), "unit": "positions/s",
                       "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
               "roofline": {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peak,
                            "unit": "GB/s", "frac": achieved / peak, "traffic": traffic,
                            "peak_kind": peak_kind,
                            "all_gemms_gbs": all_w / (all_ms / 1e3) / 1e9,
                            "pass": {"bytes": pass_bytes, "achieved_gbs": pass_gbs,
                                     "frac_of_measured": pass_gbs / peak,
                                     "frac_of_nominal_8tbs": pass_gbs / 8000.0}},
               # per kernel class, from events around every launch of an eager pass
               # (no graph; each class's PDL waits are inside its events, so the
               # classes sum to more than the step)
               "kernel_ms_per_step_eager": {k: v["ms"] / args.steps for k, v in prof.items()
                                            if v["launches"]},
               "clocks": clk.summary(),
               "other_workloads": others,
               "cpu_baseline": cpu}
        print(json.dumps(out), flush=True)
    cache.close()
    model.close()
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
