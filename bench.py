"""Throughput of the ACRL vocabulary-wide hot path on GB300.

One step = one on-policy pass of the whole path over one batch of the
Qwen-vocabulary workload (16 prompts x 8 responses, lengths U[256, 2048],
V = 151,936, bf16 logits, Student-t(4) x 2): token statistics, discrepancy
statistics, GRPO advantages, the controller and the loss gradient w.r.t. the
logits, all through the C ABI.  Inputs are generated on the device from fixed
seeds and are far larger than L2 (44.8 GB of logits), so no L2 flush is needed
between steps.

Prints one JSON line.  `--impl reference` times the float64 CPU oracle on a
bounded row sample of the same workload instead (rank 0 only).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""

from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import threading
import time

# The CPU oracle legs run one thread per process and report the processes as
# their cores: keep numpy's BLAS (the LM-head projection's matrix product) to
# one thread too.  Set before numpy is imported, which is when the BLAS library
# reads them (the oracle's worker processes inherit them).
for _v in ("OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import numpy as np  # noqa: E402

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "tokens/s fused logprob+discrepancy+grad at V=151936; HBM GB/s vs peak"
LMHEAD_METRIC = "tokens/s fused LM-head projection + logprob + discrepancy + grad at V=151936"
UNIT = "tokens/s"
FALLBACK_HBM_GBS = 6800.0
# Kernel launches per step inside the timed region: token_stats 1, seq_discrepancy 2,
# grpo_advantage 1, controller_step 3, loss_grad_logits 2.
LAUNCHES_PER_STEP = 9
# DRAM traffic of one launch of each kernel (dram__bytes_read.sum + dram__bytes_write.sum
# from ncu, one pass), captured on a small case of its workload and scaled to a full
# launch by the algorithmic bytes (or, for the GEMM, the flops) of each: the streaming
# kernels' traffic grows in proportion to the rows, the GEMM's to the bands of 32 row
# tiles (the weight is read once per band).  Valid only for the kernel source it was
# taken on (sha256 of the code, comments left out, of the file and the headers beside it; 16 hex digits).
NCU_TRAFFIC = {
    # qwen_profile (8,192 rows x 151,936), the two timed launches averaged
    "loss_grad.cu": {"src": "3cf528e15f6c625e", "bytes": 2.48948e9 + 2.43282e9, "units": 4978778112},
    "token_stats.cu": {"src": "94cd212729153580", "bytes": 2.48999e9 + 1.78e6, "units": 2489458688},
    # lmhead_profile (4,096 x 4,096 x 151,936: one band), two launches averaged, flops as the unit
    "lmhead.cu": {"src": "4e28862dd431d57b", "bytes": 2.0298e9 + 1.2914e9, "units": 2.0 * 4096 * 151936 * 4096},
}


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def _code_only(text):
    """C/C++ source without its comments, blank lines and trailing blanks."""
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"//[^\n]*", "", text)
    return "\n".join(line.rstrip() for line in text.splitlines() if line.strip())


def _src_hash(name):
    """Hash of the code of a kernel source and of every header beside it
    (comments left out: editing one does not change the kernel)."""
    csrc = os.path.join(ROOT, "paper_2607_24062_gb300", "csrc")
    headers = sorted(f for f in os.listdir(csrc) if f.endswith((".cuh", ".h")))
    d = hashlib.sha256()
    for f in (name, *headers):
        with open(os.path.join(csrc, f), encoding="utf-8") as fh:
            d.update(_code_only(fh.read()).encode())
    return d.hexdigest()[:16]


TRAFFIC_SOURCE = ("ncu dram__bytes_read.sum + dram__bytes_write.sum on a small case (qwen_profile, 8,192 rows; "
                  "lmhead_profile, 4,096 rows) scaled by algorithmic bytes (flops for the GEMM)")


def _traffic_of(name, units):
    """ncu DRAM bytes per launch of a kernel source scaled to a launch of `units`
    algorithmic bytes (flops for the GEMM), if taken on the source as it is now."""
    tr = NCU_TRAFFIC.get(name)
    return tr["bytes"] * units / tr["units"] if tr and tr["src"] == _src_hash(name) else None


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []
        self.thread = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-i", str(self.index), "-lms", "100"], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            if self.thread is not None:
                self.thread.join(timeout=2)

    def summary(self):
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        sm, mx, reasons = [], [], set()
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) != 6:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for n, v in zip(names, parts[2:]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def _dist():
    import torch
    import torch.distributed as dist
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1 and not dist.is_initialized():
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    return world, rank, local


def _lmhead_spec(W, name):
    return W.LMHEAD if name == "lmhead" else W.small_variant(W.LMHEAD, name="lmhead_profile", n_prompts=2)


def _lmhead_desc(b):
    return (f"lmhead: hidden bf16 [{b.T}, {b.K}] ~N(0,1), weight bf16 [{b.N}, {b.K}] ~N(0, 0.02^2), "
            "mu from E4M3 per-token/per-channel copies")


def _logits_config(spec, batch, world):
    """`config` of a logits workload's line; both arms print the same one."""
    return {"workload": _workload_desc(spec), "T": batch.T, "V": batch.V, "ld": batch.ld,
            "tokens_per_step": int(batch.mask.sum()), "logits": "bf16 in, gradient bf16 out, fp32 arithmetic",
            "l2": f"no flush: inputs ({batch.T * batch.ld * 2 / 1e9:.1f} GB of logits) far larger than the 129 MB L2",
            "parallelism": f"data-parallel over prompts, {world} rank(s); 3-scalar all-reduce per step"}


def _lmhead_config(b):
    """`config` of the LM-head workload's line; both arms print the same one."""
    return {"workload": _lmhead_desc(b), "M": b.T, "N": b.N, "K": b.K, "tokens_per_step": int(b.mask.sum())}


def _workload_desc(spec):
    return (f"{spec.name}: {spec.n_prompts} prompts x {spec.group_size} responses, lengths U[{spec.len_lo},"
            f"{spec.len_hi}], V={spec.V}, bf16 logits {spec.dist}(scale {spec.scale}), mu = FP8-E4M3 "
            f"{spec.fp8_scale}-scaled round-trip")


# --------------------------------------------------------------------------
# CPU oracle leg
# --------------------------------------------------------------------------

def _oracle_params(params):
    import oracle as O
    return O.Params(gamma=params.gamma, C=params.C, clip_eps=params.clip_eps, adv_eps=params.adv_eps)


def _oracle_rows(O, z, ids, mask, op):
    """The oracle's vocabulary-wide stages on a block of rows: statistics, then
    the gradient with a representative weight and advantage."""
    lse, logp, H, _ = O.token_stats(z, ids, mask)
    r = len(ids)
    O.loss_grad_logits(z, ids, mask, lse, None, np.ones(r), np.ones(r), np.arange(r + 1),
                       {"n": np.ones(r, dtype=np.int64), "group": np.zeros(r, dtype=np.int64)},
                       {"n_valid_seqs": np.array([r])}, {"n_groups_valid": 1, "n_tokens": r}, op)


def _oracle_ot_seconds(O, batch, op):
    """The oracle's O(T) stages over the whole batch; the rollout log-probs stand
    in for pi's (same cost)."""
    mask = batch.mask.cpu().numpy()
    mu = batch.logp_mu.cpu().numpy().astype(np.float64)
    R = batch.rewards.cpu().numpy().astype(np.float64)
    so = batch.seq_offsets.cpu().numpy()
    go = batch.group_offsets.cpu().numpy()
    tc = time.perf_counter()
    lr, d, seq, grp, bst, _ = O.seq_discrepancy(mu, mu, mask, so, go)
    adv = O.grpo_advantage(R, go, op)
    w, alpha, st, info, _ = O.controller_step(O.controller_init(op), op, lr, mask, so, go, seq, grp, bst, adv)
    O.loss_coefficients(w, adv, mask, so, seq, grp, bst, op)
    return time.perf_counter() - tc


def _bf16_rows_f64(O, t, rows, cols):
    import torch
    idx = torch.as_tensor(rows, device=t.device)
    bits = t.index_select(0, idx)[:, :cols].contiguous().view(torch.int16).cpu().numpy().view(np.uint16)
    return O.bf16_bits_to_f64(bits)


_POOL = None


def _cpu_model():
    """The host CPU's model name (lscpu), or the machine type."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.startswith("Model name:"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    import platform
    return platform.machine()


def _oracle_pool():
    """Worker processes for the oracle's row blocks, one per host core the
    process may run on (spawned, so they never inherit a CUDA context), all
    started and warm before any timing."""
    global _POOL
    if _POOL is None:
        import atexit
        import concurrent.futures
        import multiprocessing
        n = max(1, min(len(os.sched_getaffinity(0)), 32))
        _POOL = (concurrent.futures.ProcessPoolExecutor(max_workers=n,
                                                        mp_context=multiprocessing.get_context("spawn")), n)
        list(_POOL[0].map(_oracle_worker_ready, [0.2] * n))
        atexit.register(_POOL[0].shutdown)
    return _POOL


def _oracle_worker_ready(pause):
    import oracle  # noqa: F401
    time.sleep(pause)  # hold this worker so that the others take the remaining start-up tasks
    return os.getpid()


def _oracle_rows_block(bits, ids, mask, op):
    import oracle as O
    _oracle_rows(O, O.bf16_bits_to_f64(bits), ids, mask, op)
    return len(ids)


def _bf16_rows_bits(t, rows, cols):
    import torch
    idx = torch.as_tensor(rows, device=t.device)
    return t.index_select(0, idx)[:, :cols].contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def _oracle_rows_parallel(batch, rows, ids, mask, op, budget_s, block=16):
    """The oracle's vocabulary-wide stages on `rows`, in blocks spread over the
    worker processes, until `budget_s` of wall time has passed.  Returns
    (wall seconds, rows done, processes)."""
    pool, n = _oracle_pool()
    t0 = time.perf_counter()
    pending, done, k = set(), 0, 0
    while k < len(rows) or pending:
        while k < len(rows) and len(pending) < 2 * n and time.perf_counter() - t0 < budget_s:
            rr = rows[k:k + block]
            pending.add(pool.submit(_oracle_rows_block, _bf16_rows_bits(batch.logits, rr, batch.V), ids[rr],
                                    mask[rr], op))
            k += len(rr)
        if not pending:
            break
        finished = {f for f in pending if f.done()}
        if not finished:
            import concurrent.futures
            finished, _ = concurrent.futures.wait(pending, return_when=concurrent.futures.FIRST_COMPLETED)
        for f in finished:
            done += f.result()
        pending -= finished
        if time.perf_counter() - t0 >= budget_s:
            k = len(rows)  # submit nothing more; let the blocks in flight finish
    return time.perf_counter() - t0, done, n


def oracle_tokens_per_s(batch, params, rows_budget_s=10.0, max_rows=4096, rng_seed=0, lmhead=False):
    """Time the float64 oracle on a bounded sample: the O(T) stages over the
    whole batch once, the vocabulary-wide stages (for the LM-head workload the
    projection first, then log-softmax statistics and the gradient) on sampled
    rows until `rows_budget_s` has passed.  The logits workloads spread row
    blocks over one process per host core; the LM-head workload (whose
    float64 weight copy is 5 GB) runs in this process on one core.  Returns
    (tokens/s extrapolated to the whole batch, description, rows done, cores)."""
    import oracle as O

    op = _oracle_params(params)
    mask = batch.mask.cpu().numpy()
    ids = batch.ids.cpu().numpy()
    rng = np.random.default_rng(rng_seed)
    rows = rng.permutation(np.flatnonzero(mask))[:max_rows]
    if not lmhead:
        t_rows, done, cores = _oracle_rows_parallel(batch, rows, ids, mask, op, rows_budget_s)
        t_ot = _oracle_ot_seconds(O, batch, op)
        n_valid = int(mask.sum())
        per_token = t_rows / max(1, done) + t_ot / max(1, n_valid)
        desc = (f"float64 numpy oracle, {cores} processes (one per host core, one thread each): log-softmax "
                f"statistics + gradient on {done} sampled rows ({t_rows:.1f} s wall) and, in one process, the O(T) "
                f"stages on all {n_valid} tokens ({t_ot:.1f} s), extrapolated per token")
        return 1.0 / per_token, desc, done, cores
    # the LM-head workload: the weight's float64 copy is set-up (a model load), not timed
    W64 = _bf16_rows_f64(O, batch.weight, np.arange(batch.N), batch.K)
    t0 = time.perf_counter()
    done = 0
    t_rows = 0.0
    while done < len(rows) and time.perf_counter() - t0 < rows_budget_s:
        rr = rows[done:done + 4]
        h = _bf16_rows_f64(O, batch.hidden, rr, batch.K)
        tc = time.perf_counter()
        _oracle_rows(O, O.lmhead_logits(h, W64), ids[rr], mask[rr], op)
        t_rows += time.perf_counter() - tc
        done += len(rr)
    t_ot = _oracle_ot_seconds(O, batch, op)
    n_valid = int(mask.sum())
    per_token = t_rows / max(1, done) + t_ot / max(1, n_valid)
    desc = (f"float64 numpy oracle, 1 thread: LM-head projection + log-softmax statistics + gradient on {done} "
            f"sampled rows ({t_rows:.1f} s) and the O(T) stages on all {n_valid} tokens ({t_ot:.1f} s), "
            "extrapolated per token")
    return 1.0 / per_token, desc, done, 1


def run_reference(args):
    world, rank, local = _dist()
    if rank != 0:
        return 0
    import torch

    import paper_2607_24062_gb300 as acrl
    import workloads as W
    lmhead = args.workload in ("lmhead", "lmhead_profile")
    dev = torch.device(f"cuda:{local}" if torch.cuda.is_available() else "cpu")
    if dev.type == "cuda":
        torch.cuda.set_device(dev)
    if lmhead:
        spec = _lmhead_spec(W, args.workload)
        batch = W.generate_lmhead(spec, device=dev)
        config = _lmhead_config(batch)
    else:
        spec = W.SPECS[args.workload]
        batch = W.generate(spec, seed=W.seed_for(spec.name), device=dev)
        config = _logits_config(spec, batch, world)
    params = acrl.Params()
    vals = []
    t_all = []
    # each step's row sample is time-boxed so that the whole run stays within about three minutes
    budget = min(args.ref_seconds, max(1.0, 150.0 / max(1, args.warmup + args.steps)))
    for k in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        v, desc, n, cores = oracle_tokens_per_s(batch, params, rows_budget_s=budget, max_rows=4096, rng_seed=k,
                                                lmhead=lmhead)
        t_all.append(time.perf_counter() - t0)
        if k >= args.warmup:
            vals.append(v)
    value = float(np.median(vals))
    out = {"impl": "reference", "metric": LMHEAD_METRIC if lmhead else METRIC, "value": value, "unit": UNIT,
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": float(np.median(t_all[args.warmup:])) * 1e3,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": config,
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc,
                            "cpu": _cpu_model()},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out))
    return 0


# --------------------------------------------------------------------------
# our arm
# --------------------------------------------------------------------------

def run_ours(args):
    import torch
    import torch.distributed as dist

    import paper_2607_24062_gb300 as acrl
    import workloads as W
    from paper_2607_24062_gb300 import build

    world, rank, local = _dist()
    build.build()
    dev = torch.device(f"cuda:{local}")
    torch.cuda.set_device(dev)
    spec = W.SPECS[args.workload]
    # weak scaling: each rank owns its own batch of prompts; the ranks sum three scalars of the batch statistics
    # before the controller (one global X and the global loss normalisation), the path's only exchange
    from paper_2607_24062_gb300 import distributed as D
    batch = W.generate(spec, seed=D.shard_seed(W.seed_for(spec.name), rank), device=dev)
    params = acrl.Params()
    step = acrl.AcrlStep.for_batch(batch, params, device=dev)
    stream = torch.cuda.current_stream(dev)
    exchange = D.allreduce_batch_stats if world > 1 else None

    for _ in range(args.warmup):
        step.run_batch(batch, exchange=exchange)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()

    n_valid = int(batch.mask.sum())
    mask_h = batch.mask.bool().cpu()
    coef_h = step.coef.cpu()
    ids_h = batch.ids.cpu()
    live = mask_h & (coef_h != 0) & (ids_h >= 0) & (ids_h < batch.V)
    V = batch.V
    # algorithmic bytes per launch
    k5_bytes = int(live.sum()) * 4 * V + (batch.T - int(live.sum())) * 2 * V + batch.T * 17
    k1_bytes = n_valid * 2 * V + batch.T * 17

    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True),
           torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    start = torch.cuda.Event(enable_timing=True)
    end = torch.cuda.Event(enable_timing=True)
    with ClockSampler(dev.index) as clocks:
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        start.record(stream)
        for k in range(args.steps):
            e0, e1, e2, e3 = ev[k]
            e0.record(stream)
            acrl.token_stats(batch.logits, batch.ids, batch.mask, V=V, lse=step.lse, logp=step.logp,
                             entropy=step.entropy, flags=step.flags)
            e1.record(stream)
            # the rest of the statistics pass (seq_discrepancy, grpo_advantage, controller_step)
            acrl.seq_discrepancy(step.logp, batch.logp_mu, batch.mask, batch.seq_offsets, batch.group_offsets,
                                 step.entropy, out=step.disc, flags=step.flags)
            if exchange is not None:
                exchange(step.disc.batch)
            acrl.grpo_advantage(batch.rewards, batch.group_offsets, params, adv=step.adv, flags=step.flags)
            acrl.controller_step(step.state, params, step.disc, batch.mask, batch.seq_offsets, batch.group_offsets,
                                 step.adv, weight=step.weight, coef=step.coef, alpha=step.alpha, flags=step.flags)
            e2.record(stream)
            acrl.loss_grad_logits(batch.logits, batch.ids, batch.mask, step.lse, None, step.coef, params.clip_eps,
                                  V=V, grad=step.grad, token_loss=step.token_loss, loss=step.loss, flags=step.flags)
            e3.record(stream)
        end.record(stream)
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
    total_ms = start.elapsed_time(end)
    if world > 1:
        t = torch.tensor([total_ms], device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t)
        nt = torch.tensor([n_valid], device=dev, dtype=torch.float64)
        dist.all_reduce(nt)
        tokens_all = float(nt)
    else:
        tokens_all = float(n_valid)
    # cached-old variant: the gradient call recomputes each row's LSE itself (a second sweep over the row);
    # the weights would come from cached old log-probs, here the statistics pass's own
    def cached_old():
        acrl.loss_grad_logits(batch.logits, batch.ids, batch.mask, None, step.logp, step.coef, params.clip_eps,
                              V=V, grad=step.grad, token_loss=step.token_loss, loss=step.loss, flags=step.flags)

    # entropy-bonus variant (App. A's entropy coefficient): every valid row carries a bonus coefficient
    ent_coef = batch.mask.float() * 1e-6

    def entropy_bonus():
        acrl.loss_grad_logits(batch.logits, batch.ids, batch.mask, step.lse, None, step.coef, params.clip_eps,
                              V=V, entropy=step.entropy, ent_coef=ent_coef, grad=step.grad,
                              token_loss=step.token_loss, loss=step.loss, flags=step.flags)

    def median_ms(fn, n):
        fn()                # a kernel's first launch also loads it: keep that out of the timing
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n)]
        for a, b in evs:
            a.record(stream)
            fn()
            b.record(stream)
        torch.cuda.synchronize()
        return float(np.median([a.elapsed_time(b) for a, b in evs]))

    co_ms = median_ms(cached_old, min(5, args.steps))
    weights_sec54 = _weight_calls_ms(acrl, W, dev, median_ms) if rank == 0 else None
    eb_ms = median_ms(entropy_bonus, min(5, args.steps))
    live_e = mask_h & (ids_h >= 0) & (ids_h < batch.V)
    eb_bytes = int(live_e.sum()) * 4 * V + (batch.T - int(live_e.sum())) * 2 * V + batch.T * 25
    k1_ms = [ev[k][0].elapsed_time(ev[k][1]) for k in range(args.steps)]
    mid_ms = [ev[k][1].elapsed_time(ev[k][2]) for k in range(args.steps)]
    k5_ms = [ev[k][2].elapsed_time(ev[k][3]) for k in range(args.steps)]
    ms_per_step = total_ms / args.steps
    value = tokens_all * args.steps / (total_ms / 1e3)

    peak, peak_kind = _peaks()
    k5_avg = float(np.mean(k5_ms))
    k1_avg = float(np.mean(k1_ms))
    k5_gbs = k5_bytes / (k5_avg / 1e3) / 1e9
    k1_gbs = k1_bytes / (k1_avg / 1e3) / 1e9
    traffic = _traffic_of("loss_grad.cu", k5_bytes)

    # the same step replayed from a CUDA graph (launch gaps removed); reported beside the eager step
    # (single process only: the multi-rank step keeps its collective outside any graph)
    graph_ms = None
    if world == 1:
        graph = step.capture(batch)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        for _ in range(args.steps):
            graph.replay()
        g1.record(stream)
        torch.cuda.synchronize()
        graph_ms = g0.elapsed_time(g1) / args.steps
        del graph

    # end to end through host buffers: on rank 0 only (each rank would page-lock 90 GB of host memory)
    e2e = None
    if not args.no_e2e and rank == 0:
        e2e = run_e2e(batch, step, params, args, dev)
        if world > 1 and e2e is not None:
            e2e["ranks_measured"] = 1
            e2e["note"] = ("rank 0 alone, the other ranks idle: one GPU's host link, not the whole job; the host "
                           "pipeline has no rank exchange, so its weights use rank 0's batch statistics and its "
                           "gradient is not compared with the exchanged step's")
            e2e["download_matches_device"] = None
    if world > 1:
        dist.barrier()
    if rank != 0:
        return 0
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": _logits_config(spec, batch, world),
        "roofline": {"bound": "hbm", "kernel": "acrl_loss_grad_logits", "achieved": k5_gbs, "peak": peak,
                     "unit": "GB/s", "frac": k5_gbs / peak, "traffic": traffic, "peak_kind": peak_kind,
                     "traffic_source": TRAFFIC_SOURCE, "algorithmic_bytes_per_launch": k5_bytes,
                     "ms_per_launch": k5_avg},
        "kernels": {
            "acrl_token_stats": {"ms": k1_avg, "GB/s": k1_gbs, "frac": k1_gbs / peak, "bytes": k1_bytes,
                                 "traffic": _traffic_of("token_stats.cu", k1_bytes)},
            "acrl_loss_grad_logits": {"ms": k5_avg, "GB/s": k5_gbs, "frac": k5_gbs / peak, "bytes": k5_bytes},
            "seq_discrepancy+grpo_advantage+controller_step": {"ms": float(np.mean(mid_ms))},
            "acrl_loss_grad_logits (lse recomputed, cached-old)": {
                "ms": co_ms, "GB/s": k5_bytes / (co_ms / 1e3) / 1e9, "frac": k5_bytes / (co_ms / 1e3) / 1e9 / peak,
                "note": "algorithmic bytes as the streaming call (4 B per element of a live row)"},
            "acrl_loss_grad_logits (entropy bonus)": {
                "ms": eb_ms, "GB/s": eb_bytes / (eb_ms / 1e3) / 1e9, "frac": eb_bytes / (eb_ms / 1e3) / 1e9 / peak,
                "bytes": eb_bytes},
            "weight calls on the Sec. 5.4 batch shape": weights_sec54,
            "whole_step_GB/s": (k1_bytes + k5_bytes) / (ms_per_step / 1e3) / 1e9,
            "step_replayed_from_cuda_graph": ({"ms": graph_ms, "tokens/s": n_valid / (graph_ms / 1e3)}
                                              if graph_ms else None),
        },
        "clocks": clocks.summary(),
        "gpu_launches": LAUNCHES_PER_STEP * args.steps,
    }
    if e2e is not None:
        out["e2e"] = e2e
    if not args.no_cpu and world == 1:
        v, desc, n, cores = oracle_tokens_per_s(batch, params, rows_budget_s=args.ref_seconds, max_rows=16384)
        out["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc,
                               "cpu": _cpu_model()}
    if not args.no_lmhead and world == 1:
        # The fused LM-head workload (hidden 32,768 x 4,096, weight 151,936 x 4,096) in the same process, once
        # the Qwen batch's buffers are released: its own K steps after W warm-up steps, its own clock record.
        # Reported beside the step above; the line's value, timing and launch count are the Qwen step's.
        import gc
        del step, batch, ent_coef
        gc.collect()
        torch.cuda.empty_cache()
        lm, _, _ = lmhead_measure("lmhead", dev, args.steps, args.warmup)
        out["kernels"]["lmhead_step (fused LM-head workload)"] = lm
    print(json.dumps(out))
    return 0


def _weight_calls_ms(acrl, W, dev, median_ms):
    """The three calls that make the importance weights from per-token
    log-probs (seq_discrepancy, grpo_advantage, controller_step) on a batch of
    the shape of the paper's overhead measurement (64 prompts x 8 responses,
    lengths U[1, 2048]); the paper reports 0.059 s for its call on that
    setting, hardware not stated."""
    spec = W.WEIGHTS_SEC54
    d = W.token_level(spec, W.seed_for(spec.name), device=dev)
    p = acrl.Params()
    state = acrl.controller_init(p, device=dev)
    flags = acrl.api.new_flags(dev)

    def calls():
        acrl.importance_weights(state, p, d["logp_pi"], d["logp_mu"], d["mask"], d["rewards"], d["seq_offsets"],
                                d["group_offsets"], flags=flags)

    ms = median_ms(calls, 20)
    return {"ms": ms, "tokens": int(d["mask"].sum()), "rows": d["T"], "flags": acrl.read_flags(flags),
            "workload": W.describe(spec) + ", token-level log-probs only",
            "note": "includes the output allocations of the Python calls; the paper's 0.059 s is context only"}


def _tensor_peaks():
    """Measured bf16 tensor throughput (TFLOP/s): (burst, sustained, kind)."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["bf16_tflops"]), float(d["bf16_tflops_sustained"]), "measured"
    except Exception:
        return 1900.0, 1700.0, "fallback"


def lmhead_measure(workload, dev, steps, warmup):
    """Time the fused LM-head workload (32,768 tokens x 4,096 hidden x 151,936
    vocabulary for "lmhead"): a step is the GEMM with the statistics epilogue,
    the merge, the O(T) stages and the gradient on the stored bf16 logits,
    every call through the C ABI.  Returns (summary dict, batch, params)."""
    import torch

    import paper_2607_24062_gb300 as acrl
    import workloads as W

    b = W.generate_lmhead(_lmhead_spec(W, workload), device=dev)
    p = acrl.Params()
    M, N, K = b.T, b.N, b.K
    stream = torch.cuda.current_stream(dev)
    flags = acrl.api.new_flags(dev)
    ldl = ((N + 7) // 8) * 8
    logits = torch.empty((M, ldl), dtype=torch.bfloat16, device=dev)
    partials = torch.empty(acrl.api.lmhead_workspace_bytes(M, N) // 4, dtype=torch.float32, device=dev)
    f32 = dict(dtype=torch.float32, device=dev)
    lse, logp, ent = torch.empty(M, **f32), torch.empty(M, **f32), torch.empty(M, **f32)
    grad = torch.empty((M, ldl), dtype=torch.bfloat16, device=dev)
    state = acrl.controller_init(p, device=dev)

    def one(ev=None):
        if ev:
            ev[0].record(stream)
        acrl.api.lmhead_logits_stats(b.hidden, b.weight, N=N, logits=logits, partials=partials, flags=flags)
        if ev:
            ev[1].record(stream)
        acrl.api.lmhead_merge(partials, logits, b.ids, b.mask, N=N, lse=lse, logp=logp, entropy=ent, flags=flags)
        if ev:
            ev[2].record(stream)
        disc = acrl.seq_discrepancy(logp, b.logp_mu, b.mask, b.seq_offsets, b.group_offsets, ent, flags=flags)
        adv = acrl.grpo_advantage(b.rewards, b.group_offsets, p, flags=flags)
        w, coef, alpha = acrl.controller_step(state, p, disc, b.mask, b.seq_offsets, b.group_offsets, adv,
                                              flags=flags)
        if ev:
            ev[3].record(stream)
        acrl.loss_grad_logits(logits, b.ids, b.mask, lse, None, coef, p.clip_eps, V=N, grad=grad, flags=flags)
        if ev:
            ev[4].record(stream)

    for _ in range(warmup):
        one()
    torch.cuda.synchronize()
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(5)] for _ in range(steps)]
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(dev.index) as clocks:
        torch.cuda.synchronize()
        t0.record(stream)
        for k in range(steps):
            one(evs[k])
        t1.record(stream)
        torch.cuda.synchronize()
    fl = acrl.read_flags(flags)
    total_ms = t0.elapsed_time(t1)
    gemm_ms = float(np.mean([e[0].elapsed_time(e[1]) for e in evs]))
    merge_ms = float(np.mean([e[1].elapsed_time(e[2]) for e in evs]))
    ot_ms = float(np.mean([e[2].elapsed_time(e[3]) for e in evs]))
    grad_ms = float(np.mean([e[3].elapsed_time(e[4]) for e in evs]))
    flop = 2.0 * M * N * K
    tf = flop / (gemm_ms / 1e3) / 1e12
    burst, sustained, kind = _tensor_peaks()
    n_valid = int(b.mask.sum())
    ms_step = total_ms / steps
    summary = {
        "workload": _lmhead_desc(b), "M": M, "N": N, "K": K, "steps": steps, "warmup": warmup, "flags": fl,
        "ms_per_step": ms_step, "tokens/s": n_valid / (ms_step / 1e3), "tokens_per_step": n_valid,
        "gemm": {"kernel": "acrl_lmhead_logits_stats", "ms": gemm_ms, "TFLOP/s": tf, "flop_per_launch": flop,
                 "frac_burst": tf / burst, "frac_sustained": tf / sustained, "peak_burst": burst,
                 "peak_sustained": sustained, "peak_kind": kind, "traffic": _traffic_of("lmhead.cu", flop),
                 "traffic_source": TRAFFIC_SOURCE},
        "merge_ms": merge_ms, "seq_discrepancy+grpo_advantage+controller_step_ms": ot_ms,
        "loss_grad_logits": {"ms": grad_ms, "GB/s": 4.0 * M * N / (grad_ms / 1e3) / 1e9},
        "clocks": clocks.summary(), "gpu_launches": 10 * steps,
    }
    return summary, b, p


def run_lmhead(args):
    """The fused LM-head workload on its own line (`--workload lmhead` or
    `lmhead_profile`)."""
    import torch

    from paper_2607_24062_gb300 import build

    world, rank, local = _dist()
    build.build()
    dev = torch.device(f"cuda:{local}")
    torch.cuda.set_device(dev)
    lm, b, p = lmhead_measure(args.workload, dev, args.steps, args.warmup)
    g = lm["gemm"]
    out = {"metric": LMHEAD_METRIC,
           "value": lm["tokens/s"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": lm["ms_per_step"], "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "bf16 (tensor cores, fp32 accumulate)", "data": "synthetic",
           "config": _lmhead_config(b), "device_flags": lm["flags"],
           "roofline": {"bound": "tensor", "kernel": g["kernel"], "achieved": g["TFLOP/s"],
                        "peak": g["peak_sustained"], "unit": "TFLOP/s", "frac": g["frac_sustained"],
                        "frac_burst": g["frac_burst"], "peak_burst": g["peak_burst"],
                        "traffic": _traffic_of("lmhead.cu", g["flop_per_launch"]),
                        "peak_kind": g["peak_kind"] + " (sustained)", "flop_per_launch": g["flop_per_launch"],
                        "ms_per_launch": g["ms"]},
           "kernels": {"acrl_lmhead_logits_stats": {"ms": g["ms"], "TFLOP/s": g["TFLOP/s"]},
                       "acrl_lmhead_merge": {"ms": lm["merge_ms"]},
                       "acrl_loss_grad_logits": lm["loss_grad_logits"]},
           "clocks": lm["clocks"], "gpu_launches": lm["gpu_launches"]}
    if not args.no_cpu:
        v, desc, _, cores = oracle_tokens_per_s(b, p, rows_budget_s=args.ref_seconds, lmhead=True)
        out["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc,
                               "cpu": _cpu_model()}
    print(json.dumps(out))
    return 0


class _PinnedHost:
    """Page-locked host arrays for the end-to-end run.  First choice: driver
    allocations of exactly the requested size (cuMemHostAlloc), which move at
    the link rate whatever the page size.  If that fails: ordinary memory
    advised onto transparent huge pages before first touch and registered in
    place (fast only when the kernel finds huge pages for it)."""

    def __init__(self):
        import ctypes
        self.ctypes = ctypes
        self.allocs = []        # cuMemHostAlloc pointers
        self.registered = []    # registered numpy arrays
        self.kind = None
        try:
            self.cuda = ctypes.CDLL("libcuda.so.1")
        except OSError:
            self.cuda = None

    def empty(self, shape, dtype):
        import torch
        ct = self.ctypes
        nbytes = int(np.prod(shape)) * np.dtype(dtype).itemsize
        if self.cuda is not None and self.kind != "registered":
            p = ct.c_void_p()
            if self.cuda.cuMemHostAlloc(ct.byref(p), ct.c_size_t(nbytes), ct.c_uint(0)) == 0 and p.value:
                self.allocs.append(p)
                self.kind = "cuMemHostAlloc"
                buf = (ct.c_uint8 * nbytes).from_address(p.value)
                return np.frombuffer(buf, dtype=dtype).reshape(shape)
        if self.kind == "cuMemHostAlloc":
            raise RuntimeError("cuMemHostAlloc failed for the second buffer")
        arr = _huge_empty(shape, dtype)
        if int(torch.cuda.cudart().cudaHostRegister(arr.ctypes.data, arr.nbytes, 0)) != 0:
            raise RuntimeError("cudaHostRegister failed")
        self.registered.append(arr)
        self.kind = "registered"
        return arr

    def describe(self):
        return ("user buffers from cuMemHostAlloc (page-locked by the driver)" if self.kind == "cuMemHostAlloc" else
                "user buffers page-locked in place with cudaHostRegister (advised onto huge pages)")

    def free(self):
        import torch
        torch.cuda.synchronize()
        for p in self.allocs:
            self.cuda.cuMemFreeHost(p)
        for arr in self.registered:
            torch.cuda.cudart().cudaHostUnregister(arr.ctypes.data)
        self.allocs, self.registered = [], []


def _huge_empty(shape, dtype):
    """np.empty whose pages are advised as transparent huge pages (Linux), before any page is touched."""
    import ctypes
    arr = np.empty(shape, dtype=dtype)
    try:
        libc = ctypes.CDLL("libc.so.6")
        page = os.sysconf("SC_PAGE_SIZE")
        start = arr.ctypes.data & ~(page - 1)
        libc.madvise(ctypes.c_void_p(start), ctypes.c_size_t(arr.nbytes + arr.ctypes.data - start), 14)
    except Exception:
        pass
    return arr


def _host_available_bytes():
    """MemAvailable of the host (Linux), or None."""
    try:
        with open("/proc/meminfo") as f:
            for line in f:
                if line.startswith("MemAvailable:"):
                    return int(line.split()[1]) * 1024
    except OSError:
        pass
    return None


def run_e2e(batch, step, params, args, dev):
    """Same metric through the C ABI with the user's buffers in host memory:
    one acrl_host_pipeline_step call per step, which uploads that step's
    inputs from page-locked host memory in row chunks, runs the whole path and
    downloads the gradient and the loss chunk by chunk on the library's own
    copy streams (consecutive steps overlap)."""
    import torch

    import paper_2607_24062_gb300 as acrl
    T, ld = batch.logits.shape
    V = batch.V
    # The user's host arrays, page-locked and of exactly their size (torch's pinned allocator would round 44.8 GB
    # up to 64 GB).  Page-locking most of the host's memory could starve it, so leave a margin.
    need = 2 * T * ld * 2
    avail = _host_available_bytes()
    if avail is not None and need + (32 << 30) > avail:
        return {"value": None, "unit": UNIT,
                "error": f"skipped: {need / 1e9:.1f} GB of page-locked buffers with {avail / 1e9:.1f} GB available"}
    pinned = _PinnedHost()
    hp = None
    try:
        try:
            h_logits_np = pinned.empty((T, ld), np.uint16)
            h_grad_np = pinned.empty((T, ld), np.uint16)
        except RuntimeError as e:
            return {"value": None, "unit": UNIT, "error": str(e)}
        h_logits = torch.from_numpy(h_logits_np).view(torch.bfloat16)
        h_grad = torch.from_numpy(h_grad_np).view(torch.bfloat16)
        h_logits.copy_(batch.logits)
        small_h = {k: getattr(batch, k).cpu().pin_memory()
                   for k in ("ids", "mask", "logp_mu", "rewards", "seq_offsets", "group_offsets")}
        loss_h = torch.empty(1, dtype=torch.float32, pin_memory=True)
        nchunk = max(1, args.e2e_chunks)
        hp = acrl.HostPipeline(T, V, ld, batch.S, batch.Gn, chunks=nchunk, device=dev)
        comp = torch.cuda.current_stream(dev)

        def one():
            hp.step(step.state, params, h_logits, small_h["ids"], small_h["mask"], small_h["logp_mu"],
                    small_h["rewards"], small_h["seq_offsets"], small_h["group_offsets"], h_grad, loss_h, step.flags)

        one()
        torch.cuda.synchronize()
        n = max(1, args.e2e_steps)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record(comp)
        for _ in range(n):
            one()
        t1.record(comp)            # the pipeline makes this stream wait for each step's downloads
        torch.cuda.synchronize()
        ms = t0.elapsed_time(t1) / n
        ok = bool(torch.equal(h_grad[:, :V].view(torch.int16)[:: max(1, T // 64)].to(dev),
                              step.grad[:, :V].view(torch.int16)[:: max(1, T // 64)]))
        h2d = T * ld * 2 + sum(v.numel() * v.element_size() for v in small_h.values())
        d2h = T * ld * 2 + 4
        return {"value": int(batch.mask.sum()) / (ms / 1e3), "unit": UNIT, "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h, "ms_per_step": ms, "steps": n, "chunks": nchunk,
                "host_link_GB/s": (h2d + d2h) / (ms / 1e3) / 1e9, "download_matches_device": ok,
                "api": "acrl_host_pipeline_step (C ABI), host buffers", "host_memory": pinned.describe()}
    finally:
        if hp is not None:
            hp.close()
        pinned.free()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default="qwen")
    ap.add_argument("--e2e-steps", type=int, default=8)
    ap.add_argument("--e2e-chunks", type=int, default=16)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-lmhead", action="store_true",
                    help="skip the fused LM-head workload that the default run times after the Qwen step")
    ap.add_argument("--ref-seconds", type=float, default=10.0)
    args = ap.parse_args()
    if args.warmup < 3 and args.impl == "ours":
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.workload in ("lmhead", "lmhead_profile"):
        return run_lmhead(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
