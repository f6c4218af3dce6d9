#!/usr/bin/env python
"""Benchmark of the fused policy-loss hot path; prints one JSON line.

One step = GRPO group advantages + per-token broadcast + the fused LM-head
clipped-surrogate forward and backward (dhidden, dW) over one batch of the
large-vocab workload: T = 65536 tokens (128 prompt groups x G=8 x 64 tokens),
H = 4096, V = 151936, bf16 hidden states and weights, 30% of the tokens masked
in spans of 8-256, clip eps 0.2 / 0.28.  Inputs are synthetic and seeded
(workloads.make_workload), resident in HBM before the timed region; W alone is
1.24 GB, larger than L2, so no extra flush runs between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--estimator grpo|group_mean|dr_grpo|rloo|reinforce_pp]
                  [--objective ppo|kl_entropy_gate] [--deterministic] [--vshard N]

--estimator picks the advantage estimator (Sec. 4.5 list); --objective
kl_entropy_gate adds a KL-to-reference term, an entropy bonus and the
sequence-level importance gate (one sequence per rollout) to the loss.  The
defaults are the headline configuration (GRPO, clipped surrogate).

With torchrun (N > 1) every rank processes its own batch (different seed)
with no collective on the data path ("scaling": "weak"); rank 0 prints.

--vshard N splits W by vocabulary into N shards and runs the step through the
vocabulary-parallel calls (shard statistics, their merge with the loss, the
shards' backward).  On one process the N shards run one after another on the
GPU; under torchrun with N ranks, rank r holds shard r and the ranks exchange
the statistics (all-gather) and the dhidden terms (all-reduce) over NCCL, one
batch per step for the whole job ("scaling": "strong").
--impl reference times the fp64 CPU oracle on the host cores instead, on a
bounded sample of rows per step.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

# torchrun starts every rank with OMP_NUM_THREADS=1.  The reference arm runs the
# oracle on rank 0 alone, so there it gets every host core back; this has to
# happen before numpy loads its BLAS.
if "LOCAL_RANK" in os.environ and os.environ.get("RANK", "0") == "0" and "reference" in sys.argv[1:]:
    for _k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[_k] = str(os.cpu_count() or 1)

import numpy as np


def blas_threads():
    """Threads numpy's BLAS runs the oracle's products on: the host cores,
    unless a thread-count variable caps them."""
    n = os.cpu_count() or 1
    for k in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        v = os.environ.get(k, "")
        if v.isdigit() and int(v) > 0:
            return min(n, int(v))
    return n

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "policy-loss fwd+bwd tokens/s on 1 GB300; % of dense bf16 tensor peak"


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return {"hbm_gbs": d["hbm_gbs"], "bf16": d["bf16_tflops"], "bf16_sustained": d["bf16_tflops_sustained"],
                "source": "measured"}
    return {"hbm_gbs": 6800.0, "bf16": 1900.0, "bf16_sustained": 1700.0, "source": "fallback"}


def code_hash(path):
    """First 16 hex digits of the sha256 of a C++/CUDA source with its comments
    removed and its whitespace collapsed: edits to comments leave it unchanged,
    any change to the code does not."""
    import hashlib
    import re
    with open(path, encoding="utf-8") as f:
        src = f.read()
    src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
    src = re.sub(r"//[^\n]*", " ", src)
    src = " ".join(src.split())
    return hashlib.sha256(src.encode()).hexdigest()[:16]


def recorded_traffic(kernel, workload, schedule, rows):
    """DRAM bytes per launch of `kernel` on `workload` under `schedule`
    ("default" or "deterministic") from the ncu summaries under profiles/, or
    None if no summary matches them and the current source of the kernel.
    A summary captured on fewer token rows (the same H and V) is scaled to
    `rows` by 256-row token tiles: each is formed, read and added to the same
    number of times whatever their number.  Returns (bytes, note)."""
    import glob
    tiles = lambda r: -(-r // 256)
    for path in sorted(glob.glob(os.path.join(ROOT, "profiles", "*.md"))):
        with open(path) as f:
            for line in f:
                if not line.startswith("traffic:"):
                    continue
                kv = dict(tok.split("=", 1) for tok in line.split()[1:] if "=" in tok)
                if (kv.get("kernel") != kernel or kv.get("workload") != workload
                        or kv.get("schedule") != schedule):
                    continue
                src = os.path.join(ROOT, kv.get("source", ""))
                if not (os.path.isfile(src) and code_hash(src) == kv.get("code_sha256_16")):
                    continue
                b = float(kv["dram_bytes_per_launch"])
                r = int(kv.get("rows", "0"))
                if r > 0 and r != rows:
                    return b * tiles(rows) / tiles(r), (f"ncu capture on {r} backward rows ({tiles(r)} token tiles), "
                                                        f"scaled to {tiles(rows)} tiles")
                return b, "ncu capture of this launch"
    return None, None


def workload_desc(w, microbatch=0):
    window = w.extra.get("window_tokens")
    return (f"{w.name}: T={w.T}, H={w.H}, V={w.V}, bf16, "
            f"{100 * (1 - w.mask.mean()):.0f}% masked in spans, clip {w.eps_lo}/{w.eps_hi}"
            + (f", microbatch {microbatch} of a {window}-token window" if window else ""))


# ------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
    NAMES = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200",
                 "-i", str(self.gpu)], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    mx.append(float(parts[2]))
                except ValueError:
                    continue
                for name, v in zip(self.NAMES, parts[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(name)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def gpu_index_for(local_rank):
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        ids = [v.strip() for v in vis.split(",") if v.strip()]
        if local_rank < len(ids) and ids[local_rank].isdigit():
            return int(ids[local_rank])
    return local_rank


# -------------------------------------------------------------- cpu oracle
def oracle_rows_rate(w, n_rows_target_s, seed=0, max_rows=4096):
    """Time the fp64 oracle (forward, dhidden rows and dW contribution) on a
    bounded sample of active rows of the workload; returns (tokens/s, rows, s)."""
    from oracle import molt_oracle as O
    rng = np.random.default_rng(seed)
    act = np.nonzero(w.mask)[0]
    W64 = O.widen_bf16(w.weight)
    adv = rng.standard_normal(w.T)
    b = rng.normal(-np.log(w.V) - 1.0, 1.0, w.T)
    D = float(w.mask.sum())

    def run(rows):
        h_rows = np.zeros((w.T, w.H))
        h_rows[rows] = O.widen_bf16(w.hidden[rows])
        t0 = time.perf_counter()
        O.policy_loss_rows(h_rows, W64, w.tokens, b, adv, w.mask, w.eps_lo, w.eps_hi, D, rows, want_dW=True)
        return time.perf_counter() - t0

    # size the sample from a 64-row probe, charging the call's fixed cost (the
    # V x H dW accumulator) to its rows: this never overshoots the target
    t64 = run(rng.choice(act, size=min(64, act.size), replace=False))
    n = int(min(max_rows, max(8, n_rows_target_s * 64 / max(t64, 1e-6))))
    n = max(8, (n // 8) * 8)
    rows = rng.choice(act, size=min(n, act.size), replace=False)
    dt = run(rows)
    return len(rows) / dt, len(rows), dt


def oracle_tiny_whole_rate():
    """Oracle tokens/s on the whole tiny workload (T=512, H=256, V=4096): the
    full forward and backward of every row."""
    from oracle import molt_oracle as O
    from workloads import make_workload
    w = make_workload("tiny")
    rng = np.random.default_rng(0)
    adv = rng.standard_normal(w.T)
    b = rng.normal(-np.log(w.V) - 1.0, 1.0, w.T)
    h64, W64 = O.widen_bf16(w.hidden), O.widen_bf16(w.weight)
    t0 = time.perf_counter()
    O.policy_loss(h64, W64, w.tokens, b, adv, w.mask, w.eps_lo, w.eps_hi)
    return w.T / (time.perf_counter() - t0)


def oracle_single_thread_rate():
    """oracle_tiny_whole_rate in a child process whose BLAS runs one thread."""
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1")
    code = "import bench; print(bench.oracle_tiny_whole_rate())"
    try:
        r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True,
                           timeout=120)
        return float(r.stdout.strip().splitlines()[-1])
    except Exception:   # the extra figure is optional; the line stays valid without it
        return None


def microbatch_of(args):
    """Microbatch of a windowed workload: the ragged window's first one holds only
    its two constant-reward groups (every advantage 0, no gradient), so it
    defaults to microbatch 1."""
    if args.microbatch is not None:
        return args.microbatch
    return 1 if args.workload == "ragged" else 0


def run_reference(args):
    """--impl reference: the fp64 oracle on the host cores, per step a bounded
    sample of rows of the same workload."""
    from workloads import make_workload
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    w = make_workload(args.workload, microbatch=microbatch_of(args))
    from oracle import molt_oracle as O
    rng = np.random.default_rng(1)
    act = np.nonzero(w.mask)[0]
    W64 = O.widen_bf16(w.weight)
    adv = rng.standard_normal(w.T)
    b = rng.normal(-np.log(w.V) - 1.0, 1.0, w.T)
    D = float(w.mask.sum())
    rows_per_step = args.ref_rows
    h64 = np.zeros((w.T, w.H))

    def step(i):
        rows = np.sort(rng.choice(act, size=rows_per_step, replace=False))
        h64[rows] = O.widen_bf16(w.hidden[rows])
        t0 = time.perf_counter()
        O.policy_loss_rows(h64, W64, w.tokens, b, adv, w.mask, w.eps_lo, w.eps_hi, D, rows, want_dW=True)
        return time.perf_counter() - t0

    for i in range(args.warmup):
        step(i)
    ts = [step(i) for i in range(args.steps)]
    tot = sum(ts)
    value = rows_per_step * args.steps / tot
    cores = blas_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "tokens/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * tot / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_desc(w, microbatch_of(args)), "sample": f"{rows_per_step} random active rows per step"},
        "cpu_baseline": {"value": value, "unit": "tokens/s", "cores": cores, "kind": "oracle",
                         "sample": f"{rows_per_step} active rows per step (forward, dhidden rows, dW contribution)"},
        "e2e": {"value": value, "unit": "tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------- multi-rank
def rank_seed(workload_seed_default, rank, world):
    """Seed of each rank's batch: the workload's own seed on a single GPU, a
    distinct seed per rank otherwise (independent replicas, weak scaling)."""
    return None if world == 1 else 2 + 100 * rank


def max_over_ranks(value_ms, world, device=None):
    """Slowest rank's time: every rank contributes its own elapsed time."""
    if world == 1:
        return float(value_ms)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value_ms)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(tokens_per_rank, world, steps, ms):
    """Whole-job tokens/s: all ranks' tokens over the slowest rank's time."""
    return world * tokens_per_rank * steps / (ms / 1e3)


# ------------------------------------------------------------------ our arm
def run_ours(args):
    import torch
    import torch.distributed as dist

    import paper_2607_21653_gb300 as molt
    from workloads import make_workload

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    molt.build()
    molt.load()
    peaks = load_peaks()

    w = make_workload(args.workload, seed=rank_seed(None, rank, world), microbatch=microbatch_of(args),
                      T=args.tokens)
    T, H, V = w.T, w.H, w.V

    def bf(bits):
        return torch.from_numpy(bits.view(np.int16)).to(dev).view(torch.bfloat16)

    hidden = bf(w.hidden)
    weight = bf(w.weight)
    tokens = torch.from_numpy(w.tokens).to(dev)
    mask = torch.from_numpy(w.mask).to(dev)
    rewards = torch.from_numpy(w.rewards).to(dev)
    gids = torch.from_numpy(w.group_ids).to(dev)
    rot = torch.from_numpy(w.resp_of_token).to(dev)
    # behaviour log-probs: the current policy's log-probs plus N(0, sigma) lag
    lp, _ = molt.token_logprobs(hidden, weight, tokens, None, want_entropy=False)
    noise = np.random.default_rng(w.seed + 17).normal(0.0, w.behavior_sigma, T).astype(np.float32)
    b = (lp + torch.from_numpy(noise).to(dev)).contiguous()
    adv_resp = torch.empty(w.rewards.shape[0], dtype=torch.float32, device=dev)
    adv_tok = torch.empty(T, dtype=torch.float32, device=dev)
    dW = torch.empty(V, H, dtype=torch.float32, device=dev)
    n_active = int(w.mask.sum())
    extended = args.objective == "kl_entropy_gate" or args.deterministic
    ex_opts = {"deterministic": args.deterministic}
    if args.objective == "kl_entropy_gate":
        # reference-policy log-probs: the current ones plus an independent lag;
        # one gated sequence per rollout; a band wide enough that the gate
        # rejects (and so skips) no work at this behaviour lag
        rnoise = np.random.default_rng(w.seed + 29).normal(0.0, 0.1, T).astype(np.float32)
        ex_opts = dict(kl_coef=0.01, ref_logp=(lp + torch.from_numpy(rnoise).to(dev)).contiguous(),
                       entropy_coef=1e-3, seq_of_token=rot, gate_lo=0.5, gate_hi=2.0,
                       deterministic=args.deterministic)

    def step(tok=tokens, msk=mask, hid=hidden, bb=b, rw=rewards, gi=gids, ro=rot, rf=None):
        if args.estimator == "grpo":
            molt.group_advantages(rw, gi, out=adv_resp)
        else:
            molt.advantages(rw, None if args.estimator == "reinforce_pp" else gi, estimator=args.estimator,
                            out=adv_resp)
        molt.broadcast_advantages(adv_resp, ro, out=adv_tok)
        if extended:
            opts = dict(ex_opts)
            if "seq_of_token" in opts:
                opts.update(seq_of_token=ro, ref_logp=opts["ref_logp"] if rf is None else rf)
            return molt.policy_loss_fwd_bwd_ex(hid, weight, tok, bb, adv_tok, msk, w.eps_lo, w.eps_hi, dW=dW,
                                               want_token_outputs=False, **opts)
        return molt.policy_loss_fwd_bwd(hid, weight, tok, bb, adv_tok, msk, w.eps_lo, w.eps_hi, dW=dW,
                                        want_token_outputs=False)

    vshard = args.vshard
    mine = []
    if vshard > 1:
        if world not in (1, vshard):
            raise SystemExit("--vshard N runs on one process or on N ranks")
        if extended or args.estimator != "grpo":
            raise SystemExit("--vshard runs the headline objective (GRPO, clipped surrogate)")
        bounds = molt.vocab_shard_bounds(V, vshard)
        mine = [bounds[rank]] if world > 1 else bounds
        w_sh = [weight[a:e] for a, e in mine]
        dW_sh = [torch.empty(e - a, H, dtype=torch.float32, device=dev) for a, e in mine]
        dh_sum = torch.empty(T, H, dtype=torch.float32, device=dev)
        vp_timer = {"t": None, "k": 0}

        def arm():
            if vp_timer["t"] is not None:
                vp_timer["t"].arm(vp_timer["k"])
                vp_timer["k"] += 1

        def step(tok=tokens, msk=mask, hid=hidden, bb=b, rw=rewards, gi=gids, ro=rot, rf=None):
            molt.group_advantages(rw, gi, out=adv_resp)
            molt.broadcast_advantages(adv_resp, ro, out=adv_tok)
            parts = []
            for (a, e), ws in zip(mine, w_sh):
                arm()
                parts.append(molt.vp_partials(hid, ws, tok, a, msk))
            parts = molt.gather_shard_partials(parts[0]) if world > 1 else torch.stack(parts)
            arm()
            out = molt.vp_loss(parts, bb, adv_tok, msk, w.eps_lo, w.eps_hi)
            dh_sum.zero_()
            for (a, e), ws, dws in zip(mine, w_sh, dW_sh):
                arm()
                dh_s, _ = molt.vp_backward(hid, ws, tok, out["lse"], out["coef"], a, dW=dws)
                dh_sum.add_(dh_s)
            if world > 1:
                molt.sum_dhidden(dh_sum)
            out["dhidden"] = dh_sum
            return out

    def barrier():
        if world > 1:
            dist.barrier()

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    assert molt.device_status() == 0
    barrier()

    calls_per_step = 2 * len(mine) + 1 if vshard > 1 else 1
    timer = molt.KernelTimer(args.steps * calls_per_step)
    if vshard > 1:
        vp_timer["t"] = timer
    clocks = ClockSampler(gpu_index_for(local_rank))
    clocks.start()
    time.sleep(0.3)
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    barrier()
    torch.cuda.synchronize()
    launches0 = molt.kernel_launches()
    # an event between consecutive steps as well, for the per-step median
    marks = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps - 1)]
    t0.record()
    for k in range(args.steps):
        if k > 0:
            marks[k - 1].record()
        if vshard <= 1:
            timer.arm(k)
        out = step()
    t1.record()
    launches = molt.kernel_launches() - launches0
    timer.disarm()
    if vshard > 1:
        vp_timer["t"] = None
    torch.cuda.synchronize()
    barrier()
    clk = clocks.stop()
    ms = t0.elapsed_time(t1)
    bounds = [t0] + marks + [t1]
    step_ms = sorted(bounds[k].elapsed_time(bounds[k + 1]) for k in range(args.steps))
    ms_median = 0.5 * (step_ms[(args.steps - 1) // 2] + step_ms[args.steps // 2])
    per = timer.elapsed_ms()
    timer.close()
    assert molt.device_status() == 0
    loss_val = float(out["loss"].item())
    step_stats = molt.stats_dict(out["stats"])
    ms = max_over_ranks(ms, world, dev)
    ms_median = max_over_ranks(ms_median, world, dev)

    # ---- end to end through the public API with host buffers
    e2e = None
    if not args.no_e2e and vshard <= 1:
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
        h_hid = pin(w.hidden.view(np.int16))
        h_tok, h_msk, h_b = pin(w.tokens), pin(w.mask), pin(b.cpu().numpy())
        h_rw, h_gi, h_ro = pin(w.rewards), pin(w.group_ids), pin(w.resp_of_token)
        h_rf = pin(ex_opts["ref_logp"].cpu().numpy()) if "ref_logp" in ex_opts else None
        h_loss = torch.empty(1, dtype=torch.float32).pin_memory()
        # two sets of device inputs: step k computes from set k % 2 while the
        # host-to-device copies of step k + 1 fill the other set on a copy stream
        sets = []
        for _ in range(2):
            d_hid = torch.empty(T, H, dtype=torch.int16, device=dev)
            d_tok, d_msk, d_b = torch.empty_like(tokens), torch.empty_like(mask), torch.empty_like(b)
            d_rw, d_gi, d_ro = torch.empty_like(rewards), torch.empty_like(gids), torch.empty_like(rot)
            d_rf = torch.empty_like(ex_opts["ref_logp"]) if h_rf is not None else None
            cps = [(d_hid, h_hid), (d_tok, h_tok), (d_msk, h_msk), (d_b, h_b), (d_rw, h_rw), (d_gi, h_gi),
                   (d_ro, h_ro)] + ([(d_rf, h_rf)] if h_rf is not None else [])
            sets.append((cps, (d_tok, d_msk, d_hid.view(torch.bfloat16), d_b, d_rw, d_gi, d_ro, d_rf)))
        h2d = sum(src.numel() * src.element_size() for _, src in sets[0][0])
        e_steps = max(2, args.steps // 2)
        comp = torch.cuda.current_stream(dev)
        copy_stream = torch.cuda.Stream(device=dev)
        copied = [torch.cuda.Event() for _ in range(2)]
        freed = [torch.cuda.Event() for _ in range(2)]
        go = torch.cuda.Event()

        def issue_copies(k):
            with torch.cuda.stream(copy_stream):
                copy_stream.wait_event(freed[k % 2] if k >= 2 else go)   # set free, timed region open
                for dst, src in sets[k % 2][0]:
                    dst.copy_(src, non_blocking=True)
                copied[k % 2].record(copy_stream)

        def run_e2e(n):
            go.record(comp)
            issue_copies(0)
            out = None
            for k in range(n):
                if k + 1 < n:
                    issue_copies(k + 1)
                comp.wait_event(copied[k % 2])
                out = step(*sets[k % 2][1])
                freed[k % 2].record(comp)
                h_loss.copy_(out["loss"], non_blocking=True)
            return out

        run_e2e(2)
        torch.cuda.synchronize()
        barrier()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        run_e2e(e_steps)
        e1.record()
        torch.cuda.synchronize()
        assert molt.device_status() == 0
        ems = e0.elapsed_time(e1)
        ems = max_over_ranks(ems, world, dev)
        e2e = {"value": job_throughput(T, world, e_steps, ems), "unit": "tokens/s", "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": 4, "steps": e_steps,
               "note": "hidden, tokens, mask, behaviour log-probs, rewards, group ids and the token->rollout map "
                       + ("(and reference log-probs) " if "ref_logp" in ex_opts else "")
                       + "copied from pinned host memory every step, on a copy stream into one of two device "
                         "input sets while the previous step computes; W stays resident; loss read back every step"}

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return 0

    # ---- roofline of the dominant kernel (backward): algorithmic flops = dhidden
    # and dW products, 4 T_p H V per launch, over its CUDA-event time.  T_p is
    # the rows the backward processes (active rows with a gradient), the
    # forward's are the active rows: rows left out never count as work done.
    # With vocabulary shards on N ranks each rank's V is its shard's.
    tp = step_stats["n_grad_rows"]
    V_work = (mine[0][1] - mine[0][0]) if (vshard > 1 and world > 1) else V
    bwd_s = per["backward"] / 1e3 / args.steps
    fwd_s = per["forward"] / 1e3 / args.steps
    peak = peaks["bf16_sustained"]
    achieved_bwd = 4.0 * tp * H * V_work / bwd_s / 1e12
    step_s = ms / 1e3 / args.steps
    step_flops = (2.0 * n_active + 4.0 * tp) * H * V_work
    step_frac = step_flops / step_s / 1e12 / peak
    V_launch = mine[0][1] - mine[0][0] if vshard > 1 else V
    bwd_kernel = molt.backward_plan(T, H, V_launch, bool(args.deterministic))["kernel"]
    executed = 6.0 * tp * H * V_work / bwd_s / 1e12
    traffic, traffic_note = (None, None) if vshard > 1 else recorded_traffic(
        bwd_kernel, w.name, "deterministic" if args.deterministic else "default", tp)
    roofline = {
        "kernel": bwd_kernel, "bound": "tensor", "achieved": achieved_bwd, "peak": peak, "unit": "TFLOP/s",
        "frac": achieved_bwd / peak,
        "traffic": traffic,
        "traffic_source": traffic_note,
        "limiter": limiter(executed / peak, clk, args.deterministic),
        "peak_source": f"{peaks['source']} bf16 sustained (kernel timed inside a long step)",
        "kernels_per_step": launches / args.steps,
        "algorithmic_flops_per_launch": 4.0 * tp * H * V_work / max(1, len(mine)),
        "backward_rows": tp,
        "executed_tflops": executed,
        "forward_kernel_tflops": 2.0 * n_active * H * V_work / fwd_s / 1e12,
        "kernel_ms_per_step": {k: v / args.steps for k, v in per.items()},
    }

    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        rate, nrows, secs = oracle_rows_rate(w, args.cpu_seconds)
        cpu = {"value": rate, "unit": "tokens/s", "cores": blas_threads(), "kind": "oracle",
               "sample": f"{nrows} random active rows of the same batch (forward, dhidden rows, dW contribution), "
                         f"{secs:.1f} s, numpy fp64 BLAS on all host cores",
               "tiny_whole_tokens_per_s": oracle_tiny_whole_rate(),
               "tiny_whole_single_thread_tokens_per_s": oracle_single_thread_rate()}

    line = {
        "metric": METRIC,
        "value": job_throughput(T, 1 if vshard > 1 else world, args.steps, ms),
        "unit": "tokens/s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": ms / args.steps,
        "ms_per_step_median": ms_median,
        "higher_is_better": True,
        "scaling": "strong" if vshard > 1 else "weak",
        "vs_baseline": None,
        "dtype": "bf16",
        "data": "synthetic",
        "config": {"workload": workload_desc(w, microbatch_of(args)), "global_batch_tokens": world * T, "active_tokens": n_active,
                   "parallelism": (f"vocab-parallel x{vshard}" + (" (shards one after another on one GPU)"
                                                                  if world == 1 else " over NCCL")
                                   if vshard > 1 else f"replicas x{world}" if world > 1 else "single GPU"),
                   "backward_rows": tp,
                   "l2": l2_note(T, H, V),
                   "active_tokens_per_s": job_throughput(n_active, 1 if vshard > 1 else world, args.steps, ms),
                   "tensor_peak_frac_6THV": step_frac,
                   "tensor_peak_frac_8THV": (2.0 * n_active + 6.0 * tp) * H * V_work / step_s / 1e12 / peak,
                   "tensor_peak_frac_6THV_of_burst": step_flops / step_s / 1e12 / peaks["bf16"],
                   "loss": loss_val, "estimator": args.estimator, "objective": args.objective,
                   "deterministic": bool(args.deterministic),
                   **({"kl_coef": 0.01, "entropy_coef": 1e-3, "gate": [0.5, 2.0],
                       "seq_rejected": step_stats.get("n_seq_rejected")}
                      if args.objective == "kl_entropy_gate" else {})},
        "roofline": roofline,
        "cpu_baseline": cpu,
        "clocks": clk,
        "e2e": e2e,
        "gpu_launches": launches,
    }
    print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def limiter(executed_frac, clk, deterministic):
    """What bounds the backward in this run: the logits are formed again in it, so it
    executes 6 T_p H V where 4 T_p H V are counted."""
    at = f"{100 * executed_frac:.0f}% of the sustained cuBLAS rate on what is executed (6 T_p H V; 4 T_p H V counted)"
    if executed_frac < 0.8:
        why = "additions of 512-token and 512-column terms to the sums" if deterministic else "waits between tiles"
        return f"not the tensor cores alone: {at}; {why}"
    cap = "sw_power_cap" in (clk or {}).get("reasons", [])
    return f"tensor cores{' under the board power cap' if cap else ''}: {at}"


def l2_note(T, H, V):
    """Why no L2 flush runs between steps: what one step reads and writes."""
    w_gb, h_gb = V * H * 2 / 1e9, T * H * 2 / 1e9
    total = w_gb + h_gb + (V * H * 4 + T * H * 4) / 1e9
    return (f"no flush: each step reads W ({w_gb:.2f} GB) and hidden ({h_gb:.2f} GB) and writes "
            f"fp32 dW and dhidden, {total:.2f} GB in all, against 129 MB of L2")


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    # the timed workloads: each moves far more than L2 per step, so no flush
    # runs between steps (the tiny configuration is a parity case only)
    ap.add_argument("--workload", default="large_vocab", choices=("mid", "large_vocab", "long_traj", "ragged"))
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--ref-rows", type=int, default=32)
    ap.add_argument("--estimator", default="grpo", choices=("grpo", "group_mean", "dr_grpo", "rloo", "reinforce_pp"))
    ap.add_argument("--objective", default="ppo", choices=("ppo", "kl_entropy_gate"))
    ap.add_argument("--microbatch", type=int, default=None,
                    help="microbatch of a windowed workload (ragged: default 1)")
    ap.add_argument("--deterministic", action="store_true",
                    help="bitwise-reproducible dW / dhidden (reduce-adds take turns in a fixed order)")
    ap.add_argument("--tokens", type=int, default=None,
                    help="fewer token rows than the workload's (same H, V and structure): small profiling cases")
    ap.add_argument("--vshard", type=int, default=1,
                    help="vocabulary-parallel step over N shards (one GPU: one after another; N ranks: one each)")
    args = ap.parse_args()
    if args.warmup < 3 and args.impl == "ours":
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
