"""The work that a training program has this library do, as measurable cases.

A policy update calls the library in a few ways, each through the public
binding: the advantages of a rollout batch, the actor's recomputed
log-probabilities (a forward), the fused loss with its backward (plain, with the
extended objective, or bitwise reproducible) and the same step on one
tensor-parallel rank's slice of the vocabulary.  `listed` holds one case or two
of each over the range of sizes, `draw` further ones of the same ranges.

Inputs follow the synthetic workloads of the repository: hidden states N(0, 1)
and W N(0, 0.02) in bf16, tokens uniform, spans of masked tokens, group
advantages of per-response rewards, behaviour log-probs = current log-prob +
N(0, sigma).  Everything is drawn on the device from the seed alone; as in the
parity tests, behaviour offsets keep clear of the clip boundaries, where the
rounding of one log-prob would decide a row's branch.
"""
import math

import numpy as np
import torch

import paper_2607_21653_gb300 as molt

G = 8                    # responses per prompt group
CLIP_LO, CLIP_HI = 0.2, 0.28
SIGMA = 0.1              # behaviour lag
T_MIN, T_MAX = 32, 65536
H_CHOICES = (256, 320, 512, 896, 1024, 1536, 2048, 2560, 3072, 3584, 4096, 5120)
V_MIN, V_MAX = 1000, 151936
LARGEST = 65536 * 4096 * 151936   # T H V of the largest listed case
EXACT_FLOPS = 1.2e12              # fp64 work up to which `exact` computes a case


def listed():
    return [
        # the advantages of one optimiser window: every rollout's reward normalised in its
        # prompt group and spread over the window's tokens (launch-bound)
        {"name": "advantages window", "kind": "advantages", "n": 4096, "mean_len": 64},
        # a smoke-sized update: the repository's smallest configuration, bound by launches
        {"name": "loss tiny", "kind": "loss", "T": 512, "H": 256, "V": 4096, "masked": 0.0},
        # log-probs of one short response against a large vocabulary: W is read once, almost nothing else
        {"name": "logprobs one response", "kind": "logprobs", "T": 100, "H": 4096, "V": 151936, "masked": 0.0},
        # the allocation-free forward in a runtime that owns all memory, mid model, a few long responses
        {"name": "logprobs noalloc 8k", "kind": "noalloc", "T": 8192, "H": 2048, "V": 32000, "masked": 0.2},
        # recomputed log-probs of a whole microbatch
        {"name": "logprobs 32k", "kind": "logprobs", "T": 32768, "H": 4096, "V": 151936, "masked": 0.3},
        # a small microbatch at an odd length against the large vocabulary: dW's bytes weigh as much as the products
        {"name": "loss 1k large vocab", "kind": "loss", "T": 1031, "H": 4096, "V": 151936, "masked": 0.1},
        # the mid configuration
        {"name": "loss mid", "kind": "loss", "T": 32768, "H": 2048, "V": 32000, "masked": 0.2},
        # the headline configuration
        {"name": "loss large vocab", "kind": "loss", "T": 65536, "H": 4096, "V": 151936, "masked": 0.3},
        # a hidden size that is not a multiple of 128, ragged sizes everywhere
        {"name": "loss ragged h320", "kind": "loss", "T": 5003, "H": 320, "V": 50257, "masked": 0.2},
        # KL to a reference policy, entropy bonus and sequence gate on a ragged microbatch, the widest model
        {"name": "loss extended h5120", "kind": "extended", "T": 16001, "H": 5120, "V": 151936, "masked": 0.05},
        # the bitwise reproducible update
        {"name": "loss deterministic", "kind": "deterministic", "T": 16384, "H": 4096, "V": 65536, "masked": 0.3},
        # one rank of two of the tensor-parallel step: statistics, merge, loss, shard backward
        {"name": "vocab shard of two", "kind": "shard", "T": 8192, "H": 4096, "V": 151936, "masked": 0.3},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("advantages", "logprobs", "noalloc", "loss", "loss", "loss", "extended", "deterministic", "shard"))
    if kind == "advantages":
        return {"kind": kind, "n": _log_uniform(rng, 64, 16384), "mean_len": _log_uniform(rng, 16, 512)}
    hs = [h for h in H_CHOICES if kind != "deterministic" or h % 128 == 0]   # the reproducible mode's own condition
    while True:
        T, H, V = _log_uniform(rng, T_MIN, T_MAX), rng.choice(hs), _log_uniform(rng, V_MIN, V_MAX)
        if kind == "noalloc":
            T = min(T, molt.NOALLOC_MAX_TOKENS)
        # half of the largest, since some kinds cost more per token than the plain loss
        if T * H * V <= LARGEST // 2:
            return {"kind": kind, "T": T, "H": H, "V": V, "masked": round(rng.uniform(0.0, 0.5), 3)}


# ------------------------------------------------------------------- inputs
def _mask(rng, T, frac):
    """1 except on spans of 8-256 tokens covering about `frac` of the batch."""
    m = np.ones(T, dtype=np.uint8)
    left = int(frac * T)
    while left > 0:
        n = min(left, int(rng.integers(8, 257)))
        s = int(rng.integers(0, max(1, T - n)))
        left -= int(m[s:s + n].sum())
        m[s:s + n] = 0
    m[0] = 1
    return m


def _responses(rng, T):
    """Response of each token (lengths log-uniform in [16, 1024], shorter where the batch would not
    hold a group of them) and the group of each response."""
    lo, hi = max(1, min(16, T // 32)), max(2, min(1024, T // 4))
    n = T // lo + 2
    ends = np.cumsum(np.exp(rng.uniform(math.log(lo), math.log(hi), n)).astype(np.int64))
    of_token = np.searchsorted(ends, np.arange(T), side="right").astype(np.int32)
    n_resp = int(of_token[-1]) + 1
    return of_token, (np.arange(n_resp) // G).astype(np.int32)


def _offsets(rng, T):
    """N(0, SIGMA) with the ratio at least 2 % clear of both clip boundaries."""
    off = rng.normal(0.0, SIGMA, T)
    for _ in range(1000):
        bad = (np.abs(-off - math.log1p(-CLIP_LO)) < 0.02) | (np.abs(-off - math.log1p(CLIP_HI)) < 0.02)
        if not bad.any():
            break
        off[bad] = rng.normal(0.0, SIGMA, int(bad.sum()))
    return off.astype(np.float32)


def _logp(h, W, x):
    """Current log-probs, good to a few 1e-3: what a rollout engine would have captured."""
    out = torch.empty(h.shape[0], dtype=torch.float32, device=h.device)
    step = max(1, (1 << 30) // W.shape[0])
    for a in range(0, h.shape[0], step):
        z = h[a:a + step] @ W.t()
        zx = (h[a:a + step].float() * W[x[a:a + step].long()].float()).sum(1)
        out[a:a + step] = zx - torch.logsumexp(z, 1, keepdim=False).float()
    return out


def prepare(case, seed):
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    if case["kind"] == "advantages":
        n = case["n"]
        total = n * case["mean_len"]
        of_token = np.searchsorted(np.sort(rng.integers(0, total, n - 1)), np.arange(total), side="right")
        return {"case": case, "rewards": up(rng.random(n).astype(np.float32)),
                "groups": up((np.arange(n) // G).astype(np.int32)),
                "of_token": up(of_token.astype(np.int32)),
                "mask": up((rng.random(total) < 0.7).astype(np.uint8))}
    T, H, V = case["T"], case["H"], case["V"]
    s = {"case": case,
         "h": torch.randn(T, H, device=dev, generator=gen, dtype=torch.bfloat16),
         "x": up(rng.integers(0, V, T).astype(np.int32)),
         "m": up(_mask(rng, T, case["masked"]))}
    W = torch.empty(V, H, device=dev, dtype=torch.bfloat16).normal_(0.0, 0.02, generator=gen)
    s["W"] = W
    if case["kind"] in ("logprobs", "noalloc"):
        return s
    of_token, groups = _responses(rng, T)
    lp = _logp(s["h"], W, s["x"])
    s.update(rewards=up(rng.random(groups.size).astype(np.float32)), groups=up(groups), of_token=up(of_token),
             b=lp + up(_offsets(rng, T)))
    if case["kind"] == "extended":
        s["ref"] = lp + up(rng.normal(0.0, 0.1, T).astype(np.float32))
    if case["kind"] == "shard":
        half = V // 2
        s["bounds"] = (half, V)
        s["W"], s["other"] = W[half:].clone(), W[:half].clone()
        # the other rank's statistics, as its all-gather delivers them
        s["theirs"] = _partials(s["h"], s.pop("other"), s["x"], s["m"], 0, half)
    return s


def _partials(h, W, x, m, v0, v1):
    """(max, sum e^(z - max), sum e^(z - max)(z - max), z_x or -inf) of columns [v0, v1), as the peer sends it."""
    T = h.shape[0]
    out = torch.empty(T, 4, dtype=torch.float32, device=h.device)
    step = max(1, (1 << 28) // W.shape[0])
    for a in range(0, T, step):
        z = (h[a:a + step] @ W.t()).float()
        M = z.max(1, keepdim=True).values
        e = torch.exp(z - M)
        out[a:a + step, 0] = M[:, 0]
        out[a:a + step, 1] = e.sum(1)
        out[a:a + step, 2] = (e * (z - M)).sum(1)
    xi = x.long()
    inside = (xi >= v0) & (xi < v1)
    zx = torch.empty(T, dtype=torch.float32, device=h.device)
    for a in range(0, T, 4096):
        zx[a:a + 4096] = (h[a:a + 4096].float() * W[(xi[a:a + 4096] - v0).clamp(0, v1 - v0 - 1)].float()).sum(1)
    out[:, 3] = torch.where(inside, zx, torch.full_like(zx, -math.inf))
    off = m == 0
    out[off] = torch.tensor([-math.inf, 0.0, 0.0, -math.inf], device=h.device)
    return out


# ---------------------------------------------------------------------- run
def _advantages(s):
    a = molt.group_advantages(s["rewards"], s["groups"])
    return a, molt.broadcast_advantages(a, s["of_token"])


def _named(out, n_stats):
    """The call's dict with its statistics split into sums (fp64) and counts (int64)."""
    out = dict(out)
    st = out.pop("stats")
    out["sums"], out["counts"] = st[:5], st.view(torch.int64)[5:9]
    if n_stats == 12:
        out["sum_kl"], out["rejected"] = st[9:10], st.view(torch.int64)[10:12]
    return out


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "advantages":
        a, tok = _advantages(s)
        return {"response": a, "token": tok, "count": molt.mask_count(s["mask"])}
    if kind in ("logprobs", "noalloc"):
        call = molt.token_logprobs if kind == "logprobs" else molt.token_logprobs_noalloc
        logp, ent = call(s["h"], s["W"], s["x"], s["m"])
        return {"logp": logp, "entropy": ent}
    _, adv = _advantages(s)
    if kind == "loss":
        return _named(molt.policy_loss_fwd_bwd(s["h"], s["W"], s["x"], s["b"], adv, s["m"], CLIP_LO, CLIP_HI), 9)
    if kind == "extended":
        return _named(molt.policy_loss_fwd_bwd_ex(
            s["h"], s["W"], s["x"], s["b"], adv, s["m"], CLIP_LO, CLIP_HI, kl_coef=0.02, ref_logp=s["ref"],
            entropy_coef=0.001, seq_of_token=s["of_token"], gate_lo=0.5, gate_hi=2.0), 12)
    if kind == "deterministic":
        return _named(molt.policy_loss_fwd_bwd_ex(s["h"], s["W"], s["x"], s["b"], adv, s["m"], CLIP_LO, CLIP_HI,
                                                  deterministic=True), 12)
    v0, _ = s["bounds"]
    mine = molt.vp_partials(s["h"], s["W"], s["x"], v0, s["m"])
    out = _named(molt.vp_loss(torch.stack([s["theirs"], mine]), s["b"], adv, s["m"], CLIP_LO, CLIP_HI), 9)
    out["dhidden"], out["dW"] = molt.vp_backward(s["h"], s["W"], s["x"], out["lse"], out["coef"], v0)
    return out


# ----------------------------------------------------------------- measures
def work(case):
    if case["kind"] == "advantages":
        return {"bytes": case["n"] * 12 + case["n"] * case["mean_len"] * 9, "flops": 0}
    T, H, V = case["T"], case["H"], case["V"]
    act = T * (1.0 - case["masked"])
    if case["kind"] == "shard":
        V -= V // 2
    rows = act * H * 2 + V * H * 2 + T * 13
    if case["kind"] in ("logprobs", "noalloc"):
        return {"bytes": rows, "flops": 2.0 * act * H * V}
    return {"bytes": rows + T * H * (4 if case["kind"] == "shard" else 2) + V * H * 4, "flops": 6.0 * act * H * V}


def tolerance(case):
    """Advantages are correctly rounded fp64 and compare bit for bit.  A forward
    is fp32 sums over H and V of exact bf16 products.  The gradients are products
    of a bf16-rounded softmax gradient (2.5e-3 relative 2-norm against 64 bits)."""
    if case["kind"] == "advantages":
        return "exact"
    if case["kind"] in ("logprobs", "noalloc"):
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.1}


# ----------------------------------------------------------------- 64 bits
def _exact_advantages(s):
    r, g = s["rewards"].double().cpu().numpy(), s["groups"].cpu().numpy()
    a = np.zeros_like(r)
    for k in range(0, r.size, G):
        q = r[k:k + G]
        assert (g[k:k + G] == g[k]).all()
        if q.size > 1:
            a[k:k + G] = (q - q.mean()) / (q.std(ddof=1) + 1e-6)
    a = torch.from_numpy(a).to(s["rewards"].device)
    return a, a[s["of_token"].long()]


def exact(case, seed):
    kind = case["kind"]
    if kind != "advantages" and work(case)["flops"] > EXACT_FLOPS:
        return None
    s = prepare(case, seed)
    if kind == "advantages":
        a, tok = _exact_advantages(s)
        return {"response": a, "token": tok, "count": None}
    if kind == "shard":
        return None
    h, W, x, act = s["h"].double(), s["W"].double(), s["x"].long(), s["m"] != 0
    T, V = case["T"], case["V"]
    zero = torch.zeros(T, dtype=torch.float64, device=h.device)
    logp, ent, lse = zero.clone(), zero.clone(), zero.clone()
    step = max(1, (1 << 27) // V)
    for a in range(0, T, step):
        z = h[a:a + step] @ W.t()
        l = torch.logsumexp(z, 1)
        p = torch.exp(z - l[:, None])
        lse[a:a + step] = l
        logp[a:a + step] = z.gather(1, x[a:a + step, None])[:, 0] - l
        ent[a:a + step] = l - (p * z).sum(1)
        del z, p
    if kind in ("logprobs", "noalloc"):
        return {"logp": torch.where(act, logp, zero), "entropy": torch.where(act, ent, zero)}
    _, A = _exact_advantages(s)
    A = A.float().double()
    D = float(act.sum())
    b = s["b"].double()
    ratio = torch.exp(logp - b)
    lo, hi = 1.0 - CLIP_LO, 1.0 + CLIP_HI
    clipped = ((A > 0) & (ratio > hi)) | ((A < 0) & (ratio < lo))
    tl = -torch.where(clipped, ratio.clamp(lo, hi) * A, ratio * A)
    c = torch.where(clipped, zero, ratio * A)
    ecoef, keep = zero, act
    if kind == "extended":
        r = s["ref"].double() - logp
        kl = torch.expm1(r) - r
        seq = s["of_token"].long()
        n = int(seq[-1]) + 1
        tot = torch.zeros(n, dtype=torch.float64, device=h.device).index_add_(0, seq, torch.where(act, logp - b, zero))
        cnt = torch.zeros(n, dtype=torch.float64, device=h.device).index_add_(0, seq, act.double())
        g = torch.exp(tot / cnt.clamp(min=1))
        keep = act & ((g >= 0.5) & (g <= 2.0))[seq]
        tl = tl + 0.02 * kl - 0.001 * ent
        c = c + 0.02 * torch.expm1(r)
        ecoef = torch.where(keep, torch.full_like(zero, 0.001 / D), zero)
    tl = torch.where(keep, tl, zero)
    coef = torch.where(keep, c / D, zero)
    mu = lse - ent
    dh = torch.empty_like(h)
    dW = torch.zeros_like(W)
    for a in range(0, T, step):
        z = h[a:a + step] @ W.t()
        g = torch.exp(z - lse[a:a + step, None]) * (coef[a:a + step, None]
                                                    + ecoef[a:a + step, None] * (z - mu[a:a + step, None]))
        g.scatter_add_(1, x[a:a + step, None], -coef[a:a + step, None])
        dh[a:a + step] = g @ W
        dW.addmm_(g.t(), h[a:a + step])
        del z, g
    out = {"loss": (tl.sum() / D).reshape(1), "dhidden": dh, "dW": dW, "logp": torch.where(act, logp, zero),
           "entropy": torch.where(act, ent, zero), "token_loss": tl, "sums": None, "counts": None}
    if kind in ("extended", "deterministic"):
        out.update(sum_kl=None, rejected=None)
    return out
