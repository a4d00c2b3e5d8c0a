"""What is measured: the calls of the SAO loss head as a training program makes them.

A case is a plain dict. `kind` says which calls one pass makes, all of them
through `paper_2607_07508_gb300.sao`:

  head     the LM-head log-probs alone: forward and backward (`path`
           "recompute" or "cached"), or the forward only ("score", as a program
           does that scores rollouts under another policy)
  step     the six calls of one training step: advantages, log-prob forward,
           policy loss forward and backward, log-prob backward, value loss
  tokens   the per-token calls of a step, without the LM head: advantages,
           policy loss forward and backward, value loss
  turns    step-level (one conversation turn = one action) advantages
  grpo     the GRPO comparison arm: group advantages, clipped surrogate
           forward and backward, one weight per sequence
  running  the running-mean comparison arm: running-mean advantages, then the
           decoupled three-policy objective forward and backward

Sizes are those of the repository's configurations (tiny, small, moe, long,
large: hidden size, vocabulary, tokens, trajectory lengths, clip bounds and
lambdas), of micro-batches of them with odd token counts, and for the
per-token calls up to the largest batch that the method's paper trains on (128
trajectories of up to 128k tokens). Inputs are drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2607_07508_gb300 import sao

DEV = "cuda"
F64 = torch.float64

# The heads (hidden size, vocabulary) of the repository's configurations.
HEADS = {"tiny": (256, 4096), "small": (1024, 32000), "moe": (2048, 151936), "long": (4096, 151936),
         "large": (6144, 154880)}


def _head_case(name, **kw):
    h, V = HEADS[kw.pop("head")]
    return dict(name=name, h=h, V=V, **kw)


def listed():
    return [
        # the tiny configuration: a whole fp32 step on 8 short trajectories, as in a unit test or a debug run
        _head_case("tiny_step_f32", kind="step", head="tiny", dtype="f32", N=2304, median=288, obs=0.0, lam=1.0,
                   alpha=0.0, eps_low=0.2, eps_high=0.28),
        # an fp32 reference run of the small head on one ragged micro-batch
        _head_case("small_head_f32", kind="head", head="small", dtype="f32", path="recompute", N=4099, obs=0.25,
                   accumulate=False),
        # one short trajectory per micro-batch on the moe head, gradients accumulated into dW
        _head_case("moe_micro_bf16", kind="head", head="moe", dtype="bf16", path="recompute", N=517, obs=0.25,
                   accumulate=True),
        # a few trajectories per micro-batch, with the forward's probabilities kept for the backward
        _head_case("moe_cached_bf16", kind="head", head="moe", dtype="bf16", path="cached", N=8192, obs=0.25,
                   accumulate=False),
        # log-probs of rollouts under the policy of the large head, no gradient
        _head_case("large_score_bf16", kind="head", head="large", dtype="bf16", path="score", N=4095, obs=0.4,
                   accumulate=False),
        # the small configuration, whole step (no observation tokens, gamma = lambda = 1)
        _head_case("small_step_bf16", kind="step", head="small", dtype="bf16", N=98304, median=1024, obs=0.0, lam=1.0,
                   alpha=0.0, eps_low=0.2, eps_high=0.28),
        # the moe configuration, whole step: the repository's benchmark
        _head_case("moe_step_bf16", kind="step", head="moe", dtype="bf16", N=65536, median=4096, obs=0.25, lam=0.95,
                   alpha=0.0, eps_low=0.3, eps_high=5.0),
        # the per-token calls of a step of the moe configuration's size: latency and launches
        dict(name="tokens_64k", kind="tokens", N=65536, median=4096, obs=0.25, lam=0.95, alpha=0.0, eps_low=0.3,
             eps_high=5.0),
        # the same calls on the largest batch of the paper's runs, length-adaptive lambda, masked tool output
        dict(name="tokens_16m", kind="tokens", N=128 * 131072 - 77, median=65536, obs=0.40, lam=1.0, alpha=1.5,
             eps_low=0.8, eps_high=3.0),
        # step-level advantages of a large multi-turn batch
        dict(name="turns_4m", kind="turns", N=(1 << 22) + 1021, median=32768, obs=0.40, lam=0.95, alpha=0.0,
             mode="average"),
        # GRPO with DIS bounds: groups of 8 rollouts
        dict(name="grpo_4m", kind="grpo", N=1 << 22, median=4096, obs=0.25, group=8, eps_low=0.2, eps_high=0.28),
        # running-mean baseline (window 8 per prompt) and the decoupled objective
        dict(name="running_1m", kind="running", N=(1 << 20) + 333, median=2048, obs=0.25, prompts=256, window=8,
             eps_low=0.2, eps_high=0.28),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if n % 2 == 0 and rng.random() < 0.5:  # odd ones among them
        n += 1 if n < hi else -1
    return n


def draw(rng):
    kind = rng.choice(["head", "head", "step", "tokens", "tokens", "turns", "grpo", "running"])
    c = {"kind": kind}
    if kind in ("head", "step"):
        c["dtype"] = rng.choice(["f32", "bf16", "bf16"])
        if c["dtype"] == "f32":
            c["h"] = rng.choice([96, 256, 515, 1024])
            c["V"] = _log_int(rng, 1000, 32000)
            c["N"] = _log_int(rng, 64, 4096)
        else:
            c["h"], c["V"] = HEADS[rng.choice(["small", "moe", "long", "large"])]
            most = 1.2e14 / (6.0 * c["h"] * c["V"])  # no more than the moe step
            c["N"] = _log_int(rng, 64, int(min(65536, most)))
        c["obs"] = rng.choice([0.0, 0.25, 0.4])
        if kind == "head":
            c["path"] = rng.choice(["recompute", "recompute", "score"] + (["cached"] if c["dtype"] == "bf16" else []))
            if c["path"] == "cached":
                c["N"] = min(c["N"], 16384)
            c["accumulate"] = rng.random() < 0.3
        else:
            c.update(median=_log_int(rng, 64, 8192), lam=rng.choice([1.0, 0.95]), alpha=rng.choice([0.0, 0.0, 1.5]),
                     eps_low=0.3, eps_high=5.0)
        return c
    c["N"] = _log_int(rng, 1000, 1 << 25)
    c["median"] = _log_int(rng, 256, 65536)
    c["obs"] = rng.choice([0.0, 0.25, 0.4])
    if kind == "tokens":
        c.update(lam=rng.choice([1.0, 0.95, 0.95]), alpha=rng.choice([0.0, 0.0, 1.5]), eps_low=0.3, eps_high=5.0)
    elif kind == "turns":
        c["N"] = min(c["N"], 1 << 24)
        c.update(lam=rng.choice([1.0, 0.95]), alpha=rng.choice([0.0, 1.5]), mode=rng.choice(["average", "last"]))
    elif kind == "grpo":
        c.update(group=rng.choice([4, 8, 16]), eps_low=0.2, eps_high=0.28)
    else:
        c.update(prompts=rng.choice([1, 64, 1024]), window=rng.choice([8, 128]), eps_low=0.2, eps_high=0.28)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float32)


def _cu(seed, N, median):
    """Packed offsets of lognormal(median, sigma 1) trajectories of at most 131,072 tokens, N tokens in all."""
    rng = np.random.Generator(np.random.PCG64(seed))
    ends, at = [], 0
    while at < N:
        x = np.clip(rng.lognormal(math.log(max(median, 16)), 1.0, 64 + N // max(median, 16)), 16, 131072)
        e = at + np.cumsum(x.astype(np.int64))
        ends.append(e)
        at = int(e[-1])
    e = np.concatenate(ends)
    e = np.concatenate([[0], e[e < N], [N]])
    return torch.from_numpy(e.astype(np.int32)).to(DEV)


def _mask(g, N, obs):
    """Alternating turns: geometric action spans (mean 256 tokens) and observation spans, `obs` of all tokens."""
    if obs == 0.0:
        return torch.ones(N, dtype=torch.uint8, device=DEV)
    mean_obs = 256.0 * obs / (1.0 - obs)
    m = torch.empty(0, dtype=torch.uint8, device=DEV)
    while m.numel() < N:
        k = 64 + int(1.1 * N / (256.0 + mean_obs))
        spans = torch.empty(k, 2, device=DEV)
        spans[:, 0].geometric_(1.0 / 256.0, generator=g)
        spans[:, 1].geometric_(1.0 / max(mean_obs, 1.0), generator=g)
        kind = torch.tensor([1, 0], dtype=torch.uint8, device=DEV).repeat(k)
        m = torch.cat([m, torch.repeat_interleave(kind, spans.reshape(-1).long())])
    return m[:N].contiguous()


def _staleness(g, N, case):
    """Log-ratio of the policy to the stale rollout policy: N(0, 0.05 k), k in 1..4 versions old, a tenth of the
    tokens pushed past a clip bound. Ratios within 3 % of a bound are moved off it: there one rounding decides whether
    a token is kept, and a token kept by one correct implementation and dropped by another says nothing."""
    k = torch.randint(1, 5, (N,), generator=g, device=DEV).float()
    d = _randn(g, N) * 0.05 * k
    push = _rand(g, N) < 0.10
    far = torch.where(_rand(g, N) < 0.5, math.log1p(case["eps_high"]) + 0.2 + 0.3 * _rand(g, N),
                      math.log(max(1.0 - case["eps_low"], 0.05)) - 0.2 - 0.3 * _rand(g, N))
    d = torch.where(push, far, d)
    for b in (math.log1p(case["eps_high"]), math.log(max(1.0 - case["eps_low"], 0.05))):
        d = torch.where((d - b).abs() < 0.03, torch.full_like(d, b + math.copysign(0.06, b)), d)
    return d


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, dtype=dtype, device=DEV)


def _dense(g, case):
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    H = _randn(g, case["N"], case["h"]).to(dt)
    W = (_randn(g, case["V"], case["h"]) * 0.02).to(dt)
    y = torch.randint(0, case["V"], (case["N"],), generator=g, device=DEV, dtype=torch.int32)
    return H, W, y


def _rough_logp(H, W, y):
    """Sampled tokens' log-probs for weights drawn from N(0, 0.02): close enough to place the stale log-probs."""
    out = _empty(H.shape[0])
    for i in range(0, H.shape[0], 8192):
        h, w = H[i:i + 8192].float(), W[y[i:i + 8192].long()].float()
        out[i:i + 8192] = (h * w).sum(1) - math.log(W.shape[0]) - 0.0002 * h.square().sum(1)
    return out


def _prepare_head(case, g, s):
    N, h, V = case["N"], case["h"], case["V"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s["H"], s["W"], s["y"] = _dense(g, case)
    s["mask"] = _mask(g, N, case["obs"])
    s["rows"] = s["mask"] if case["obs"] > 0 else None
    # d loss / d log-prob of action tokens; one in a hundred is masked by the clip bounds
    grad = -_randn(g, N) * 0.5 / N * s["mask"] * (_rand(g, N) > 0.01)
    s["G"] = (grad + 0.0).contiguous()
    s["logp"], s["lse"] = _empty(N), _empty(N)
    s["ws"] = sao.workspace(N, h, V, dt)
    if case["path"] != "score":
        s["dH"] = torch.empty_like(s["H"])
        s["dW"] = torch.zeros(V, h, device=DEV)
    if case["path"] == "cached":
        s["cache"] = sao.logprob_cache(N, V)


def _prepare_tokens(case, g, s):
    N = case["N"]
    s["cu"] = _cu(s["seed"], N, case["median"])
    B = s["cu"].numel() - 1
    s["mask"] = _mask(g, N, case["obs"])
    s["values"] = _randn(g, N) * 0.2 + 0.4
    s["rewards"] = (_rand(g, B) < 0.4).float()
    s["adv"], s["ret"] = _empty(N), _empty(N)
    return B


def _prepare_losses(case, g, s):
    N = case["N"]
    s["loss"], s["vloss"] = _empty(1), _empty(1)
    s["one"] = torch.ones(1, device=DEV)
    s["coef"], s["flags"], s["G"] = _empty(N), _empty(N, dtype=torch.uint8), _empty(N)
    s["counts"] = _empty(6 if case["kind"] == "running" else 4, dtype=torch.int64)
    s["gv"], s["ev"] = _empty(N), _empty(4, dtype=F64)


def prepare(case, seed):
    g = _gen(seed)
    s = {"case": case, "seed": seed}
    kind, N = case["kind"], case["N"]
    if kind == "head":
        _prepare_head(case, g, s)
        return s
    B = _prepare_tokens(case, g, s)
    if kind == "step":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        s["H"], s["W"], s["y"] = _dense(g, case)
        s["old"] = _rough_logp(s["H"], s["W"], s["y"]) - _staleness(g, N, case)
        s["logp"], s["lse"] = _empty(N), _empty(N)
        s["dH"], s["dW"] = torch.empty_like(s["H"]), _empty(case["V"], case["h"])
        s["rows"] = s["mask"] if case["obs"] > 0 else None
        s["ws"] = sao.workspace(N, case["h"], case["V"], dt)
        _prepare_losses(case, g, s)
        return s
    s["ws"] = sao.workspace(N)
    if kind == "turns":
        s["vmask"] = _empty(N, dtype=torch.uint8)
        return s
    s["logp"] = torch.empty(N, device=DEV).exponential_(0.5, generator=g).neg_()
    s["old"] = s["logp"] - _staleness(g, N, case)
    _prepare_losses(case, g, s)
    if kind == "grpo":
        # a prompt's rollouts lie together in the batch
        s["gid"] = (torch.arange(B, device=DEV) // case["group"]).to(torch.int32)
    elif kind == "running":
        s["pid"] = torch.randint(0, case["prompts"], (B,), generator=g, device=DEV, dtype=torch.int32)
        s["history"] = (_rand(g, case["prompts"], case["window"]) < 0.4).float()
        s["seen"] = torch.randint(0, 3 * case["window"], (case["prompts"],), generator=g, device=DEV)
        # training engine against rollout engine: a small mismatch, a few tokens outside the band (0.5, 2)
        e = _randn(g, N) * 0.05
        e = torch.where(_rand(g, N) < 0.01, torch.full_like(e, 0.9), e)
        s["prox"] = s["old"]
        s["rollout"] = s["prox"] - e
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

LAM_CRITIC, GAMMA = 1.0, 1.0
EPS_STAB = 1e-6
W_LOW, W_HIGH = 0.5, 2.0


def _advantages(s):
    c = s["case"]
    sao.sao_advantages(s["values"], s["rewards"], s["mask"], s["cu"], GAMMA, c["lam"], LAM_CRITIC, c["alpha"],
                       s["adv"], s["ret"], s["ws"])


def _policy(s):
    c = s["case"]
    sao.sao_policy_loss_fwd(s["logp"], s["old"], s["adv"], s["mask"], c["eps_low"], c["eps_high"], s["loss"],
                            s["counts"], s["ws"], coef=s["coef"], flags=s["flags"])
    sao.sao_policy_loss_bwd(s["logp"], s["old"], s["adv"], s["mask"], c["eps_low"], c["eps_high"], s["one"], s["G"],
                            s["ws"])


def _value(s):
    sao.sao_value_loss(s["values"], s["ret"], s["mask"], s["vloss"], s["gv"], s["ws"], ev_sums=s["ev"])


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "head":
        if c["path"] == "cached":
            sao.sao_token_logprobs_fwd_cached(s["H"], s["W"], s["y"], s["logp"], s["lse"], s["cache"], s["ws"],
                                              row_mask=s["rows"])
            sao.sao_token_logprobs_bwd_cached(s["H"], s["W"], s["y"], s["lse"], s["G"], s["dH"], s["dW"], s["cache"],
                                              s["ws"], accumulate_dW=c["accumulate"])
        else:
            sao.sao_token_logprobs_fwd(s["H"], s["W"], s["y"], s["logp"], s["lse"], s["ws"], row_mask=s["rows"])
            if c["path"] == "score":
                return {"logp": s["logp"], "lse": s["lse"]}
            sao.sao_token_logprobs_bwd(s["H"], s["W"], s["y"], s["lse"], s["G"], s["dH"], s["dW"], s["ws"],
                                       accumulate_dW=c["accumulate"])
        return {"logp": s["logp"], "lse": s["lse"], "dH": s["dH"], "dW": s["dW"]}
    if kind == "turns":
        mode = sao.SAO_STEP_AVERAGE if c["mode"] == "average" else sao.SAO_STEP_LAST
        sao.sao_step_advantages(s["values"], s["rewards"], s["mask"], s["cu"], GAMMA, c["lam"], LAM_CRITIC,
                                c["alpha"], mode, s["adv"], s["ret"], s["ws"], value_mask=s["vmask"])
        return {"adv": s["adv"], "ret": s["ret"], "value_mask": s["vmask"]}
    losses = {k: s[k] for k in ("adv", "loss", "coef", "flags", "counts", "G")}
    if kind == "grpo":
        sao.sao_group_advantages(s["rewards"], s["gid"], s["mask"], s["cu"], EPS_STAB, s["adv"], s["ws"])
        sao.sao_clip_loss_fwd(s["logp"], s["old"], s["adv"], s["mask"], s["cu"], c["eps_low"], c["eps_high"],
                              sao.SAO_NORM_SEQUENCE, s["loss"], s["counts"], s["ws"], coef=s["coef"],
                              flags=s["flags"])
        sao.sao_clip_loss_bwd(s["logp"], s["old"], s["adv"], s["mask"], s["cu"], c["eps_low"], c["eps_high"],
                              sao.SAO_NORM_SEQUENCE, s["one"], s["G"], s["ws"])
        return losses
    if kind == "running":
        sao.sao_running_mean_advantages(s["rewards"], s["pid"], s["history"], s["seen"], s["mask"], s["cu"],
                                        s["adv"], s["ws"])
        sao.sao_decoupled_loss_fwd(s["logp"], s["prox"], s["rollout"], s["adv"], s["mask"], c["eps_low"],
                                   c["eps_high"], W_LOW, W_HIGH, s["loss"], s["counts"], s["ws"], coef=s["coef"],
                                   flags=s["flags"])
        sao.sao_decoupled_loss_bwd(s["logp"], s["prox"], s["rollout"], s["adv"], s["mask"], c["eps_low"],
                                   c["eps_high"], W_LOW, W_HIGH, s["one"], s["G"], s["ws"])
        return {**losses, "history": s["history"], "seen": s["seen"]}
    _advantages(s)
    if kind == "step":
        sao.sao_token_logprobs_fwd(s["H"], s["W"], s["y"], s["logp"], s["lse"], s["ws"], row_mask=s["rows"])
    _policy(s)
    if kind == "step":
        sao.sao_token_logprobs_bwd(s["H"], s["W"], s["y"], s["lse"], s["G"], s["dH"], s["dW"], s["ws"])
    _value(s)
    out = {**losses, "ret": s["ret"], "value_loss": s["vloss"], "grad_values": s["gv"], "ev_sums": s["ev"]}
    if kind == "step":
        out.update(logp=s["logp"], lse=s["lse"], dH=s["dH"], dW=s["dW"])
    return out


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------

def work(case):
    N, kind = case["N"], case["kind"]
    act = N * (1.0 - case["obs"])
    by = fl = 0.0
    if kind in ("head", "step"):
        e = 2 if case["dtype"] == "bf16" else 4
        h, V = case["h"], case["V"]
        by += e * (act * h + V * h) + 4 * N + 8 * N  # H, W, y in; logp, lse out
        fl += 2.0 * act * h * V
        if case.get("path") != "score":
            by += 4 * N + e * N * h + 4.0 * V * h * (2 if case.get("accumulate") else 1)  # G in; dH, dW out
            fl += 4.0 * act * h * V
    if kind in ("step", "tokens"):
        # each array once: values, mask, log-probs (a step's own stay on the chip's side of the call), advantages,
        # returns, coefficients, flags, gradients
        by += N * (4 + 1 + 4 + 4 + 4 + 4 + 4 + 1 + 4 + 4)
        fl += 40.0 * N
    elif kind == "turns":
        by += N * (4 + 1 + 4 + 4 + 1)
        fl += 4.0 * N
    elif kind == "grpo":
        by += N * (1 + 4 + 4 + 4 + 4 + 1 + 4)
        fl += 20.0 * N
    elif kind == "running":
        by += N * (1 + 4 + 4 + 4 + 4 + 4 + 1 + 4)
        fl += 25.0 * N
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    if case.get("path") == "score" and case["dtype"] == "bf16":
        # exact bf16 products, fp32 sums over h: 1.4e-6 from fp64 at h = 6144
        return {"rel": 6e-6, "max": 6e-5}
    if case.get("dtype") == "bf16":
        # dZ (or the stored probabilities) and dH are rounded to bf16: 2.3e-3 from fp64
        return {"rel": 1e-2, "max": 0.2}
    if case.get("dtype") == "f32":
        # fp32 sums over up to 32,000 terms: 3.2e-6 from fp64
        return {"rel": 1.2e-5, "max": 5e-4}
    # fp32 per token, sums in more than fp32: 5.6e-7 from fp64 (a clipped loss near zero)
    return {"rel": 2e-6, "max": 2e-5}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

MOST_FLOPS = 9e12  # fp64 products that take a few seconds on this GPU


def _exact_head(s, G, want_grad):
    """log-probs, lse and (want_grad) dH, dW in fp64, vocabulary chunk by chunk; None for what would take too long."""
    H, W, y = s["H"], s["W"], s["y"].long()
    N, h = H.shape
    V = W.shape[0]
    out = {"logp": None, "lse": None, "dH": None, "dW": None}
    if 2.0 * N * h * V > MOST_FLOPS:
        return out
    Hd = H.to(F64)
    step = max(1, min(V, (1 << 28) // max(N, 1)))
    lse = torch.full((N,), -math.inf, dtype=F64, device=DEV)
    zy = torch.zeros(N, dtype=F64, device=DEV)
    for v in range(0, V, step):
        z = Hd @ W[v:v + step].to(F64).t()
        lse = torch.logaddexp(lse, torch.logsumexp(z, 1))
        here = ((y >= v) & (y < v + step)).nonzero().squeeze(1)
        zy[here] = z[here, y[here] - v]
    rows = s["rows"].bool() if s["rows"] is not None else torch.ones(N, dtype=torch.bool, device=DEV)
    zero = torch.zeros((), dtype=F64, device=DEV)
    out["logp"], out["lse"] = torch.where(rows, zy - lse, zero), torch.where(rows, lse, zero)
    if want_grad and G is not None and 8.0 * N * h * V <= MOST_FLOPS:
        Gd = G.to(F64)
        dH = torch.zeros(N, h, dtype=F64, device=DEV)
        dW = torch.empty(V, h, dtype=F64, device=DEV)
        for v in range(0, V, step):
            Wd = W[v:v + step].to(F64)
            dz = torch.exp(Hd @ Wd.t() - lse[:, None]).mul_(-Gd[:, None])
            here = ((y >= v) & (y < v + step)).nonzero().squeeze(1)
            dz[here, y[here] - v] += Gd[here]
            dH += dz @ Wd
            dW[v:v + step] = dz.t() @ Hd
        out["dH"], out["dW"] = dH, dW
    return out


def _affine_back(c, m):
    """x[j] = c[j] + m[j] x[j + 1] (m = 0 where a chain ends), by doubling."""
    c, m, d, n = c.clone(), m.clone(), 1, c.numel()
    while d < n and bool(m.any()):
        c[:n - d] += m[:n - d] * c[d:]
        m = torch.cat([m[:n - d] * m[d:], torch.zeros(d, dtype=F64, device=DEV)])
        d *= 2
    return c


def _traj(s):
    cu = s["cu"].long()
    return torch.repeat_interleave(torch.arange(cu.numel() - 1, device=DEV), cu[1:] - cu[:-1])


def _gae(V, b, s, lam, alpha, n_of):
    """Advantages of the units (tokens or turns) with values V, in order, of trajectory b; n_of: units per trajectory."""
    last = torch.ones(V.numel(), dtype=torch.bool, device=DEV)
    last[:-1] = b[1:] != b[:-1]
    nxt = torch.zeros_like(V)
    nxt[:-1] = V[1:]
    nxt[last] = 0
    delta = torch.where(last, s["rewards"].to(F64)[b], torch.zeros_like(V)) + GAMMA * nxt - V
    lam64 = float(np.float32(lam))
    if alpha > 0:
        l = (1.0 - 1.0 / (alpha * n_of.to(F64).clamp(min=1))).clamp(0, 1)[b]
    else:
        l = torch.full_like(V, lam64)
    return _affine_back(delta, torch.where(last, torch.zeros_like(V), GAMMA * l))


def _exact_advantages(s):
    c, N = s["case"], s["case"]["N"]
    idx = s["mask"].bool().nonzero().squeeze(1)
    b = _traj(s)[idx]
    V = s["values"].to(F64)[idx]
    n_of = torch.bincount(b, minlength=s["rewards"].numel())
    adv, ret = torch.zeros(N, dtype=F64, device=DEV), torch.zeros(N, dtype=F64, device=DEV)
    adv[idx] = _gae(V, b, s, c["lam"], c["alpha"], n_of)
    ret[idx] = _gae(V, b, s, LAM_CRITIC, 0.0, n_of) + V
    return adv, ret


def _exact_turns(s):
    c, N = s["case"], s["case"]["N"]
    t, m = _traj(s), s["mask"].bool()
    start = m.clone()
    start[1:] &= ~m[:-1] | (t[1:] != t[:-1])
    turn = torch.cumsum(start.long(), 0) - 1
    idx = m.nonzero().squeeze(1)
    k = int(start.sum())
    of = turn[idx]
    n_tok = torch.bincount(of, minlength=k)
    val = s["values"].to(F64)[idx]
    end = torch.ones(idx.numel(), dtype=torch.bool, device=DEV)
    end[:-1] = of[1:] != of[:-1]
    if c["mode"] == "average":
        V = torch.zeros(k, dtype=F64, device=DEV).index_add_(0, of, val) / n_tok
        vm = m.to(torch.uint8)
    else:
        V = val[end]
        vm = torch.zeros(N, dtype=torch.uint8, device=DEV)
        vm[idx[end]] = 1
    b = t[start.nonzero().squeeze(1)]
    n_of = torch.bincount(b, minlength=s["rewards"].numel())
    adv, ret = torch.zeros(N, dtype=F64, device=DEV), torch.zeros(N, dtype=F64, device=DEV)
    adv[idx] = _gae(V, b, s, c["lam"], c["alpha"], n_of)[of]
    ret[idx] = (_gae(V, b, s, LAM_CRITIC, 0.0, n_of) + V)[of]
    return {"adv": adv, "ret": ret, "value_mask": vm}


def _bounds(c):
    return float(np.float32(1.0) - np.float32(c["eps_low"])), float(np.float32(1.0) + np.float32(c["eps_high"]))


def _exact_policy(s, adv):
    lo, hi = _bounds(s["case"])
    m = s["mask"].bool()
    r = torch.exp(s["logp"].to(F64) - s["old"].to(F64))
    low, high = r <= lo, r >= hi
    kept = m & ~low & ~high
    n = int(m.sum())
    f = torch.where(kept, r * adv, torch.zeros_like(r))
    flags = torch.where(low, 1, torch.where(high, 2, 0))
    flags = torch.where(m, flags, 4).to(torch.uint8)
    counts = torch.tensor([n, int((m & low).sum()), int((m & high).sum()), 0], device=DEV)
    return {"loss": -f.sum().reshape(1) / n, "coef": -f / n, "flags": flags, "counts": counts, "G": -f / n}


def _exact_value(s, ret):
    m = s["mask"].bool()
    n = int(m.sum())
    v, r = s["values"].to(F64), ret
    zero = torch.zeros_like(v)
    d = torch.where(m, v - r, zero)
    rm = torch.where(m, r, zero)
    return {"value_loss": d.square().sum().reshape(1) / n, "grad_values": 2 * d / n,
            "ev_sums": torch.stack([-d.sum(), d.square().sum(), rm.sum(), rm.square().sum()])}


def _clipped(s, adv, r, weight):
    lo, hi = _bounds(s["case"])
    m = s["mask"].bool()
    high, low = (adv > 0) & (r > hi), (adv < 0) & (r < lo)
    f = torch.where(high, torch.full_like(r, hi), torch.where(low, torch.full_like(r, lo), r)) * adv * weight
    f = torch.where(m, f, torch.zeros_like(f))
    return m, low, high, f


def _exact_grpo(s):
    c, N = s["case"], s["case"]["N"]
    t, m = _traj(s), s["mask"].bool()
    B, gid = s["rewards"].numel(), s["gid"].long()
    R = s["rewards"].to(F64)
    k = int(gid.max()) + 1
    n_g = torch.bincount(gid, minlength=k).to(F64)
    mean = torch.zeros(k, dtype=F64, device=DEV).index_add_(0, gid, R) / n_g
    var = torch.zeros(k, dtype=F64, device=DEV).index_add_(0, gid, (R - mean[gid]).square()) / n_g
    a = (R - mean[gid]) / torch.sqrt(var[gid] + float(np.float32(EPS_STAB)))
    zero = torch.zeros(N, dtype=F64, device=DEV)
    adv = torch.where(m, a[t], zero)
    n_t = torch.bincount(t[m], minlength=B)
    weight = 1.0 / (n_t.clamp(min=1).to(F64)[t] * int((n_t > 0).sum()))
    r = torch.exp(s["logp"].to(F64) - s["old"].to(F64))
    m, low, high, f = _clipped(s, adv, r, weight)
    coef = torch.where(low | high, zero, -f)
    flags = torch.where(m, torch.where(high, 2, torch.where(low, 1, 0)), 4).to(torch.uint8)
    counts = torch.tensor([int(m.sum()), int((m & low).sum()), int((m & high).sum()), 0], device=DEV)
    return {"adv": adv, "loss": -f.sum().reshape(1), "coef": coef, "flags": flags, "counts": counts, "G": coef}


def _exact_running(s):
    c, N = s["case"], s["case"]["N"]
    P, win = c["prompts"], c["window"]
    R, pid = s["rewards"].double().cpu().numpy(), s["pid"].cpu().numpy()
    hist, seen = s["history"].double().cpu().numpy().copy(), s["seen"].cpu().numpy().copy()
    a = np.empty(len(R))
    for b in range(len(R)):
        p = pid[b]
        n = min(int(seen[p]), win)
        a[b] = R[b] - (hist[p, :n].sum() / n if n else 0.0)
        hist[p, seen[p] % win] = R[b]
        seen[p] += 1
    t = _traj(s)
    zero = torch.zeros(N, dtype=F64, device=DEV)
    adv = torch.where(s["mask"].bool(), torch.from_numpy(a).to(DEV)[t], zero)
    w = torch.exp(s["prox"].to(F64) - s["rollout"].to(F64))
    r = torch.exp(s["logp"].to(F64) - s["prox"].to(F64))
    n = int(s["mask"].bool().sum())
    m, low, high, f = _clipped(s, adv, r, w / n)
    wl, wh = w <= W_LOW, w >= W_HIGH
    f = torch.where(wl | wh, zero, f)
    coef = torch.where(low | high, zero, -f)
    flags = torch.where(wl, 5, torch.where(wh, 6, torch.where(high, 2, torch.where(low, 1, 0))))
    flags = torch.where(m, flags, 4).to(torch.uint8)
    counts = torch.tensor([n, int((flags == 1).sum()), int((flags == 2).sum()), 0, int((flags == 5).sum()),
                           int((flags == 6).sum())], device=DEV)
    return {"adv": adv, "loss": -f.sum().reshape(1), "coef": coef, "flags": flags, "counts": counts, "G": coef,
            "history": torch.from_numpy(hist).float().to(DEV), "seen": torch.from_numpy(seen).to(DEV)}


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "head":
        out = _exact_head(s, s["G"], case["path"] != "score")
        return {k: out[k] for k in (("logp", "lse") if case["path"] == "score" else ("logp", "lse", "dH", "dW"))}
    if kind == "turns":
        return _exact_turns(s)
    if kind == "grpo":
        return _exact_grpo(s)
    if kind == "running":
        return _exact_running(s)
    adv, ret = _exact_advantages(s)
    out = {"adv": adv, "ret": ret, **_exact_value(s, ret)}
    if kind == "tokens":
        return {**out, **_exact_policy(s, adv)}
    head = _exact_head(s, None, False)
    policy = dict.fromkeys(("loss", "coef", "flags", "counts", "G"))
    if head["logp"] is not None:
        s["logp"] = head["logp"]
        policy = _exact_policy(s, adv)
        head = _exact_head(s, policy["G"], True)
    return {**out, **policy, **head}
