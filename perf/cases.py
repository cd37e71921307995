"""The calls whose speed is measured: the fused loss, its split, chunked,
graphed, forward-only and vocabulary-sharded forms, through the package's
public entry points, on the repository's own synthetic batches.

A case names a recipe of ``workloads.RECIPES`` (which sets the temperature,
clips, coefficients, rewards and mask) and what of it is changed: the number
of prompts, attempts per prompt and tokens per attempt, the vocabulary, the
data type, the estimator, the correction and the way the call is made
(``mode``):

  fused    rl_loss_fwd_bwd, called as it is
  graph    the same, captured once and replayed
  split    rl_loss_fwd, then rl_loss_bwd
  fwd      rl_loss_fwd alone (scoring)
  chunked  rl_loss_fwd_bwd_rows over blocks of rows
  vshard   two column shards of the vocabulary, driven from one process
"""

from __future__ import annotations

from dataclasses import replace

import torch

from paper_2609_08368_gb300 import api, workloads

DEVICE = "cuda"
CHUNK_ROWS = 4096         # rows per block of a chunked call (the benchmark's)
MOST_BYTES = 8 << 30      # of a drawn case's logits
EXACT_ELEMENTS = 3 << 30  # dLogits past this many elements are not formed in 64 bits


def _case(name, recipe, mode, n_prompts, group, traj_len, vocab, dtype="bf16", estimator="grpo",
          topk=0, correction="none"):
    return dict(name=name, recipe=recipe, mode=mode, n_prompts=n_prompts, group=group,
                traj_len=traj_len, vocab=vocab, dtype=dtype, estimator=estimator, topk=topk,
                correction=correction)


def listed():
    return [
        # the smallest training call, made eagerly: host work, launches and latency
        _case("tiny_fused", "tiny", "fused", 2, 4, 256, 4096),
        # the same call captured in a graph by a program that repeats it
        _case("tiny_graph", "tiny", "graph", 2, 4, 256, 4096),
        # one short micro-batch of a large vocabulary: few rows per SM
        _case("micro_graph", "glm", "graph", 1, 4, 80, 154880),
        # a training batch with group-relative advantages over a 152K vocabulary
        _case("qwen_fused", "qwen", "fused", 16, 8, 128, 151936),
        # the headline batch: KL term, dual clip
        _case("glm_fused", "glm", "fused", 4, 16, 1024, 154880),
        # long agentic sessions with masked tool output, logits made a block of rows at a time
        _case("agentic_chunked", "agentic", "chunked", 1, 4, 8192, 151936),
        # fp32 logits, entropy bonus, equal-reward groups
        _case("fp32_fused", "fp32", "fused", 64, 8, 64, 32768, "f32"),
        # the sequence-level ratio: forward, per-trajectory pass, gradient
        _case("gspo_fused", "qwen", "fused", 8, 8, 128, 151936, estimator="gspo"),
        # forward and backward as separate calls, with a ratio correction
        _case("split_tis", "qwen", "split", 8, 8, 96, 65536, correction="tis"),
        # a vocabulary that no padding rounds up: rows start on any element
        _case("ragged_fused", "glm", "fused", 4, 16, 64, 45003),
        # two tensor-parallel shards of a batch
        _case("vshard_tp2", "glm", "vshard", 2, 8, 256, 154880),
        # scoring a batch under a small vocabulary: log-probs and entropies only
        _case("score_fwd", "glm", "fwd", 8, 16, 128, 20480),
    ]


def _log_uniform(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """One more case: rows from 64 to 65,536, vocabularies from 2,048 to
    262,144 (half of them padded to a multiple of 128, as trainers pad; a
    quarter to whole 16-byte vectors; a quarter not at all), every mode, both
    data types, the estimators, corrections and top-K distillation."""
    recipe = rng.choice(["qwen", "glm", "agentic", "fp32"])
    mode = rng.choice(["fused"] * 6 + ["graph", "split", "split", "fwd", "fwd", "chunked", "vshard"])
    dtype = "f32" if recipe == "fp32" else "bf16"
    es = 4 if dtype == "f32" else 2
    vocab = int(_log_uniform(rng, 2048, 262144))
    step = rng.choice([128, 128, 8, 1])
    vocab = vocab // step * step
    rows = min(_log_uniform(rng, 64, 65536), MOST_BYTES / (vocab * es))
    group = rng.choice([4, 8, 16])
    n_prompts = max(1, min(64, int(_log_uniform(rng, 1, max(1.01, rows / (group * 8))))))
    traj_len = max(2, int(rows / (group * n_prompts)))
    extra = rng.random()
    estimator, topk, correction = "grpo", 0, "none"
    if extra < 0.12 and mode in ("fused", "split", "fwd"):
        estimator = "gspo"
    elif extra < 0.24:
        topk = rng.choice([8, 16, 32])
    elif extra < 0.34:
        correction = rng.choice(["tis", "clip_or_pop"])
    elif extra < 0.42:
        estimator = rng.choice(["reinforcepp", "reinforcepp_baseline"])
    c = _case("", recipe, mode, n_prompts, group, traj_len, vocab, dtype, estimator, topk, correction)
    del c["name"]
    return c


def _recipe(case, seed):
    base = workloads.RECIPES[case["recipe"]]
    params = dict(base.params, estimator=case["estimator"], correction=case["correction"])
    if case["topk"]:
        params.update(opd_topk=case["topk"], opd_coef=0.1)
    return replace(base, n_prompts=case["n_prompts"], group_size=case["group"],
                   traj_len=case["traj_len"], vocab=case["vocab"], dtype=case["dtype"],
                   topk=case["topk"], params=params, seed=1 + int(seed))


def _stats(raw):
    """The statistics' fields as tensors on the raw bytes the call writes."""
    return dict(means=raw[:72].view(torch.float64), ratio_range=raw[72:80].view(torch.float32),
                counts=raw[80:120].view(torch.int64))


def prepare(case, seed):
    w = workloads.make(_recipe(case, seed), DEVICE)
    n_traj, R, V = int(w.rewards.shape[0]), w.n_rows, w.vocab
    mode = case["mode"]
    if mode == "vshard":
        cut = V // 2 // 8 * 8
        cols, shards = [0, cut, V], []
        for k in range(2):
            wk = replace(w, logits=w.logits[:, cols[k]:cols[k + 1]].contiguous())
            buf = api.alloc(R, n_traj, w.n_groups, DEVICE, vocab=cols[k + 1] - cols[k],
                            dlogits_dtype=w.logits.dtype)
            shards.append(api.VocabShard(wk, k, cols, buf))
        bufs = [s.buf for s in shards]
        out = dict(_stats(bufs[0].stats), logp=bufs[0].token_logprobs, entropy=bufs[0].entropy,
                   advantages=bufs[0].advantages, group_sizes=bufs[0].group_sizes,
                   dlogits=[b.dlogits for b in bufs])
        return dict(call=lambda: api.vocab_sharded_fwd_bwd_local([shards]), out=out)
    buf = api.alloc(R, n_traj, w.n_groups, DEVICE, vocab=V,
                    dlogits_dtype=None if mode == "fwd" else w.logits.dtype)
    out = dict(_stats(buf.stats), logp=buf.token_logprobs, entropy=buf.entropy,
               advantages=buf.advantages, group_sizes=buf.group_sizes)
    if mode != "fwd":
        out["dlogits"] = buf.dlogits
    if mode == "fused":
        call = lambda: api.fwd_bwd(w, buf)
    elif mode == "graph":
        call = api.GraphedCall(w, buf)
        keep = (w, buf)
        return dict(call=call, out=out, keep=keep)
    elif mode == "split":
        def call():
            api.fwd(w, buf)
            api.bwd(w, buf)
    elif mode == "fwd":
        call = lambda: api.fwd(w, buf)
    elif case["estimator"] == "gspo":
        raise ValueError("a chunked call takes no GSPO")
    else:
        call = lambda: api.fwd_bwd_chunked(w, buf, CHUNK_ROWS)
    return dict(call=call, out=out)


def run(state):
    state["call"]()
    return state["out"]


def _sizes(case):
    n_traj = case["n_prompts"] * case["group"]
    return n_traj, n_traj * case["traj_len"], case["vocab"], 4 if case["dtype"] == "f32" else 2


def work(case):
    """The logits read once and dLogits written once; the per-row inputs
    (target, mask, rollout and reference log-probs, candidates) and outputs.
    Per logit: scale, exponential, two sums; scale, exponential, product."""
    n_traj, R, V, es = _sizes(case)
    grad = case["mode"] != "fwd"
    per_row = 4 + 1 + 4 + 4 + 8 * case["topk"] + 8
    return {"bytes": R * V * es * (2 if grad else 1) + R * per_row + n_traj * 20 + 120,
            "flops": R * V * (8 if grad else 5)}


def tolerance(case):
    """bf16 dLogits: two roundings to 8 bits that fall on either side (against
    64 bits 1.7e-3 of the norm was measured, 3.9e-3 of a value). fp32: the
    order of the row sums and the exponential's last bits (1e-6 measured)."""
    if case["dtype"] == "bf16" and case["mode"] != "fwd":
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 1e-5, "max": 1e-4}


# --------------------------------------------------------------- in 64 bits

def _advantages(w, p, n_tok):
    f64 = torch.float64
    rew, gid = w.rewards.to(f64), w.group_id.long()
    n = torch.zeros(w.n_groups, dtype=f64, device=DEVICE).index_add_(0, gid, torch.ones_like(rew))
    mu = torch.zeros_like(n).index_add_(0, gid, rew) / n.clamp(min=1)
    floor = p.get("std_floor", 1e-6)
    est = p["estimator"]
    if est in ("grpo", "gspo"):
        d = rew - mu[gid]
        ss = torch.zeros_like(n).index_add_(0, gid, d * d)
        hi = torch.full_like(n, -float("inf")).scatter_reduce_(0, gid, rew, "amax")
        lo = torch.full_like(n, float("inf")).scatter_reduce_(0, gid, rew, "amin")
        den = (ss / (n - 1).clamp(min=1)).sqrt().clamp(min=floor)
        return torch.where((hi == lo)[gid], torch.zeros_like(d), d / den[gid]), n
    b = rew if est == "reinforcepp" else rew - mu[gid]
    N = n_tok.sum()
    m = (b * n_tok).sum() / N
    std = (((b - m) ** 2 * n_tok).sum() / (N - 1)).sqrt().clamp(min=floor)
    trains = b[n_tok > 0]
    if trains.numel() == 0 or bool(trains.max() == trains.min()):
        return torch.zeros_like(b), n
    return (b - m) / std, n


def exact(case, seed):
    f64 = torch.float64
    w = workloads.make(_recipe(case, seed), DEVICE)
    p, (n_traj, R, V, _) = w.params, _sizes(case)
    invT = 1.0 / float(p.get("temperature", 1.0))
    gamma, beta = p.get("entropy_coef", 0.0), p.get("kl_coef", 0.0)
    lo_c, hi_c = 1.0 - p["eps_lo"], 1.0 + p["eps_hi"]
    traj = torch.arange(n_traj, device=DEVICE).repeat_interleave(case["traj_len"])
    m = (w.loss_mask != 0).to(f64)
    n_tok = torch.zeros(n_traj, dtype=f64, device=DEVICE).index_add_(0, traj, m)
    A, sizes = _advantages(w, p, n_tok)
    N = float(m.sum())
    step = max(1, (1 << 27) // V)
    y = w.targets.long()

    # row statistics, a block of rows at a time
    logp, H, lse = (torch.empty(R, dtype=f64, device=DEVICE) for _ in range(3))
    opd = torch.zeros(R, dtype=f64, device=DEVICE)
    for r0 in range(0, R, step):
        r = slice(r0, min(R, r0 + step))
        s = w.logits[r].to(f64) * invT
        lse[r] = torch.logsumexp(s, 1)
        logp[r] = s.gather(1, y[r, None])[:, 0] - lse[r]
        if case["topk"]:
            z = s.gather(1, w.topk_ids[r].long())
            opd[r] = (torch.softmax(z, 1) * (z - lse[r, None] - w.topk_teacher[r].to(f64))).sum(1)
        s -= lse[r, None]
        H[r] = -(s.exp() * s).sum(1)

    # the per-token objective
    rho = w.rollout_logprobs.to(f64)
    rows_A = A[traj] - p.get("opd_coef", 0.0) * opd
    ratio = (logp - rho).exp()

    def weight(rc):
        lo, hi = p.get("corr_lo", 0.0), p.get("corr_hi", 2.0)
        if case["correction"] == "tis":
            return rc.clamp(lo, hi)
        if case["correction"] == "clip_or_pop":
            return torch.where((rc < lo) | (rc > hi), torch.zeros_like(rc), rc)
        return torch.ones_like(rc)

    rc = ratio if case["correction"] != "none" else torch.ones_like(ratio)
    wt = weight(rc)
    c_lo, c_hi = p.get("corr_lo", 0.0), p.get("corr_hi", 2.0)
    pops = ((rc < c_lo) | (rc > c_hi)) & (case["correction"] != "none")

    def policy(r, adv):
        u, c = -adv * r, -adv * r.clamp(lo_c, hi_c)
        cut = c > u
        pg, dual = torch.maximum(u, c), torch.zeros_like(cut)
        if p.get("dual_clip_c", 0.0) > 0:
            cap = -adv * p["dual_clip_c"]
            dual = (adv < 0) & (cap < pg)
            pg = torch.where(dual, cap, pg)
        return pg, torch.where(cut | dual, torch.zeros_like(u), u), cut & (r > hi_c), cut & (r < lo_c), dual

    if p["estimator"] == "gspo":
        n = n_tok.clamp(min=1)
        mean = torch.zeros_like(n).index_add_(0, traj, m * (logp - rho)) / n
        mean_w = torch.zeros_like(n).index_add_(0, traj, m * wt) / n
        seq = mean.exp()
        pg, g, hi, lo, dual = policy(seq, A)
        scale = N / (float((n_tok > 0).sum()) * n)
        pg, G = (scale * pg)[traj] * wt, (scale * mean_w * g)[traj]
        hi, lo, dual, ratio = hi[traj], lo[traj], dual[traj], seq[traj]
    else:
        pg, G, hi, lo, dual = policy(ratio, rows_A)
        pg, G = pg * wt, G * wt
    k3 = torch.zeros_like(logp)
    if w.ref_logprobs is not None:
        d = w.ref_logprobs.to(f64) - logp
        k3 = torch.expm1(d) - d
        G = G - beta * torch.expm1(d)
    ell = pg + beta * k3 - gamma * H
    means = [(m * v).sum() / N for v in (ell, pg, k3, H, ratio, (ratio - 1).abs(), (logp - rho).abs(),
                                         rc, (rc - 1).abs())]
    on = m > 0
    out = dict(means=torch.stack(means), ratio_range=torch.stack([ratio[on].min(), ratio[on].max()]),
               counts=torch.stack([(on & v).sum() for v in (on, hi, lo, dual, pops)]), logp=logp,
               entropy=H, advantages=A, group_sizes=sizes.to(torch.int32))
    if case["mode"] == "fwd":
        return out
    if R * V > EXACT_ELEMENTS:
        out["dlogits"] = None
        return out
    dl = torch.empty((R, V), dtype=f64, device=DEVICE)
    for r0 in range(0, R, step):
        r = slice(r0, min(R, r0 + step))
        lp = w.logits[r].to(f64) * invT - lse[r, None]
        x = gamma * (lp + H[r, None]) - G[r, None]
        x *= lp.exp_()
        x.scatter_add_(1, y[r, None], G[r, None])
        dl[r] = x * (m[r, None] * (invT / N))
    if case["mode"] == "vshard":
        cut = V // 2 // 8 * 8
        out["dlogits"] = [dl[:, :cut], dl[:, cut:]]
    else:
        out["dlogits"] = dl
    return out
