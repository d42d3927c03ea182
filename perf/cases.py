"""The work that is timed when this library is made faster: calls of its public entry points at the sizes a trainer
runs them at, from the smallest micro-batch to the largest policy-update step.

Every case makes its own inputs from a seed: a batch of responses (right-padded or with masked observation spans),
hidden states whose logits run from flat to strongly peaked at the sampled token (a trained policy is sure of most of
its tokens), token ids with the skew of natural text, behaviour and reference log-probabilities near the policy's own.
"""
import math

import torch

from paper_2512_21450_b200 import Context

DEVICE = "cuda:0"


def listed():
    def case(name, kind, d, V, prompts, G, L_max, len_lo, w_std=0.02, **kw):
        return dict(dict(name=name, kind=kind, d=d, V=V, prompts=prompts, G=G, L_max=L_max, len_lo=len_lo, w_std=w_std,
                         eps_low=0.2, eps_high=0.2, beta=0.04, ent_coef=0.0, span=0.0, accumulate=False, agg_mode=0,
                         sequence_level=False), **kw)

    return [
        # the smallest update: a unit-test sized policy, where launches and host time are all there is
        case("tiny_step", "step", 256, 4096, 4, 4, 16, 16),
        # one micro-batch of gradient accumulation on a 3B-class head: a few hundred tokens added to dW
        case("micro_3b", "step", 2048, 151936, 1, 4, 160, 20, accumulate=True),
        # one prompt's group on a 7B-class head with the sequence-level ratio
        case("group_7b", "step", 3584, 152064, 1, 8, 512, 128, w_std=0.015, sequence_level=True),
        # an ordinary update of a 3B-class head (the benchmark's workload)
        case("step_3b", "step", 2048, 151936, 8, 8, 512, 64),
        # an update of a 7B-class head, continuous rewards
        case("step_7b", "step", 3584, 152064, 16, 8, 1024, 128, w_std=0.015),
        # long multi-turn rollouts: 30 % of the rows are tool output and take no part in the loss
        case("step_long", "step", 2560, 151936, 4, 8, 4096, 4096, span=0.3),
        # the largest update: asymmetric clip, no KL term, entropy bonus
        case("step_entropy", "step", 2048, 151936, 64, 16, 512, 32, eps_high=0.28, beta=0.0, ent_coef=1e-3),
        # scoring the tokens of one short turn
        case("score_turn", "score", 2560, 151936, 1, 1, 77, 77, models=1),
        # scoring a batch under the old policy and the reference before an update
        case("score_models", "score", 2048, 151936, 8, 8, 512, 64, models=2),
        # one rank's share of a head split over four ranks by vocabulary: statistics, merge, backward
        case("shard_7b", "shard", 3584, 152064, 4, 8, 512, 64, w_std=0.015, ranks=4, rank=1),
        # the full-distribution KL to a reference model of the same width
        case("full_kl_3b", "full_kl", 2048, 151936, 2, 8, 384, 48),
        # the per-token arithmetic of a large batch on its own: advantages, KL-shaped returns, token loss
        case("token_values", "tokens", 0, 151936, 64, 16, 512, 32, ent_coef=1e-3),
    ]


def draw(rng):
    """Another case of the same ranges: rows over three decades, hidden sizes and vocabularies of 0.5B to 7B-class
    heads, ragged lengths, every option that the listed cases use."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "score", "score", "shard", "full_kl", "tokens"])
    d = 64 * log(4, 56)
    V = rng.choice([log(4000, 152064), log(100000, 152064), 151936, 152064])
    G = rng.choice([2, 4, 5, 8, 16])
    limit = 4e14 / (12.0 * d * V) if kind == "full_kl" else 6e14 / (8.0 * d * V)
    rows = log(40, max(80, min(2 ** 19 if kind != "tokens" else 2 ** 20, limit)))
    L_max = max(8, min(4096, log(8, max(9, rows // G + 1))))
    prompts = max(1, rows // (G * L_max))
    case = dict(kind=kind, d=d if kind != "tokens" else 0, V=V, prompts=prompts, G=G, L_max=L_max,
                len_lo=max(1, L_max // rng.choice([1, 2, 4, 8, 16])), w_std=rng.choice([0.015, 0.02]), eps_low=0.2,
                eps_high=rng.choice([0.2, 0.28]), beta=rng.choice([0.04, 0.04, 0.01, 0.0]), ent_coef=0.0,
                span=0.3 if L_max >= 256 and rng.random() < 0.3 else 0.0, accumulate=False, agg_mode=0,
                sequence_level=False)
    if kind == "step":
        case["accumulate"] = rng.random() < 0.3
        case["ent_coef"] = rng.choice([0.0, 0.0, 1e-3])
        case["agg_mode"] = rng.choice([0, 0, 0, 1, 2])
        case["sequence_level"] = rng.random() < 0.2
    elif kind == "score":
        case["models"] = rng.choice([1, 1, 2])
    elif kind == "shard":
        case["ranks"] = rng.choice([2, 4, 8])
        case["rank"] = rng.randrange(case["ranks"])
    elif kind == "full_kl":
        case["beta"] = 0.04
    elif kind == "tokens":
        case["ent_coef"] = rng.choice([0.0, 1e-3])
        case["beta"] = 0.04
    return case


def _slice(case):
    """First vocabulary row and number of rows of this rank's part of the head (all of it unless it is split)."""
    ranks = case.get("ranks", 1)
    if ranks == 1:
        return 0, case["V"]
    tiles = -(-case["V"] // 256)
    lo = tiles * case["rank"] // ranks * 256
    hi = min(case["V"], tiles * (case["rank"] + 1) // ranks * 256)
    return lo, hi - lo


def _rows(case, gen):
    """Row mask and row ranges of the batch, responses padded to L_max."""
    n_seq, L = case["prompts"] * case["G"], case["L_max"]
    lens = torch.randint(case["len_lo"], L + 1, (n_seq,), generator=gen, device=DEVICE)
    pos = torch.arange(L, device=DEVICE)
    mask = pos[None, :] < lens[:, None]
    if case["span"] > 0:
        # observation spans of 32 to 256 rows: each response loses `span` of its rows in all
        n_spans = max(1, int(case["span"] * L / 144 * 1.2))
        start = (torch.rand(n_seq, n_spans, generator=gen, device=DEVICE) * L).long() + 1
        length = torch.randint(32, 257, (n_seq, n_spans), generator=gen, device=DEVICE).clamp(max=max(1, L // 4))
        for k in range(n_spans):
            mask &= ~((pos[None, :] >= start[:, k:k + 1]) & (pos[None, :] < (start + length)[:, k:k + 1]))
        mask[:, 0] = True
    return mask.reshape(-1).to(torch.uint8), torch.arange(0, n_seq * L + 1, L, dtype=torch.int32, device=DEVICE)


def _valid_rows(case):
    """Expected number of rows that take part."""
    rows = case["prompts"] * case["G"] * 0.5 * (case["len_lo"] + case["L_max"])
    if case["span"] > 0:
        n_spans = max(1, int(case["span"] * case["L_max"] / 144 * 1.2))
        rows *= (1 - min(144, max(1, case["L_max"] // 4)) / case["L_max"]) ** n_spans
    return rows


def _head(gen, V, d, std):
    return torch.randn(V, d, generator=gen, device=DEVICE, dtype=torch.bfloat16).mul_(std)


def _hidden(gen, W, row_of_token, peak, chunk=32768):
    """Hidden states [T, d]: noise plus a component along the sampled token's row of W that lifts its logit by `peak`
    (0: a flat softmax; 12 and more: an almost certain token).  row_of_token < 0: the row is not held here."""
    T, d = row_of_token.numel(), W.shape[1]
    H = torch.empty(T, d, device=DEVICE, dtype=torch.bfloat16)
    zy, sq = torch.empty(T, device=DEVICE), torch.empty(T, device=DEVICE)
    for i in range(0, T, chunk):
        j = slice(i, min(T, i + chunk))
        w = W[row_of_token[j].clamp(min=0)].float() * (row_of_token[j] >= 0)[:, None]
        h = torch.randn(w.shape, generator=gen, device=DEVICE)
        h += w * (peak[j] / w.square().sum(1).clamp(min=1e-12))[:, None]
        H[j] = h.to(torch.bfloat16)
        h = H[j].float()
        zy[j], sq[j] = (h * w).sum(1), h.square().sum(1)
    return H, zy, sq


def _logsumexp(zy, sq, V, std):
    """log sum_j exp z_j: the sampled token's own term, and V - 1 logits that are normal with variance std^2 |h|^2."""
    return torch.logaddexp(zy, math.log(max(V - 1, 1)) + 0.5 * std * std * sq)


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    mask, offsets = _rows(case, gen)
    T, n_seq, V, d = mask.numel(), offsets.numel() - 1, case["V"], case["d"]
    off, Vs = _slice(case)
    s = dict(case=case, ctx=Context(0), mask=mask, offsets=offsets, T=T)
    # token ids: a few words make up much of a text (log-uniform rank), spread over the vocabulary
    rank = torch.exp(torch.rand(T, generator=gen, device=DEVICE) * math.log(V)).long().clamp(1, V) - 1
    tokens = (rank * 7919 + 13) % V
    peak = 16.0 * torch.rand(T, generator=gen, device=DEVICE)
    rewards = torch.rand(n_seq, generator=gen, device=DEVICE)
    s["rewards"] = rewards if case["w_std"] == 0.015 else (rewards < 0.4).float()
    if case["kind"] == "tokens":
        logp = -torch.log1p(math.exp(11.0) * torch.exp(-peak))
        s["entropy"] = -logp
    else:
        W = s["W"] = _head(gen, Vs, d, case["w_std"])
        held = tokens - off
        s["H"], zy, sq = _hidden(gen, W, torch.where((held >= 0) & (held < Vs), held, -1), peak)
        if case["kind"] == "shard":
            away = (held < 0) | (held >= Vs)
            zy = torch.where(away, peak + case["w_std"] * sq.sqrt() * torch.randn(T, generator=gen, device=DEVICE), zy)
            s["gathered"] = _other_slices(case, tokens, mask, zy, sq)
        logp = zy - _logsumexp(zy, sq, V, case["w_std"])
    noise = torch.randn(2, T, generator=gen, device=DEVICE)
    s["tokens"] = (tokens * mask).to(torch.int32)
    s["logp"] = logp * mask
    s["old_logp"] = (logp + 0.05 * noise[0]) * mask
    s["ref_logp"] = (logp + 0.1 * noise[1]) * mask if case["beta"] > 0 else None
    if case["kind"] in ("step", "shard", "full_kl"):
        s["loss"] = torch.zeros(1, device=DEVICE)
        s["dH"] = torch.zeros(T, d, device=DEVICE, dtype=torch.float32 if case["kind"] == "shard" else torch.bfloat16)
        s["dW"] = torch.zeros(Vs, d, device=DEVICE)
    if case["accumulate"] or case["kind"] == "shard":
        # a micro-batch or a rank gets its rows' advantages with the batch
        s["adv"] = torch.randn(n_seq, generator=gen, device=DEVICE).repeat_interleave(case["L_max"])
        s["token_count"] = (mask.sum() * 16).to(torch.int64).reshape(1)
    if case.get("models", 1) > 1 or case["kind"] == "full_kl":
        # the second model is the first before training: the same tensors plus a drift
        drift = torch.randn(Vs, d, generator=gen, device=DEVICE, dtype=torch.bfloat16)
        s["W_ref"] = W * (1.0 + 0.05 * drift)
        s["H_ref"] = s["H"] + 0.05 * torch.randn(T, d, generator=gen, device=DEVICE, dtype=torch.bfloat16)
    return s


def _other_slices(case, tokens, mask, zy, sq):
    """Softmax statistics (M, S, A, z_y) per slice of a split head, as the other ranks would send them: logits of
    variance std^2 |h|^2, and the sampled token's where it is held.  This rank's own are written by the call."""
    out = torch.zeros(case["ranks"], tokens.numel(), 4, device=DEVICE)
    var = case["w_std"] ** 2 * sq
    for r in range(case["ranks"]):
        lo, n = _slice(dict(case, rank=r))
        here = ((tokens >= lo) & (tokens < lo + n)).float()
        M = torch.maximum(zy * here, var.sqrt() * math.sqrt(2 * math.log(n)))
        mass, own = n * torch.exp(0.5 * var - M), here * torch.exp(zy - M)
        out[r] = torch.stack([M, mass + own, mass * var + own * zy, zy * here], 1) * mask[:, None]
    return out


def run(s):
    c, ctx = s["case"], s["ctx"]
    hyper = (c["eps_low"], c["eps_high"], c["beta"])
    if c["kind"] == "step":
        out = {}
        adv = s.get("adv")
        if adv is None:
            out["adv_seq"], adv = ctx.rl_grpo_advantages(s["rewards"], c["G"], seq_offsets=s["offsets"], T=s["T"])
        by_response = c["agg_mode"] > 0 or c["sequence_level"]
        out.update(ctx.rl_policy_loss_fwd_bwd(
            s["H"], s["W"], s["tokens"], s["old_logp"], s["ref_logp"], adv, s["mask"], *hyper, ent_coef=c["ent_coef"],
            accumulate_dW=c["accumulate"], dW=s["dW"], dH=s["dH"], loss=s["loss"], agg_mode=c["agg_mode"],
            sequence_level=c["sequence_level"], seq_offsets=s["offsets"] if by_response else None,
            token_count=s.get("token_count")))
        return out
    if c["kind"] == "score":
        if c["models"] == 1:
            return ctx.rl_token_logprobs(s["H"], s["W"], s["tokens"], s["mask"])
        return ctx.rl_token_logprobs_multi([s["H"], s["H_ref"]], [s["W"], s["W_ref"]], s["tokens"], s["mask"])
    if c["kind"] == "shard":
        off, _ = _slice(c)
        ctx.rl_shard_logit_stats(s["H"], s["W"], s["tokens"], s["mask"], off, c["V"], stats=s["gathered"][c["rank"]])
        logp, ent, lse = ctx.rl_merge_logit_stats(s["gathered"], s["mask"])
        out = ctx.rl_policy_loss_shard_bwd(s["H"], s["W"], s["tokens"], s["old_logp"], s["ref_logp"], s["adv"],
                                           s["mask"], off, c["V"], logp, ent, lse, *hyper, dH=s["dH"], dW=s["dW"])
        return dict(out, logp=logp, entropy=ent, lse=lse)
    if c["kind"] == "full_kl":
        adv_seq, adv = ctx.rl_grpo_advantages(s["rewards"], c["G"], seq_offsets=s["offsets"], T=s["T"])
        return ctx.rl_policy_loss_fwd_bwd(s["H"], s["W"], s["tokens"], s["old_logp"], None, adv, s["mask"], *hyper,
                                          dW=s["dW"], dH=s["dH"], loss=s["loss"], H_ref=s["H_ref"], W_ref=s["W_ref"])
    adv_seq, adv = ctx.rl_grpo_advantages(s["rewards"], c["G"], seq_offsets=s["offsets"], T=s["T"])
    shaped, returns = ctx.rl_kl_shaped_returns(adv_seq, s["logp"], s["ref_logp"], s["mask"], s["offsets"], s["T"], 0.02)
    out = ctx.rl_token_loss(s["logp"], s["entropy"], s["old_logp"], s["ref_logp"], adv, s["mask"], *hyper,
                            ent_coef=c["ent_coef"])
    return dict(out, adv_seq=adv_seq, adv=adv, shaped=shaped, returns=returns)


def work(case):
    """Least traffic and arithmetic of one pass: inputs read once (the rows that take part), outputs written once
    (read as well where they are added to), 2 d flop per token and vocabulary word for the logits and for each of the
    two gradients.  A split head forms its logits twice: its two calls share nothing but the statistics."""
    T, N = case["prompts"] * case["G"] * case["L_max"], _valid_rows(case)
    n_seq, d = case["prompts"] * case["G"], case["d"]
    _, V = _slice(case)
    kind = case["kind"]
    if kind == "tokens":
        return {"bytes": T * (4 + 17 + 29) + n_seq * 24, "flops": 60.0 * N}
    models = case.get("models", 1)
    if kind == "score":
        return {"bytes": models * (2 * d * (N + V) + 12 * T) + 5 * T, "flops": models * 2.0 * N * d * V}
    acc = 2 if case["accumulate"] else 1
    b = 2 * d * (N + V) + (4 if kind == "shard" else 2) * T * d + 4 * V * d * acc + 29 * T
    f = 6.0 * N * d * V
    if kind == "full_kl":
        b, f = b + 2 * d * (N + V) + 4 * T, f + 2.0 * N * d * V
    if kind == "shard":
        b, f = b + 16 * T * (1 + case["ranks"]), f + 2.0 * N * d * V
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Gradients come from bf16 factors: two correct ways of rounding them differ by 2e-3 (other tile orders alone
    give 4e-4, the rounding of dH).  Log-probabilities and entropies are sums in 32 bits of exact products, within 5e-6
    of the same sums in 64 bits; per-token values are 32-bit arithmetic."""
    if case["kind"] == "score":
        return {"rel": 2e-5}
    if case["kind"] == "tokens":
        return {"rel": 1e-5}
    return {"rel": 1e-2}
