"""Timed workloads of the selective-rollout gate library, through its Python entry points.

Each case is one of six things a training program does with the library:

``action``   one training iteration at action level: the gate on the action prefixes of
             all groups (``sr_gate``, K <= 32), then the group-relative advantages with
             the stop mask as drop mask.
``token``    the same iteration on token prefixes (K up to 1024, multi-word path).
``decide``   the token iteration with only the stop mask of the gate (``sr_gate_decide``).
``host``     token prefixes that sit packed in pinned host memory, results wanted on the
             host (``sr_gate_host_packed`` with a copy stream).
``stream``   one whole episode of the incremental gate: a fresh state, then one call per
             environment step, each step's decisions kept.
``monitor``  the figures logged for a finished batch: Appendix-B signals, the OR rule,
             batch statistics and the list of groups kept.

Inputs follow the recipes of ``paper_2605_05802_b200.workloads`` (action IDs below 4096,
per-group mutation rate from Beta(0.5, 2); token IDs below 151 936, even groups converged
with 10 % of the tokens substituted, odd groups sharing a head and then diverging), drawn
on the GPU.  ``text`` draws token IDs with the 1/rank frequencies of written language, in
which a few tokens make up much of every rollout, and spreads the converged groups'
substitution rates over 0..20 % so that d_K falls on both sides of the threshold; without
it tokens are uniform and the rate is 10 %, as in the repository's benchmark.  ``ragged``
rollouts end anywhere between K/4 (at action level: one action) and K or beyond; otherwise
all of them have reached step K.
"""
import math

import numpy as np
import torch

import paper_2605_05802_b200.binding as sr

ACTION_VOCAB = 4096
TOKEN_VOCAB = 151936
HORIZON = 30            # environment steps of an episode
EPS = 1e-6
# pairs of a drawn batch: none costs more than the largest listed one
MOST_PAIRS = {"action": 1 << 21, "token": 12 << 10, "decide": 12 << 10, "host": 12 << 10,
              "stream": 1 << 20, "monitor": 1 << 19}


def listed():
    return [
        # one on-policy iteration of the paper: 10 prompts x 8 rollouts, gate at step 10; pure latency
        {"name": "action-iteration", "kind": "action", "groups": 10, "N": 8, "K": 10, "ragged": False, "raw": False, "dist": False},
        # a batch of a larger trainer: ragged rollouts, gate at step 15
        {"name": "action-batch", "kind": "action", "groups": 512, "N": 8, "K": 15, "ragged": True, "raw": False, "dist": False},
        # groups of 16 over the whole horizon, pair distances wanted too
        {"name": "action-groups-of-16", "kind": "action", "groups": 4096, "N": 16, "K": 30, "ragged": False, "raw": False, "dist": True},
        # scoring a stored buffer of rollouts
        {"name": "action-buffer", "kind": "action", "groups": 65536, "N": 8, "K": 15, "ragged": True, "raw": False, "dist": False},
        # the paper's iteration on token prefixes
        {"name": "token-iteration", "kind": "token", "groups": 16, "N": 8, "K": 1024, "text": True, "ragged": True, "raw": False, "dist": False},
        # the repository's benchmark batch
        {"name": "token-batch", "kind": "token", "groups": 1024, "N": 8, "K": 1024, "text": False, "ragged": True, "raw": False, "dist": False},
        # odd sizes all round: 5 rollouts, K no multiple of the word, raw distances
        {"name": "token-odd", "kind": "token", "groups": 301, "N": 5, "K": 501, "text": True, "ragged": True, "raw": True, "dist": True},
        # the mask alone for a large token batch, at the paper's operating point
        {"name": "token-decide", "kind": "decide", "groups": 1024, "N": 8, "K": 1024, "text": True, "ragged": False, "raw": False},
        # rollouts handed over by an inference engine in host memory
        {"name": "token-host", "kind": "host", "groups": 1024, "N": 8, "K": 1024, "text": True, "ragged": True, "raw": False, "dist": False},
        # gate after every step of one iteration's episodes, ending at different steps
        {"name": "stream-iteration", "kind": "stream", "groups": 64, "N": 8, "steps": HORIZON, "ragged": True, "raw": False},
        # the same for a very large simulator batch
        {"name": "stream-batch", "kind": "stream", "groups": 65536, "N": 8, "steps": HORIZON, "ragged": False, "raw": False},
        # logging for one large batch
        {"name": "monitor-batch", "kind": "monitor", "groups": 4096, "N": 16, "K": 30, "ragged": True},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["action", "action", "token", "token", "decide", "host", "stream", "monitor"])
    N = rng.choice([8, 8, 16, 4, rng.randint(2, 16), rng.randint(2, 24)])
    most = MOST_PAIRS[kind] // (N * (N - 1) // 2)
    # host buffers of a handful of groups go through the same call as large ones
    groups = _log_int(rng, 4, max(8, min(most, 65536)))
    case = {"kind": kind, "groups": groups, "N": N}
    if kind in ("action", "monitor"):
        case.update(K=rng.randint(5, 32), ragged=rng.random() < 0.5)
    elif kind == "stream":
        case.update(steps=rng.randint(10, HORIZON), ragged=rng.random() < 0.5)
    else:
        case.update(K=_log_int(rng, 48, 1024), text=rng.random() < 0.6, ragged=rng.random() < 0.7)
    if kind != "monitor":
        case["raw"] = rng.random() < 0.2
    if kind in ("action", "token", "host"):
        case["dist"] = rng.random() < 0.3
    return case


# ------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _actions(case, gen, steps, seed):
    """int64 [groups, N, steps]: every rollout walks its group's base and, with the group's
    probability, emits a stray action (moving on or not) or skips one of the base."""
    G, N = case["groups"], case["N"]
    p = torch.from_numpy(np.random.default_rng(seed).beta(0.5, 2.0, size=G)).cuda().view(G, 1, 1)
    base = torch.randint(0, ACTION_VOCAB, (G, 2 * steps + 8), generator=gen, device="cuda")
    mutate = torch.rand((G, N, steps), generator=gen, device="cuda") < p
    op = torch.randint(0, 3, (G, N, steps), generator=gen, device="cuda")
    stray = torch.randint(0, ACTION_VOCAB, (G, N, steps), generator=gen, device="cuda")
    skip = mutate & (op == 2)
    move = torch.where(mutate & (op == 1), 0, torch.where(skip, 2, 1))
    at = (torch.cumsum(move, 2) - move + skip).view(G, N * steps)
    walk = torch.gather(base, 1, at).view(G, N, steps)
    equal = torch.rand((G, 1), generator=gen, device="cuda") < 1.0 - p.view(G, 1)
    return torch.where(mutate & (op < 2), stray, walk), equal


def _rewards(case, gen, equal):
    """Binary terminal rewards; the groups in ``equal`` share one outcome."""
    G, N = case["groups"], case["N"]
    own = torch.randint(0, 2, (G, N), generator=gen, device="cuda")
    return torch.where(equal, own[:, :1], own).float()


def _token_ids(shape, case, gen):
    if case["text"]:       # frequency of the r-th most common token ~ 1 / r
        u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
        return (torch.exp(u * math.log(TOKEN_VOCAB)) - 1.0).to(torch.int32)
    return torch.randint(0, TOKEN_VOCAB, shape, generator=gen, device="cuda", dtype=torch.int32)


def _tokens(case, gen):
    """int32 [groups, N, stride] and lengths."""
    G, N, K = case["groups"], case["N"], case["K"]
    stride = (K + 3) // 4 * 4
    lens = torch.full((G, N), K, dtype=torch.int32, device="cuda")
    if case["ragged"]:
        lens = torch.randint(K // 4, K + 1, (G, N), generator=gen, device="cuda", dtype=torch.int32)
    base = _token_ids((G, 1, stride), case, gen)
    own = _token_ids((G, N, stride), case, gen)
    pos = torch.arange(stride, device="cuda")
    head = (torch.rand((G, 1, 1), generator=gen, device="cuda") * (lens.amin(1).view(G, 1, 1) + 1)).int()
    rate = torch.rand((G, 1, 1), generator=gen, device="cuda") * 0.2 if case["text"] else 0.10
    substituted = torch.rand((G, N, stride), generator=gen, device="cuda") < rate
    converged = (torch.arange(G, device="cuda") % 2 == 0).view(G, 1, 1)
    take_own = torch.where(converged, substituted, pos >= head)
    seqs = torch.where(take_own, own, base)
    seqs = torch.where(pos < lens.unsqueeze(2), seqs, 0).contiguous()
    return seqs, lens


def _norm(case):
    """Normalised at the paper's d_L = 0.12, or raw distances at about the same strictness."""
    if not case.get("raw"):
        return sr.SR_NORM_MAXLEN, 0.12
    return sr.SR_NORM_NONE, 0.12 * case.get("K", case.get("steps"))


def _empty(*shape, dtype):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    gen = _generator(seed)
    G, N, kind = case["groups"], case["N"], case["kind"]
    P = N * (N - 1) // 2
    norm, threshold = _norm(case)
    s = {"kind": kind, "norm": norm, "threshold": threshold, "N": N, "K": case.get("K"),
         "stop": _empty(G, dtype=torch.uint8)}
    if kind in ("action", "monitor"):
        K = case["K"]
        actions, equal = _actions(case, gen, HORIZON + 2, seed)
        lens = torch.full((G, N), HORIZON + 2, dtype=torch.int32, device="cuda")
        if case["ragged"]:
            lens = torch.randint(1, HORIZON + 1, (G, N), generator=gen, device="cuda", dtype=torch.int32)
        live = torch.arange(HORIZON + 2, device="cuda") < lens.unsqueeze(2)
        s.update(seqs=torch.where(live, actions, 0).int().contiguous(), lens=lens, rewards=_rewards(case, gen, equal))
    if kind in ("token", "decide", "host"):
        s["seqs"], s["lens"] = _tokens(case, gen)
        s["rewards"] = torch.rand((G, N), generator=gen, device="cuda")
        stride = s["seqs"].shape[2]
    if kind in ("action", "token", "decide"):
        need = sr.sr_gate_workspace_bytes(G, N, s["seqs"].shape[2], case["K"])
        s.update(mean=_empty(G, dtype=torch.float64), adv=_empty(G, N, dtype=torch.float32), zero_var=_empty(G, dtype=torch.uint8),
                 dist=_empty(G, P, dtype=torch.int32) if case.get("dist") else None,
                 workspace=_empty(need, dtype=torch.uint8) if need else None)
    elif kind == "host":
        lens = s.pop("lens")
        live = torch.arange(stride, device="cuda") < lens.unsqueeze(2)
        symbols = s.pop("seqs")[live].cpu().pin_memory()
        start = torch.zeros(G * N + 1, dtype=torch.int64)
        start[1:] = torch.cumsum(lens.view(-1).long(), 0).cpu()
        s.update(symbols=symbols, row_start=start.pin_memory(), stride=stride,
                 mean=torch.zeros(G, dtype=torch.float64).pin_memory(), stop=torch.zeros(G, dtype=torch.uint8).pin_memory(),
                 dist=torch.zeros((G, P), dtype=torch.int32).pin_memory() if case["dist"] else None,
                 arena=_empty(sr.sr_gate_host_packed_arena_bytes(G, N, stride, case["K"]), dtype=torch.uint8),
                 copy_stream=torch.cuda.Stream())
    elif kind == "stream":
        steps = case["steps"]
        actions, _ = _actions(case, gen, steps, seed)
        if case["ragged"]:
            end = torch.randint(min(10, steps), steps + 1, (G, N, 1), generator=gen, device="cuda")
            actions = torch.where(torch.arange(steps, device="cuda") < end, actions, sr.SR_NO_ACTION)
        mean, stop = _empty(steps, G, dtype=torch.float64), _empty(steps, G, dtype=torch.uint8)
        actions = actions.permute(2, 0, 1).int().contiguous()
        s.update(state=_empty(sr.sr_incr_state_bytes(G, N, HORIZON), dtype=torch.uint8), groups=G,
                 actions=list(actions.unbind(0)), mean=mean, stop=stop, means=list(mean.unbind(0)), stops=list(stop.unbind(0)))
    elif kind == "monitor":
        s.update(adv=torch.empty(G, N, device="cuda"), zero_var=_empty(G, dtype=torch.uint8), mean=_empty(G, dtype=torch.float64))
        # what the training iteration has left behind: d_K, the decisions, the advantages
        sr.sr_gate(s["seqs"], s["lens"], case["K"], threshold, mean=s["mean"], stop=s["stop"])
        sr.sr_grpo_advantage(s["rewards"], None, EPS, adv=s["adv"], zero_var=s["zero_var"])
        s.update({k: _empty(G, dtype=torch.float64) for k in ("upr", "uar", "entropy", "jaccard", "tau")})
        s.update(either=_empty(G, dtype=torch.uint8), counts=_empty(3, dtype=torch.int64), sumsq=_empty(2, dtype=torch.float64),
                 index=_empty(G, dtype=torch.int32), count=_empty(1, dtype=torch.int32),
                 workspace=_empty(sr.sr_kept_groups_workspace_bytes(G), dtype=torch.uint8))
    return s


# ---------------------------------------------------------------------------- the passes
def run(s):
    kind = s["kind"]
    if kind in ("action", "token"):
        sr.sr_gate(s["seqs"], s["lens"], s["K"], s["threshold"], s["norm"], pair_dist=s["dist"], mean=s["mean"],
                   stop=s["stop"], workspace=s["workspace"])
        sr.sr_grpo_advantage(s["rewards"], s["stop"], EPS, adv=s["adv"], zero_var=s["zero_var"])
        return {"mean": s["mean"], "stop": s["stop"], "dist": s["dist"], "adv": s["adv"], "zero_var": s["zero_var"]}
    if kind == "decide":
        sr.sr_gate_decide(s["seqs"], s["lens"], s["K"], s["threshold"], s["norm"], stop=s["stop"], workspace=s["workspace"])
        sr.sr_grpo_advantage(s["rewards"], s["stop"], EPS, adv=s["adv"], zero_var=s["zero_var"])
        return {"stop": s["stop"], "adv": s["adv"], "zero_var": s["zero_var"]}
    if kind == "host":
        sr.sr_gate_host_packed(s["symbols"], s["row_start"], s["N"], s["stride"], s["K"], s["threshold"], s["norm"],
                               pair_dist=s["dist"], mean=s["mean"], stop=s["stop"], arena=s["arena"], copy_stream=s["copy_stream"])
        return {"mean": s["mean"], "stop": s["stop"], "dist": s["dist"]}
    if kind == "stream":
        sr.sr_incr_init(s["state"], s["groups"], s["N"], HORIZON)
        for new, mean, stop in zip(s["actions"], s["means"], s["stops"]):
            sr.sr_gate_step_incremental(s["state"], new, s["threshold"], s["norm"], mean=mean, stop=stop)
        return {"mean": s["mean"], "stop": s["stop"]}
    sr.sr_group_signals(s["seqs"], s["lens"], s["K"], unique_prefix_ratio=s["upr"], unique_action_ratio=s["uar"],
                        action_entropy=s["entropy"], bigram_jaccard_mean=s["jaccard"])
    sr.sr_gate_or_rule(s["mean"], s["lens"], None, s["N"], s["K"], s["threshold"], 0.9, tau=s["tau"], stop=s["either"])
    sr.sr_batch_stats(s["adv"], s["stop"], counts=s["counts"], sumsq=s["sumsq"])
    sr.sr_kept_groups(s["stop"], s["zero_var"], index=s["index"], count=s["count"], workspace=s["workspace"])
    return {k: s[k] for k in ("upr", "uar", "entropy", "jaccard", "tau", "either", "counts", "sumsq", "index", "count")}


# ------------------------------------------------------------------ what a pass needs
def work(case):
    """Bytes: inputs once, outputs once.  flops: integer lane operations, ten for every
    (text column, 32-row pattern block) of the bit-vector recurrence, at the mean lengths."""
    G, N, kind = case["groups"], case["N"], case["kind"]
    P = N * (N - 1) // 2
    if kind == "stream":
        T = case["steps"]
        live = 0.5 * (T + min(10, T)) if case["ragged"] else T
        # per step: pair state in and out, the actions so far, the new ones, lengths, decisions
        step = P * 32 + N * (4 * live / 2 + 4 + 4 + 8) + 9
        return {"bytes": G * T * step, "flops": G * P * live * 20}
    K = case["K"]
    if kind in ("action", "monitor"):
        m = sum(min(n, K) for n in range(1, HORIZON + 1)) / HORIZON if case["ragged"] else K
    else:
        m = 0.625 * K if case["ragged"] else K
    bytes_ = G * N * (4 * m + 4)
    if kind in ("action", "token"):
        bytes_ += G * (8 + 1 + 1 + 1) + G * N * 8
    elif kind == "decide":
        bytes_ += G * (1 + 1 + 1) + G * N * 8
    elif kind == "host":
        bytes_ += G * N * 4 + G * 9
    else:       # signals, tau and decisions; advantages, flags and the index list
        bytes_ += G * (5 * 8 + 8 + 1) + G * N * 8 + G * (1 + 1 + 1 + 4)
        return {"bytes": bytes_, "flops": G * N * m * 10}
    if case.get("dist"):
        bytes_ += G * P * 4
    return {"bytes": bytes_, "flops": G * P * m * math.ceil(m / 32) * 10}


def tolerance(case):
    """Decisions, counts, indices and distances are whole numbers and exact; d_K is an fp64
    sum in a fixed order; advantages are rounded to fp32; logged figures are fp64 sums and
    logarithms."""
    if case["kind"] in ("action", "token", "decide"):
        return {"rel": 1e-6}
    if case["kind"] == "monitor":
        return {"rel": 1e-10}
    return "exact"
