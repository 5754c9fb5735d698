"""Workloads over which the speed of the library is measured.

Each case is one pass through a public entry point of the binding, with the
inputs, weights, workspace and output buffers a decoding loop would hold.
Shapes come from the five workloads of ``workloads.CONFIGS`` (block 16 and the
151936-token vocabulary at hidden sizes 2560 and 4096, a tiny fp32 block) and,
beside them, generic ones: other batch sizes, ragged vocabularies, hidden
sizes that are no multiple of 256.

A case's fields:
  op       "round" (retrace_round), "lowrank", "sampled" (rounds with the
           low-rank conditioning, and with sampling at temperature 1),
           "verify" (retrace_verify), "halves" (retrace_align_refine, then
           retrace_gate_fuse);
  B K V d  batch, draft tokens per block, vocabulary, hidden size;
  dtype    "bf16" or "f32";
  prefix_p parameter of the geometric accepted prefix, 0: uniform over 0..K;
  std      of the logits;
  dense_e  the drafter inputs are [B, K, d] instead of one mask embedding;
  argmax   every row's argmax is an output too (greedy verification);
  ties     copies of the row maximum are planted.
"""

import torch

from paper_2608_29748_gb300 import binding as rt
from paper_2608_29748_gb300.workloads import (
    LOWRANK_CORRECTION,
    LOWRANK_LATENT,
    SAMPLING,
    RoundConfig,
    make_lowrank_weights,
    make_round_inputs,
)

# Drafter logits of the sampled cases: the target's plus noise of this share
# of the logits' spread.  With draft tokens drawn from the filtered drafter
# distribution, about two in three are accepted.
DRAFT_NOISE = 0.2


def _case(name, op, B, K, V, d, dtype="bf16", prefix_p=0.2, std=1.0, dense_e=False, argmax=False, ties=False):
    return {"name": name, "op": op, "B": B, "K": K, "V": V, "d": d, "dtype": dtype, "prefix_p": prefix_p,
            "std": std, "dense_e": dense_e, "argmax": argmax, "ties": ties}


def listed():
    return [
        # The smallest call: one sequence of a toy model in fp32, all latency.
        _case("tiny-f32", "round", 1, 8, 1024, 256, "f32", prefix_p=0.0),
        # One user, a 2560-wide model: the latency of a single stream.
        _case("stream-2560", "round", 1, 16, 151936, 2560, prefix_p=0.3),
        # A handful of users, a 4096-wide model.
        _case("batch8-4096", "round", 8, 16, 151936, 4096, prefix_p=0.3, std=2.0),
        # A medium batch with uniform acceptance and tied maxima.
        _case("batch64-2560", "round", 64, 16, 151936, 2560, prefix_p=0.0, ties=True),
        # The serving batch, the largest call.
        _case("batch256-4096", "round", 256, 16, 151936, 4096, prefix_p=0.2),
        # Drafter inputs that differ by position (a drafter fed token embeddings).
        _case("dense-e-2560", "round", 32, 16, 151936, 2560, prefix_p=0.2, dense_e=True),
        # Concurrent serving with the low-rank conditioning path.
        _case("lowrank-4096", "lowrank", 64, 16, 151936, 4096, prefix_p=0.2),
        # Sampling at temperature 1: a single stream and a batch.
        _case("sampled-stream-2560", "sampled", 1, 16, 151936, 2560, std=2.0),
        _case("sampled-batch32-4096", "sampled", 32, 16, 151936, 4096, std=2.0),
        # Verification alone, as a decoder without conditioning calls it: a
        # vocabulary with a few added tokens (rows not 16-byte aligned), a
        # short block, every argmax returned.
        _case("verify-ragged", "verify", 48, 10, 32003, 0, prefix_p=0.2, argmax=True),
        # The two conditioning entry points apart from the round (a decoder
        # with a verification of its own), hidden size no multiple of 256.
        _case("halves-1152", "halves", 24, 12, 0, 1152, prefix_p=0.2),
        # A small fp32 model and batch (validation runs).
        _case("batch8-f32-1024", "round", 8, 8, 32000, 1024, "f32", prefix_p=0.2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    op = rng.choice(["round", "round", "round", "verify", "halves", "sampled", "lowrank"])
    f32 = rng.random() < 0.2
    K = rng.choice([4, 5, 7, 8, 10, 12, 15, 16, 16, 16])
    kind = rng.random()
    if kind < 0.6:
        d = 256 * rng.randint(1, 16)
    elif kind < 0.9:
        d = 64 * rng.randint(3, 45)
    else:
        d = 8 * rng.randint(20, 300)
    # fp32 and ragged hidden sizes belong to small deployments
    most_b = 24 if f32 else 256 if d % 256 == 0 else 64
    if op == "sampled":
        most_b = min(most_b, 96)
    B = _log_int(rng, 1, most_b)
    if f32:
        d = min(d, 2048)
    if op == "verify":
        d = 0
    V = rng.choice([151936, 151936, _log_int(rng, 1000, 151936), 8 * _log_int(rng, 125, 18992), 64 * _log_int(rng, 16, 2374)])
    if op == "halves":
        V = 0
    return {"op": op, "B": B, "K": K, "V": V, "d": d, "dtype": "f32" if f32 else "bf16",
            "prefix_p": rng.choice([0.0, 0.12, 0.2, 0.2, 0.3, 0.5]),
            "std": rng.choice([1.0, 2.0]) if op != "sampled" else 2.0,
            "dense_e": op in ("round", "halves") and rng.random() < 0.25,
            "argmax": op in ("round", "verify") and rng.random() < 0.25,
            "ties": op in ("round", "verify") and rng.random() < 0.25}


def _config(case):
    # A verification alone has no hidden states, the two halves no logits; the
    # generator's tensors of those sizes are kept minimal and not used.
    return RoundConfig("case", case["B"], case["K"], case["V"] or 16, case["d"] or 8, case["dtype"], case["std"],
                       "geometric" if case["prefix_p"] else "uniform", case["prefix_p"], ties=case["ties"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _sampling_inputs(x, seed):
    """Drafter logits, draft tokens drawn from the filtered drafter distribution, uniforms."""
    g = _generator(seed)
    logits = x["logits"]
    B, K1, V = logits.shape
    draft_logits = torch.empty((B, K1 - 1, V), dtype=logits.dtype, device="cuda")
    draft = torch.empty((B, K1 - 1), dtype=torch.int32, device="cuda")
    for b in range(B):  # one sequence at a time bounds the fp32 temporary
        row = logits[b, :-1].float()
        row = row + torch.randn(row.shape, generator=g, device="cuda") * (DRAFT_NOISE * x["cfg"].logits_std)
        draft_logits[b] = row.to(logits.dtype)
        top, token = torch.topk(draft_logits[b].float(), min(SAMPLING["top_k"], V), dim=-1)
        prob = torch.softmax(top / SAMPLING["temperature"], dim=-1)
        prob[prob.cumsum(-1) - prob >= SAMPLING["top_p"]] = 0.0
        pick = torch.multinomial(prob, 1, generator=g)
        draft[b] = torch.gather(token, 1, pick)[:, 0].to(torch.int32)
    uniforms = torch.rand((B, K1), generator=g, device="cuda")
    return {"draft_logits": draft_logits, "draft": draft, "uniforms": uniforms, **SAMPLING,
            "top_k": min(SAMPLING["top_k"], V)}


def prepare(case, seed):
    cfg = _config(case)
    op, B, K, d, dt = case["op"], case["B"], case["K"], case["d"], cfg.torch_dtype
    x = make_round_inputs(cfg, device="cuda", seed=seed)
    state = {"case": case, "x": x}
    if case["dense_e"]:
        x["e"] = (torch.randn((B, K, d), generator=_generator(seed + 1), device="cuda") * 0.02).to(dt)
    if op == "sampled":
        state["s"] = _sampling_inputs(x, seed + 2)
    if op == "lowrank":
        state["w"] = make_lowrank_weights(cfg, device="cuda", seed=seed + 3)
    state["ws"] = rt.Workspace(B, K, cfg.V, cfg.d, dt)
    state["out"] = rt.RoundBuffers(B, K, cfg.d, dt)
    state["argmax"] = torch.empty((B, K + 1), dtype=torch.int32, device="cuda") if case["argmax"] else None
    if op == "halves":
        state["accept"] = x["planted_prefix"].to(torch.int32)
        state["r"] = torch.empty((B, K, d), dtype=dt, device="cuda")
    return state


def run(state):
    op, x, ws, out, argmax = state["case"]["op"], state["x"], state["ws"], state["out"], state["argmax"]
    if op == "halves":
        rt.retrace_align_refine(x["hD"], x["hT"], state["accept"], x["Wc"], x["beta"], state["r"], out.n, ws)
        rt.retrace_gate_fuse(x["e"], state["r"], out.n, x["Wv"], x["Wg"], out.e_out, ws)
        return {"n": out.n, "r": state["r"], "e_out": out.e_out}
    if op == "verify":
        rt.retrace_verify(x["logits"], x["draft"], out.accept_len, out.committed, out.bonus, ws, target_argmax=argmax)
    elif op == "round":
        rt.run_round(x, ws, out, target_argmax=argmax)
    elif op == "lowrank":
        rt.run_round_lowrank(x, state["w"], ws, out, target_argmax=argmax)
    else:
        rt.run_round_sampled(x, state["s"], ws, out)
    result = {"accept_len": out.accept_len, "committed": out.committed, "bonus": out.bonus}
    if argmax is not None:
        result["argmax"] = argmax
    if op != "verify":
        result.update(n=out.n, e_out=out.e_out)
    return result


def _expected(case):
    """Expected logits rows per sequence that the outputs depend on, and conditioned rows per sequence."""
    K, p = case["K"], case["prefix_p"]
    if case["op"] == "sampled":
        at_least = [0.67**k for k in range(K + 1)]  # P(A >= k)
    elif p:
        at_least = [(1 - p) ** k for k in range(K + 1)]
    else:
        at_least = [(K + 1 - k) / (K + 1) for k in range(K + 1)]
    exactly = [at_least[k] - (at_least[k + 1] if k < K else 0.0) for k in range(K + 1)]
    return sum(at_least), sum(q * max(0, K - 1 - A) for A, q in enumerate(exactly))


def work(case):
    """Bytes and operations one pass cannot do without, at the expected accepted lengths: the logits rows up to
    each first rejection (all of them when every argmax is returned), the hidden states of the carried rows,
    the weights once, and the outputs."""
    op, B, K, V, d = case["op"], case["B"], case["K"], case["V"], case["d"]
    s = 4 if case["dtype"] == "f32" else 2
    rows, carried = _expected(case)
    R = B * carried
    moved, flops = 0.0, 0.0
    if op != "halves":
        moved += B * (K + 1 if case["argmax"] else rows) * V * s
        moved += B * K * 4 + B * (K + 1) * 4 * (2 if case["argmax"] else 1) + 3 * B * 4
    if op == "sampled":
        moved += B * min(rows, K) * V * s + B * (K + 1) * 4
    if op == "verify":
        return {"bytes": moved, "flops": 0.0}
    e_bytes = (B * K * d if case["dense_e"] else d) * s
    moved += 2 * R * d * s + e_bytes + B * K * d * s  # m and u, e, e~
    if op == "lowrank":
        L, C = LOWRANK_LATENT, LOWRANK_CORRECTION
        moved += (L * d + C * (L + d) + L * C + d * L + d * (d + L)) * s
        flops += 2.0 * R * (L * d + C * (L + d) + L * C + 2 * d * L) + 2.0 * d * d
    else:
        moved += 5 * d * d * s
        flops += 8.0 * R * d * d + (2.0 * R * d * d if case["dense_e"] else 2.0 * d * d)
    if op == "halves":
        moved += 2 * B * K * d * s  # r is written by one call and read by the other
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    """Accepted lengths, tokens, argmaxes and row counts are whole numbers and stay the same.  The conditioned
    rows: two roundings to bf16 (r, then e~), or fp32 sums."""
    if case["op"] == "verify":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 4e-6, "max": 3e-5}
    return {"rel": 6e-3, "max": 5e-2}


def _first_argmax(rows):
    """Lowest index of each row's maximum; rows [n, V]."""
    V = rows.shape[-1]
    top = rows.amax(dim=-1, keepdim=True)
    index = torch.arange(V, device=rows.device, dtype=torch.int32)
    return torch.where(rows == top, index, V).amin(dim=-1)


def _filtered(rows):
    """Tokens [n, k] and probabilities of the top-k / top-p distributions of rows [n, V], in descending order,
    the lower index first among equal values."""
    k = min(SAMPLING["top_k"], rows.shape[-1])
    value, token = torch.sort(rows, dim=-1, descending=True, stable=True)
    value, token = value[:, :k].double(), token[:, :k]
    prob = torch.softmax(value / SAMPLING["temperature"], dim=-1)
    kept = prob.cumsum(-1) - prob < SAMPLING["top_p"]
    prob = torch.where(kept, prob, torch.zeros_like(prob))
    return token, prob / prob.sum(-1, keepdim=True)


def _sampled_sequence(target, drafter, draft, uniforms):
    """Accepted length and appended token of one sequence, by speculative sampling."""
    K = draft.numel()
    p_token, p = (t.cpu() for t in _filtered(target))
    q_token, q = (t.cpu() for t in _filtered(drafter))
    draft, u = draft.cpu().long(), uniforms.cpu().double()
    px = torch.where(p_token[:K] == draft[:, None], p[:K], 0.0).sum(-1)
    qx = torch.where(q_token == draft[:, None], q, 0.0).sum(-1)
    refused = torch.nonzero(u[:K] * qx >= px).flatten()
    A = int(refused[0]) if refused.numel() else K
    w = p[A]
    if A < K:
        q_at = torch.where(p_token[A][:, None] == q_token[A][None, :], q[A][None, :], 0.0).sum(-1)
        rest = (w - q_at).clamp_min(0.0)
        w = rest if float(rest.sum()) > 0 else w
    c = w.cumsum(0)
    j = int(torch.searchsorted(c, u[K] * c[-1], right=True))
    return A, int(p_token[A][min(j, w.numel() - 1)])


def _conditioned(x, w, A, dense):
    """r [B, K, d] and e~ [B, K, d] in float64 for accepted lengths A [B]."""
    B, K, d = x["hD"].shape
    dev = x["hD"].device
    e = x["e"].double() if dense else x["e"].double().expand(B, K, d)
    n = (K - 1 - A).clamp_min(0)
    j = torch.arange(K, device=dev)[None, :]
    b, pos = torch.nonzero(j < n[:, None], as_tuple=True)
    m = x["hD"][b, A[b] + 1 + pos].double()
    u = x["hT"][b, A[b] + pos].double()
    e_out, r_out = e.clone(), torch.zeros((B, K, d), dtype=torch.float64, device=dev)
    if b.numel():
        if w is None:
            Wc, Wv, Wg = x["Wc"].double(), x["Wv"].double(), x["Wg"].double()
            r = m + x["beta"] * (m @ Wc[:, :d].T + u @ Wc[:, d:].T)
            r_out[b, pos] = r
        else:
            P, Bc, Ac = w["P"].double(), w["Bc"].double(), w["Ac"].double()
            Wv, Wg = w["Wv_lr"].double(), w["Wg_lr"].double()
            z = m @ P.T
            r = z + x["beta"] * (torch.cat([z, u], dim=1) @ Bc.T) @ Ac.T
        pre = e[b, pos] @ Wg[:, :d].T if dense else (Wg[:, :d] @ x["e"].double())[None, :]
        e_out[b, pos] = e[b, pos] + (r @ Wv.T) * torch.sigmoid(pre + r @ Wg[:, d:].T)
    return n, r_out, e_out


def exact(case, seed):
    state = prepare(case, seed)
    op, x, B, K = case["op"], state["x"], case["B"], case["K"]
    if op == "halves":
        n, r, e_out = _conditioned(x, None, state["accept"].long(), case["dense_e"])
        return {"n": n.int(), "r": r, "e_out": e_out}
    if op == "sampled":
        s = state["s"]
        found = [_sampled_sequence(x["logits"][b], s["draft_logits"][b], s["draft"][b], s["uniforms"][b]) for b in range(B)]
        A = torch.tensor([a for a, _ in found], device="cuda")
        bonus = torch.tensor([t for _, t in found], device="cuda")
        draft, argmax = s["draft"].long(), None
    else:
        argmax = torch.stack([_first_argmax(x["logits"][b]) for b in range(B)]).long()
        draft = x["draft"].long()
        A = (argmax[:, :K] == draft).int().cumprod(dim=1).sum(dim=1).long()
        bonus = argmax.gather(1, A[:, None])[:, 0]
    i = torch.arange(K + 1, device="cuda")[None, :]
    committed = torch.where(i < A[:, None], torch.nn.functional.pad(draft, (0, 1)), -1)
    committed = torch.where(i == A[:, None], bonus[:, None], committed)
    result = {"accept_len": A.int(), "committed": committed.int(), "bonus": bonus.int()}
    if case["argmax"]:
        result["argmax"] = argmax.int()
    if op != "verify":
        n, _, e_out = _conditioned(x, state.get("w"), A, case["dense_e"])
        result.update(n=n.int(), e_out=e_out)
    return result
