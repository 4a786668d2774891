"""The work that users of the eviction library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``prepare`` makes what a serving program has in hand before the
call (the prompt's KV caches, the window queries, the plan and its buffers), ``run`` makes one pass
through the public entry points of ``paper_2606_15157_gb300.kvev``, ``exact`` gives the computed
numbers of that pass from plain torch in 64 bits.

Kinds of pass:

* ``prefill``   Plan.evict_prefill: window scores, selection and compaction of every layer at the end
                of a prompt's prefill;
* ``lse``       the same with the window rows' log-sum-exp from the caller's prefill attention;
* ``scored``    the same with every scoring layer's scores from the caller's attention: selection and
                compaction alone;
* ``h2o_full``  the prefill with the H2O layers scored over every prompt row;
* ``decode``    the decode phase of one generation: the arena filled from the compacted caches
                (DecodeArena.init_from_prefill), then ``steps`` tokens (DecodeArena.step, or
                ``decode_attn``: DecodeArena.step_attn with the caller's own attention).  With
                ``graph`` the pass is captured once and replayed, as decode loops are run in
                earnest at small batches; without it every call goes through the binding.

Inputs follow what attention looks like rather than white noise: the window queries of a KV head
share a direction (neighbouring queries resemble one another), the keys' logits against it spread
over several octaves, and the first four positions are attention sinks.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2606_15157_gb300 import kvev

FULL, SNAPKV, H2O, STREAMING, TOVA = kvev.FULL, kvev.SNAPKV, kvev.H2O, kvev.STREAMING, kvev.TOVA

SINK = 4              # StreamingLLM sinks, and the positions with raised logits
LOGIT_STD = 2.0       # spread of the keys' logits along a head's query direction
QUERY_NOISE = 0.5     # spread of a query's own logits around it
SINK_LOGIT = 6.0

# Llama-3.1-8B's geometry, the one of the paper's experiments and of the benchmark
LLAMA = {"L": 32, "H_q": 32, "H_kv": 8, "d": 128}


def _case(name, kind, B, lo, hi, S_cap, W, pool, budget, snap, h2o, stream, tova=0, avg=True, steps=0, graph=False, **geo):
    return {"name": name, "kind": kind, "B": B, "len_lo": lo, "len_hi": hi, "S_cap": S_cap, "W": W, "pool": pool,
            "avg": avg, "budget": budget, "snap": snap, "h2o": h2o, "stream": stream, "tova": tova, "steps": steps,
            "graph": graph, **geo}


def listed():
    return [
        # The smallest call: a small model's short prompt (four layers, 512 tokens), where the
        # latency of the launches is what counts.
        _case("tiny_512", "prefill", 1, 512, 512, 512, 8, 5, 64, 2, 1, 1, avg=False, L=4, H_q=4, H_kv=2, d=64),
        # One 8K prompt, every layer SnapKV with its usual 32-row window (the paper's uniform baseline).
        _case("snapkv_8k", "prefill", 1, 8192, 8192, 8192, 32, 7, 512, 32, 0, 0, **LLAMA),
        # One prompt of odd length on the heterogeneous 18/7/7 route, 32-row window.
        _case("route_8k_ragged", "prefill", 1, 7919, 7919, 8192, 32, 7, 512, 18, 7, 7, **LLAMA),
        # One long prompt, 64-row window: the batch of one that interactive use has.
        _case("route_32k_b1", "prefill", 1, 30011, 30011, 32768, 64, 7, 1024, 18, 7, 7, **LLAMA),
        # The benchmark's headline shape: eight ragged prompts of 16K to 32K tokens.
        _case("route_long_b8", "prefill", 8, 16384, 32768, 32768, 64, 7, 1024, 18, 7, 7, **LLAMA),
        # Four long prompts behind a prefill attention that hands over its rows' log-sum-exp.
        _case("lse_long_b4", "lse", 4, 16384, 32768, 32768, 64, 7, 1024, 18, 7, 7, **LLAMA),
        # Four prompts whose scores come from the caller's attention kernel: selection and compaction.
        _case("scored_long_b4", "scored", 4, 12000, 24000, 24576, 32, 7, 1024, 18, 7, 7, avg=False, **LLAMA),
        # H2O as first published: every prompt row's attention is accumulated (quadratic work).
        _case("h2o_full_6k", "h2o_full", 1, 6001, 6001, 6144, 32, 7, 512, 18, 7, 7, **LLAMA),
        # A single stream's generation on caches compacted to 2048 rows (captured loop).
        _case("decode_b1", "decode", 1, 16384, 16384, 16384, 32, 7, 2048, 18, 7, 7, steps=32, graph=True, **LLAMA),
        # The benchmark's decode batch (captured loop).
        _case("decode_b16", "decode", 16, 16384, 16384, 16384, 32, 7, 2048, 18, 7, 7, steps=32, graph=True, **LLAMA),
        # The same update when the caller's decode attention supplies the probabilities.
        _case("decode_attn_b8", "decode_attn", 8, 9000, 16384, 16384, 32, 7, 2048, 18, 7, 7, steps=32, graph=True, **LLAMA),
        # The paper's H2O / TOVA composition at 512 rows per layer, called step by step.
        _case("decode_h2o_tova_b2", "decode", 2, 4096, 8192, 8192, 32, 7, 512, 0, 16, 0, tova=16, steps=8, **LLAMA),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: kinds, geometries (GQA groups of 1 to 8, d 64 and 128),
    windows of 8 to 64 rows, lengths from 300 to 32,768, batches up to 16."""
    kind = rng.choice(["prefill", "prefill", "prefill", "lse", "scored", "h2o_full", "decode", "decode", "decode_attn"])
    H_q, H_kv = rng.choice([(32, 8), (32, 8), (32, 8), (8, 8), (16, 8), (64, 8), (8, 2), (4, 2)])
    d = rng.choice([128, 128, 64])
    L = rng.choice([4, 8, 16, 32])
    G = H_q // H_kv
    W = rng.choice([w for w in (8, 16, 32, 64) if G * w <= 256])
    snap = max(1, (L * 18) // 32)
    h2o = max(1, (L - snap) // 2)
    stream, tova = L - snap - h2o, 0
    geo = {"L": L, "H_q": H_q, "H_kv": H_kv, "d": d}
    pool, avg = rng.choice([5, 7, 7]), rng.random() < 0.6
    if kind in ("decode", "decode_attn"):
        B = rng.choice([1, 1, 2, 3, 4, 8, 16])
        budget = _log_int(rng, 128, 2048)
        hi = _log_int(rng, 4096, 16384)
        if rng.random() < 0.3:
            tova, snap, B = snap, 0, min(B, 4)  # more layers attend
        return {k: v for k, v in _case("", kind, B, max(budget + 300, hi // 2), max(budget + 300, hi),
                                       max(budget + 300, hi) + rng.choice([0, 1, 64]), W, pool, budget, snap, h2o, stream,
                                       tova=tova, avg=avg, steps=rng.choice([4, 8, 16, 32]), graph=rng.random() < 0.7,
                                       **geo).items() if k != "name"}
    if kind == "h2o_full":
        hi = _log_int(rng, 300, 6144)
        B = 1 if hi > 3000 else rng.choice([1, 2, 3])
    else:
        hi = _log_int(rng, 300, 32768)
        B = rng.choice([b for b in (1, 1, 2, 3, 4, 8) if b * hi <= 131072])
    lo = hi if B == 1 else max(200, hi // 2)
    budget = min(_log_int(rng, 96, 2048), max(96, hi // 4))
    S_cap = rng.choice([hi, (hi + 255) // 256 * 256, (hi + 255) // 256 * 256])
    return {k: v for k, v in _case("", kind, B, lo, hi, S_cap, W, pool, budget, snap, h2o, stream, avg=avg,
                                   **geo).items() if k != "name"}


# ---- shapes that follow from a case alone ---------------------------------------------------------

def _lens(c):
    r = random.Random("%d/%d/%d" % (c["B"], c["len_lo"], c["len_hi"]))
    return [r.randint(c["len_lo"], c["len_hi"]) for _ in range(c["B"])]


def _route(c):
    """(prefill, decode) operator per layer: contiguous blocks; SnapKV layers append in decode,
    TOVA layers compact with H2O's rule at the prefill."""
    pre = [SNAPKV] * c["snap"] + [H2O] * c["h2o"] + [STREAMING] * c["stream"] + [H2O] * c["tova"]
    dec = [FULL] * c["snap"] + [H2O] * c["h2o"] + [STREAMING] * c["stream"] + [TOVA] * c["tova"]
    return pre, dec


def _budgets(c):
    """Per-layer capacities: uniform for the decode arena, decreasing with depth for a mixed route."""
    L = c["L"]
    if c["kind"].startswith("decode") or c["h2o"] == 0:
        return [c["budget"]] * L
    return [max(c["W"] + 16, int(round(c["budget"] * (1.5 - l / max(L - 1, 1))))) for l in range(L)]


def _gen(seed, layer, what):
    return torch.Generator(device="cuda").manual_seed((seed * 1009 + layer) * 31 + what)


def _layer_inputs(c, seed, l, scoring):
    """K, V [B][H_kv][S_cap][d] and the window's (or, whole prompt, every position's) queries, bf16."""
    B, H, S, d, G = c["B"], c["H_kv"], c["S_cap"], c["d"], c["H_q"] // c["H_kv"]
    g = _gen(seed, l, 1)
    u = torch.randn((H, d), generator=g, device="cuda")
    u = u / u.norm(dim=1, keepdim=True)
    K = torch.randn((B, H, S, d), generator=g, device="cuda", dtype=torch.bfloat16)
    K[:, :, :SINK] += (SINK_LOGIT / LOGIT_STD * u)[None, :, None, :].to(torch.bfloat16)
    V = torch.randn((B, H, S, d), generator=g, device="cuda", dtype=torch.bfloat16)
    if not scoring:
        return K, V, None
    rows = S if c["kind"] == "h2o_full" and _route(c)[0][l] == H2O else c["W"]
    Q = torch.randn((B, H, G, rows, d), generator=g, device="cuda", dtype=torch.float32) * QUERY_NOISE
    Q += LOGIT_STD * math.sqrt(d) * u[None, :, None, None, :]
    return K, V, Q.to(torch.bfloat16).view(B, H * G, rows, d)


def _window_logits(c, K, Q, s, h, n):
    """fp64 logits [G][W][n] of the window rows of (s, h), masked causally, and which rows exist."""
    W, G, d = c["W"], c["H_q"] // c["H_kv"], c["d"]
    q = Q[s, h * G:(h + 1) * G].double()
    S = torch.matmul(q, K[s, h, :n].double().T) / math.sqrt(d)
    t = n - W + torch.arange(W, device="cuda")
    S.masked_fill_((torch.arange(n, device="cuda")[None, :] > t[:, None])[None], float("-inf"))
    return S, t >= 0


def _prefill_inputs(c, seed):
    pre, _ = _route(c)
    data = [_layer_inputs(c, seed, l, pre[l] in (SNAPKV, H2O)) for l in range(c["L"])]
    return [x[0] for x in data], [x[1] for x in data], [x[2] for x in data]


def _lse(c, seed, K, Q):
    """fp32 [B][H_q][W] log-sum-exp per scoring layer, as a prefill attention returns it."""
    out = []
    G, lens = c["H_q"] // c["H_kv"], _lens(c)
    for k, q in zip(K, Q):
        if q is None:
            out.append(None)
            continue
        x = torch.zeros((c["B"], c["H_q"], c["W"]), device="cuda")
        for s, n in enumerate(lens):
            t = n - c["W"] + torch.arange(c["W"], device="cuda")
            mask = torch.arange(n, device="cuda")[None, :] > t[:, None]
            for h in range(c["H_kv"]):
                S = torch.matmul(q[s, h * G:(h + 1) * G].float(), k[s, h, :n].float().T) / math.sqrt(c["d"])
                x[s, h * G:(h + 1) * G] = torch.logsumexp(S.masked_fill_(mask[None], float("-inf")), dim=-1)
        out.append(x)
    return out


def _supplied_scores(c, seed, l):
    """Column sums of a window's softmax rows, as a caller's attention leaves them: positive, spread
    over octaves, sinks high."""
    x = torch.randn((c["B"], c["H_kv"], c["S_cap"]), generator=_gen(seed, l, 2), device="cuda")
    x[:, :, :SINK] += SINK_LOGIT / LOGIT_STD
    x = torch.exp(LOGIT_STD * x)
    return x * (c["W"] / x.sum(dim=2, keepdim=True))


def _plan(c):
    pre, dec = _route(c)
    return kvev.Plan(c["L"], c["H_q"], c["H_kv"], c["d"], pre, _budgets(c), c["W"], c["pool"],
                     kvev.POOL_AVG if c["avg"] else kvev.POOL_MAX, SINK, route_decode=dec,
                     h2o_full_prompt=c["kind"] == "h2o_full")


# ---- decode ---------------------------------------------------------------------------------------

def _compacted(c, seed):
    """What a prefill eviction left: packed rows, positions in order, H2O seeds spread over octaves."""
    pre, budgets = _route(c)[0], _budgets(c)
    lens, units, d = _lens(c), c["B"] * c["H_kv"], c["d"]
    rows = units * sum(budgets)
    g = _gen(seed, 0, 3)
    bufs = {"out_K": torch.randn((rows, d), generator=g, device="cuda", dtype=torch.bfloat16),
            "out_V": torch.randn((rows, d), generator=g, device="cuda", dtype=torch.bfloat16),
            "h2o_state": torch.exp(LOGIT_STD * torch.randn(rows, generator=g, device="cuda")) * 1e-3,
            "out_idx": torch.empty(rows, dtype=torch.int32, device="cuda"),
            "out_count": torch.empty((c["L"], c["B"], c["H_kv"]), dtype=torch.int32, device="cuda")}
    at = 0
    for l, b in enumerate(budgets):
        idx = bufs["out_idx"][at: at + units * b].view(c["B"], c["H_kv"], b)
        at += units * b
        j = torch.arange(b, device="cuda")
        for s, n in enumerate(lens):
            if pre[l] == STREAMING:  # the sinks, then the recent rows
                idx[s] = torch.where(j < SINK, j, n - b + j).to(torch.int32)
            else:                    # spread over the prompt, then the recent rows
                old = b - b // 2
                idx[s] = torch.where(j < old, j * (n - b + old) // old, n - b + j).to(torch.int32)
        bufs["out_count"][l] = b
    return bufs


def _tokens(c, seed):
    """Per step and layer: the new token's k, v, q (or the caller's attention over the arena's slots)."""
    B, H, d, T = c["B"], c["H_kv"], c["d"], c["steps"]
    _, dec = _route(c)
    steps = []
    for t in range(T):
        g = _gen(seed, t, 4)
        k, v, x = [], [], []
        kk = torch.randn((c["L"], B, H, d), generator=g, device="cuda", dtype=torch.bfloat16)
        vv = torch.randn((c["L"], B, H, d), generator=g, device="cuda", dtype=torch.bfloat16)
        qq = torch.randn((c["L"], B, c["H_q"], d), generator=g, device="cuda", dtype=torch.bfloat16) * LOGIT_STD
        for l, b in enumerate(_budgets(c)):
            k.append(kk[l])
            v.append(vv[l])
            if dec[l] not in (H2O, TOVA):
                x.append(None)
            elif c["kind"] == "decode":
                x.append(qq[l])
            else:
                x.append(torch.softmax(LOGIT_STD * torch.randn((B, H, b + 1), generator=g, device="cuda"), dim=2))
        steps.append((k, v, x))
    return steps


def _generate(state):
    arena, c = state["arena"], state["case"]
    arena.init_from_prefill(state["bufs"], state["lens"])
    for k, v, x in state["tokens"]:
        if c["kind"] == "decode":
            arena.step(k, v, x)
        else:
            arena.step_attn(k, v, x)


# ---- the interface --------------------------------------------------------------------------------

def prepare(case, seed):
    c = case
    plan = _plan(c)
    lens = torch.tensor(_lens(c), dtype=torch.int32, device="cuda")
    state = {"case": c, "plan": plan, "lens": lens}
    if c["kind"].startswith("decode"):
        state["bufs"] = _compacted(c, seed)
        state["tokens"] = _tokens(c, seed)
        arena = kvev.DecodeArena(plan, c["B"], growth=c["steps"])
        arena.K.zero_()
        arena.V.zero_()
        state["arena"] = arena
        state["out"] = {"K": arena.K.view(torch.int16), "V": arena.V.view(torch.int16), "acc": arena.acc(),
                        "pos": arena.pos(), "count": arena.count(), "evicted": arena.evicted(), "lens": arena.lens()}
        if c["graph"]:
            _generate(state)  # the plan's first use sets up its device state, which a capture cannot
            torch.cuda.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                _generate(state)
        return state
    state["K"], state["V"], state["Q"] = _prefill_inputs(c, seed)
    state["bufs"] = plan.buffers(c["B"], c["S_cap"])
    state["bufs"]["workspace"].zero_()  # scores past a sequence's length are never written
    state["bufs"]["h2o_state"].zero_()  # rows of other layers are never written
    if c["kind"] == "lse":
        state["lse"] = _lse(c, seed, state["K"], state["Q"])
    if c["kind"] == "scored":
        pre, _ = _route(c)
        state["scores"] = [_supplied_scores(c, seed, l) if pre[l] in (SNAPKV, H2O) else None for l in range(c["L"])]
        state["Q"] = None
    bufs = state["bufs"]
    state["out"] = {"K": bufs["out_K"].view(torch.int16), "V": bufs["out_V"].view(torch.int16),
                    "idx": bufs["out_idx"], "count": bufs["out_count"], "h2o_state": bufs["h2o_state"]}
    if c["kind"] != "scored":
        state["out"]["scores"] = [plan.scores(bufs, c["B"], c["S_cap"], l) if state["Q"][l] is not None else None
                                  for l in range(c["L"])]
    return state


def run(state):
    c, plan = state["case"], state["plan"]
    if not c["kind"].startswith("decode"):
        plan.evict_prefill(state["K"], state["V"], state["Q"], state["lens"], c["B"], c["S_cap"], state["bufs"],
                           scores=state.get("scores"), lse=state.get("lse"))
    elif c["graph"]:
        state["graph"].replay()
    else:
        _generate(state)
    return state["out"]  # the caller's own buffers, which the call fills


def work(case):
    c = case
    pre, dec = _route(c)
    lens, b_l = _lens(c), _budgets(c)
    H, d, G, W = c["H_kv"], c["d"], c["H_q"] // c["H_kv"], c["W"]
    nbytes = flops = 0
    if c["kind"].startswith("decode"):
        for l in range(c["L"]):
            units, b = c["B"] * H, b_l[l]
            nbytes += units * b * (8 * d + 16)                       # hand-over: rows, position and state, read and written
            step = 8 * d                                             # the new row, read and written
            if dec[l] in (H2O, TOVA):
                step += 12 * b + (2 * d * (b + G) if c["kind"] == "decode" else 4 * (b + 1))  # pos, acc read and written, K
                flops += 2 * units * c["steps"] * G * d * b if c["kind"] == "decode" else 0
            elif dec[l] == STREAMING:
                step += 4 * b
            nbytes += units * step * c["steps"]
        return {"bytes": nbytes, "flops": flops}
    for l in range(c["L"]):
        for n in lens:
            b = min(b_l[l], n)
            nbytes += H * b * (6 * d + 4)                            # kept rows: V read, K and V written, index
            scored = pre[l] in (SNAPKV, H2O)
            if not scored:
                nbytes += H * b * 2 * d                              # StreamingLLM's kept K
                continue
            if c["kind"] == "scored":
                nbytes += H * (4 * n + 2 * d * b)
                continue
            nbytes += 2 * H * d * n                                  # every key
            rows = n if c["kind"] == "h2o_full" and pre[l] == H2O else W
            nbytes += 2 * H * G * d * rows
            flops += H * G * d * (n * (n + 1) if rows == n else 2 * n * W)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Scores are 32-bit sums of exponentials whose logits the tensor core sums in 32 bits: measured
    # against exact(), 1e-7 to 5e-7, and 1.1e-6 where the normalisers are given in 32 bits.  Positions
    # whose scores are equal to that precision may change places at a selection's threshold, which
    # moves the entries between them by one.
    if case["kind"] == "scored":
        return "exact"
    return {"rel": 5e-6, "max": 5e-5, "differ": 0.002}


def exact(case, seed):
    c = case
    if c["kind"] == "scored":
        return None  # copies and whole numbers only
    if c["kind"].startswith("decode"):
        return _exact_decode(c, seed)
    pre, _ = _route(c)
    lens, b_l, G, W = _lens(c), _budgets(c), c["H_q"] // c["H_kv"], c["W"]
    lse = None
    if c["kind"] == "lse":
        K, _, Q = _prefill_inputs(c, seed)
        lse = _lse(c, seed, K, Q)
    scores = []
    for l in range(c["L"]):
        if pre[l] not in (SNAPKV, H2O):
            scores.append(None)
            continue
        k, _, q = _layer_inputs(c, seed, l, True)
        out = torch.zeros((c["B"], c["H_kv"], c["S_cap"]), dtype=torch.float64, device="cuda")
        for s, n in enumerate(lens):
            if pre[l] == SNAPKV and n <= b_l[l]:
                continue  # every position is kept: nothing is scored
            for h in range(c["H_kv"]):
                if c["kind"] == "h2o_full" and pre[l] == H2O:
                    out[s, h, :n] = _prompt_sums(c, k[s, h, :n], q[s, h * G:(h + 1) * G, :n])
                    continue
                S, there = _window_logits(c, k, q, s, h, n)
                if lse is not None:
                    p = torch.exp(S - lse[l][s, h * G:(h + 1) * G].double()[..., None])
                else:
                    p = torch.softmax(S, dim=2)
                out[s, h, :n] = p[:, there].sum(dim=(0, 1)) / G
        scores.append(out)
    # the H2O seeds are those scores at the kept positions; which positions are kept is a matter of
    # whole numbers, compared as such
    return {"K": None, "V": None, "idx": None, "count": None, "h2o_state": None, "scores": scores}


def _prompt_sums(c, k, q):
    """(1/G) of each key's softmax weight summed over every prompt row that sees it."""
    n, G = k.shape[0], q.shape[0]
    kd = k.double()
    total = torch.zeros(n, dtype=torch.float64, device="cuda")
    pos = torch.arange(n, device="cuda")
    for g in range(G):
        for r0 in range(0, n, 2048):
            r1 = min(n, r0 + 2048)
            S = torch.matmul(q[g, r0:r1].double(), kd[:r1].T) / math.sqrt(c["d"])
            S.masked_fill_(pos[None, :r1] > pos[r0:r1, None], float("-inf"))
            total[:r1] += torch.softmax(S, dim=1).sum(dim=0)
    return total / G


def _exact_decode(c, seed):
    bufs, tokens, lens = _compacted(c, seed), _tokens(c, seed), _lens(c)
    _, dec = _route(c)
    B, H, d, G = c["B"], c["H_kv"], c["d"], c["H_q"] // c["H_kv"]
    U = B * H
    every = torch.arange(U, device="cuda")
    n0 = torch.tensor(lens, device="cuda").repeat_interleave(H)
    out, at = [], 0
    for l, b in enumerate(_budgets(c)):
        rows = slice(at, at + U * b)
        at += U * b
        pos = bufs["out_idx"][rows].long().view(U, b).clone()
        seeded = bufs["h2o_state"][rows].double().view(U, b).clone()
        if dec[l] not in (H2O, TOVA):
            # no attention is accumulated (only H2O-compacted layers are seeded, and those accumulate here)
            out.append(torch.zeros(U * (b + c["steps"] * (dec[l] == FULL)), dtype=torch.float64, device="cuda"))
            continue
        acc = seeded
        K = bufs["out_K"][rows].double().view(U, b, d)
        r = b // 2 if dec[l] == H2O else 0
        for t, (kn, _, x) in enumerate(tokens):
            k1 = kn[l].double().view(U, 1, d)
            if c["kind"] == "decode":
                q = x[l].double().view(U, G, d)
                S = torch.matmul(q, torch.cat([K, k1], dim=1).transpose(1, 2)) / math.sqrt(d)
                p = torch.softmax(S, dim=2).mean(dim=1)
            else:
                p = x[l].double().view(U, b + 1)
            a = torch.cat([acc, torch.zeros((U, 1), dtype=torch.float64, device="cuda")], dim=1) * (dec[l] == H2O) + p
            ps = torch.cat([pos, (n0 + t)[:, None]], dim=1)
            e = torch.where(ps < (n0 + t + 1 - r)[:, None], a, float("inf")).argmin(dim=1)
            acc = a[:, :b].clone()
            new = e < b  # the new token takes the evicted slot, unless it is the one evicted
            acc[every[new], e[new]] = a[new, b]
            pos[every[new], e[new]] = (n0 + t)[new]
            K[every[new], e[new]] = k1[new, 0]
        out.append(acc.reshape(-1))
    return {"K": None, "V": None, "acc": torch.cat(out), "pos": None, "count": None, "evicted": None, "lens": None}
