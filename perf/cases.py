"""The measured workloads of the decode tail: what a serving or training program has it do.

A case is a dict of sizes and options; ``kind`` names the entry point:

  tail     DecodeTail.tail            one fused block step, the call of a decode loop
  graph    DecodeTail.graph / launch  the same step captured once and replayed
  topk     DecodeTail.topk            candidate extraction alone
  select   DecodeTail.select          the corrector alone, on given candidates
  verify   DecodeTail.verify          verification alone, on given selections
  replay   DecodeTail.replay          same-state replay diagnostics of a block
  distill  DecodeTail.distill_loss    distillation loss and its gradient
  fold     DecodeTail.prepare, then DecodeTail.select: new weights, then the head on one block

Logits are drawn as a trained model's look: a N(0, 1.5) bulk over the vocabulary and 24 plausible
ids a row well above it, so that nearly all of the probability sits on a few ids (the bulk holds
about 1e-4 of it). The verifier is the proposal plus noise with its argmax planted on the
proposal's first id with probability `agree`, else on another plausible id or, rarely, on any.
"""
import functools
import math

import torch

from paper_2609_33390_gb300 import brisk

F64 = torch.float64
PLAUSIBLE = 24
BETA = 0.01
CHUNK = 1 << 27          # logits handled at once while inputs or exact values are made


def _case(name, kind, B, L, V, d, K, r, logits="bf16", hidden="bf16", select="greedy",
          verify="greedy", agree=0.9):
    return {"name": name, "kind": kind, "B": B, "L": L, "V": V, "d": d, "K": K, "r": r,
            "logits": logits, "hidden": hidden, "select": select, "verify": verify,
            "agree": agree}


def listed():
    return [
        # the smallest fp32 model, one sequence: bound by launches and latency
        _case("tail_tiny_fp32", "tail", 1, 8, 32000, 512, 4, 64, "f32", "f32"),
        # one interactive sequence on a full-size model, called block by block
        _case("tail_one_sequence", "tail", 1, 32, 126464, 4096, 8, 256),
        # the same as a captured graph, the way a latency-bound server runs it
        _case("graph_one_sequence", "graph", 1, 32, 126464, 4096, 8, 256),
        # a small batch with sampled selections and speculative-sampling verification
        _case("tail_16_stochastic", "tail", 16, 32, 126464, 4096, 8, 256, select="sample",
              verify="stochastic"),
        # long blocks, many candidates, the widest corrector and the largest vocabulary
        _case("tail_64_wide", "tail", 64, 64, 151936, 3584, 16, 512),
        # the throughput server's step: a large batch
        _case("tail_128_stream", "tail", 128, 32, 126464, 4096, 8, 256, agree=0.8),
        # candidates alone with rows that start at any alignment, for a caller with its own head
        _case("topk_ragged", "topk", 7, 13, 100003, 64, 20, 32),
        # the corrector alone with fp32 weights and odd sizes (an unquantised head in evaluation)
        _case("select_fp32", "select", 12, 24, 32003, 1000, 10, 96, "f32", "f32", "sample"),
        # verification alone of greedy selections by speculative sampling, fp32 ragged rows
        _case("verify_fp32_ragged", "verify", 5, 48, 64007, 64, 8, 32, "f32", "f32",
              verify="stochastic"),
        # diagnostics of a trained head over an evaluation batch
        _case("replay_32", "replay", 32, 32, 126464, 4096, 8, 256, select="sample"),
        # one training step's loss and gradient of the head
        _case("distill_128", "distill", 128, 32, 32000, 64, 16, 64),
        # after each weight update of the head: fold the vocabulary, then score a block
        _case("fold_126k", "fold", 8, 32, 126464, 4096, 8, 256),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tail", "tail", "tail", "graph", "topk", "select", "verify", "replay",
                       "distill", "fold"])
    logits = rng.choice(["bf16", "bf16", "f32"])
    hidden = rng.choice(["bf16", "bf16", "f32"])
    V = _log_int(rng, 1000, 152000)
    L = rng.randint(2, 64)
    K = rng.choice([4, 6, 8, 8, 13, 16, 32])
    r = 16 * rng.randint(1, 32)
    d = 8 * _log_int(rng, 8, 512)
    B = _log_int(rng, 1, 128)
    if kind == "fold":
        B, L = min(B, 16), min(L, 32)
    if kind == "fold" and hidden == "f32":
        V, d = min(V, 50000), min(d, 2048)
    # no more than the largest listed case: 2.4 GB of logits for both tensors
    size = 4 if logits == "f32" else 2
    B = max(1, min(B, int(2.4e9 / (2 * L * V * size))))
    c = _case("", kind, B, L, V, d, K, r, logits, hidden, rng.choice(["greedy", "sample"]),
              rng.choice(["greedy", "stochastic"]), round(rng.uniform(0.6, 0.98), 3))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _dt(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _rows_at_once(V):
    return max(1, CHUNK // V)


def _logits(c, g, dev, verifier=True):
    """Proposal and verifier logits [B, L, V]."""
    rows, V = c["B"] * c["L"], c["V"]
    dt = _dt(c["logits"])
    lq = torch.empty((rows, V), dtype=dt, device=dev)
    lp = torch.empty_like(lq) if verifier else None
    stratum = V // PLAUSIBLE
    first = torch.arange(PLAUSIBLE, device=dev) * stratum
    for s in range(0, rows, _rows_at_once(V)):
        n = min(_rows_at_once(V), rows - s)
        q = torch.randn((n, V), generator=g, device=dev) * 1.5
        at = first + torch.randint(stratum, (n, PLAUSIBLE), generator=g, device=dev)
        q.scatter_(1, at, 16.0 + 3.0 * torch.randn((n, PLAUSIBLE), generator=g, device=dev))
        lq[s:s + n] = q.to(dt)
        if not verifier:
            continue
        q = lq[s:s + n].float()
        p = q + 0.5 * torch.randn((n, V), generator=g, device=dev)
        u = torch.rand((n, 4), generator=g, device=dev)
        other = at.gather(1, (u[:, 1:2] * PLAUSIBLE).long().clamp_(max=PLAUSIBLE - 1))[:, 0]
        anyid = (u[:, 2] * V).long().clamp_(max=V - 1)
        other = torch.where(u[:, 3] < 0.1, anyid, other)
        target = torch.where(u[:, 0] < c["agree"], q.argmax(1), other)[:, None]
        margin = torch.empty((n, 1), device=dev).exponential_(1 / 2.0, generator=g)
        p.scatter_(1, target, p.amax(1, keepdim=True) + margin)
        lp[s:s + n] = p.to(dt)
    shape = (c["B"], c["L"], V)
    return lq.view(shape), None if lp is None else lp.view(shape)


def _weights(c, g, dev):
    r, d, S, dt = c["r"], c["d"], 2 * c["r"], _dt(c["hidden"])
    shapes = {"P_h": (r, d), "P_e": (r, d), "P_phi": (16, 5), "pos": (c["L"], 16),
              "W0": (S, 2 * r), "Wz": (S, 2 * r + 32), "Wh": (S, 2 * r + 32), "W_s": (r, S),
              "W_c": (r, d), "w_g": (S + 5,)}
    w = {k: (0.02 * torch.randn(s, generator=g, device=dev)).to(dt) for k, s in shapes.items()}
    for k in ("E_in", "E_out"):
        w[k] = torch.empty((c["V"], d), dtype=dt, device=dev)
        n = max(1, CHUNK // d)
        for s in range(0, c["V"], n):
            rows = w[k][s:s + n]
            rows.copy_(torch.randn(rows.shape, generator=g, device=dev))
    w["b_g"], w["alpha"] = 0.25, 0.5
    return w


def _small(c, g, dev):
    """Hidden states, anchors and uniforms of a block."""
    B, L, d, dt = c["B"], c["L"], c["d"], _dt(c["hidden"])
    b = {"hidden": torch.randn((B, L, d), generator=g, device=dev).to(dt),
         "h_c": torch.randn((B, d), generator=g, device=dev).to(dt),
         "x0": torch.randint(c["V"], (B,), generator=g, device=dev, dtype=torch.int32)}
    for k in ("u_sel", "u_acc", "u_res"):
        b[k] = torch.rand((B, L), generator=g, device=dev)
    return b


def _inputs(c, seed):
    """Everything that the path reads, made from the seed alone."""
    dev = torch.device("cuda")
    g = torch.Generator(dev).manual_seed(int(seed))
    kind, K = c["kind"], c["K"]
    x = {"block": _small(c, g, dev)}
    lq, lp = _logits(c, g, dev, verifier=kind in ("tail", "graph", "verify", "replay", "distill"))
    x["block"]["logits_q"], x["block"]["logits_p"] = lq, lp
    if kind in ("tail", "graph", "select", "replay", "fold"):
        x["weights"] = _weights(c, g, dev)
    if kind in ("select", "verify", "distill", "fold"):
        # what the steps before the call leave: candidates, scores, selections
        ids, lpr, _ = _candidates(lq, K)
        x["cand_ids"], x["cand_logprob"] = ids.int(), lpr.float()
        if kind in ("verify", "distill"):
            noise = torch.randn(lpr.shape, generator=g, device=dev, dtype=F64)
            x["refined"] = (lpr + 0.7 * noise).float()
            rank = _pick(x["refined"].double(), c["select"], x["block"]["u_sel"])
            x["sel"] = x["cand_ids"].gather(2, rank[..., None])[..., 0].contiguous()
            x["accepted"] = torch.randint(c["L"] + 1, (c["B"],), generator=g, device=dev,
                                          dtype=torch.int32)
            x["block"]["logits_q"] = None
    return x


def _no_weights(c):
    """Placeholder corrector parameters for a program that never calls the corrector."""
    t = torch.zeros(8, dtype=_dt(c["hidden"]), device="cuda")
    names = ("E_in", "E_out", "P_h", "P_e", "P_phi", "pos", "W0", "Wz", "Wh", "W_s", "W_c", "w_g")
    return dict({n: t for n in names}, b_g=0.0, alpha=0.0)


@functools.lru_cache(maxsize=1)
def _graph_stream():
    """The one stream of a decode loop: its replays run one after another."""
    return torch.cuda.Stream()


def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    weights = x.get("weights") or _no_weights(c)
    tail = brisk.DecodeTail(c["B"], c["L"], c["V"], c["d"], c["K"], c["r"], _dt(c["logits"]),
                            _dt(c["hidden"]), weights)
    sm, vm = brisk.mode_ids(c["select"], c["verify"])
    x.update(kind=c["kind"], tail=tail, sm=sm, vm=vm)
    if c["kind"] in ("tail", "graph", "select", "replay"):
        tail.prepare()
    if c["kind"] == "tail":
        x["out"] = tail.alloc_outputs()
    if c["kind"] == "graph":
        x["graph"] = tail.graph(x["block"], sm, vm, chain_anchor=False, stream=_graph_stream())
    return x


def run(state):
    x, tail, b = state, state["tail"], state["block"]
    kind = x["kind"]
    if kind == "tail":
        return tail.tail(b, x["sm"], x["vm"], out=x["out"])
    if kind == "graph":
        return x["graph"].launch()
    if kind == "topk":
        return tail.topk(b["logits_q"])
    if kind == "verify":
        return tail.verify(b["logits_p"], x["sel"], x["cand_ids"], x["refined"], x["sm"], x["vm"],
                           u_acc=b["u_acc"], u_res=b["u_res"])
    if kind == "replay":
        return tail.replay(b, x["sm"])
    if kind == "distill":
        return tail.distill_loss(b["logits_p"], x["cand_ids"], x["cand_logprob"], x["refined"],
                                 x["accepted"], BETA)
    if kind == "fold":
        tail.prepare()
    return tail.select(b["hidden"], b["h_c"], b["x0"], b["logits_q"], x["cand_ids"],
                       x["cand_logprob"], x["sm"], u_sel=b["u_sel"])


# ---------------------------------------------------------------- what is counted

def work(case):
    """Bytes: the logits, hidden states, weights and folded table rows that a pass reads, once
    each, and its outputs. Flops: the products, the residual dots and the sums of exponentials."""
    c = case
    B, L, V, d, K, r = (c[k] for k in ("B", "L", "V", "d", "K", "r"))
    kind, S, rows = c["kind"], 2 * c["r"], c["B"] * c["L"]
    ls = 4 if c["logits"] == "f32" else 2
    hs = 4 if c["hidden"] == "f32" else 2
    sweep_b, sweep_f = rows * V * ls, 3 * rows * V
    # the head: hidden states and their two products, K residual rows and a token row a position
    head_b = (rows + B) * d * hs + r * d * hs + 3 * S * r * hs + rows * (K + 2) * S * 4 + \
        rows * K * 12
    head_f = 2 * (rows + B) * d * r + 2 * (2 * rows + B) * S * r + 2 * rows * S * (K + 12)
    out_b = rows * K * 12
    if kind in ("tail", "graph", "replay"):
        return {"bytes": 2 * sweep_b + head_b + out_b, "flops": 2 * sweep_f + head_f}
    if kind == "topk":
        return {"bytes": sweep_b + out_b, "flops": sweep_f}
    if kind == "verify":
        return {"bytes": sweep_b + out_b, "flops": sweep_f}
    if kind == "select":
        return {"bytes": head_b + out_b, "flops": head_f}
    if kind == "distill":
        return {"bytes": rows * K * (16 + 32), "flops": 40 * rows * K}
    fold_b = 2 * V * d * hs + (2 * r * d + 4 * S * r) * hs + 4 * V * S * 4
    fold_f = 4 * V * d * r + 8 * V * S * r
    return {"bytes": fold_b + head_b + out_b, "flops": fold_f + head_f}


def tolerance(case):
    """fp32 sums over the vocabulary and the head's products: with bf16 weights the refined scores
    are up to 7e-6 off 64 bits (the products' long accumulations). `differ`: rare ties only."""
    return {"rel": 3e-5, "max": 5e-4, "differ": 0.002}


# ---------------------------------------------------------------- in 64 bits

def _ordered(x):
    """Integers in the order of the fp32 values x (-0 and +0 alike)."""
    i = (x.float() + 0.0).view(torch.int32).long()
    return torch.where(i >= 0, i, -(i & 0x7FFFFFFF))


def _candidates(logits, K):
    """Ordered candidates (logit descending, id ascending), their log-probabilities, the
    log-partition: [B, L, K] int64 and float64, [B, L] float64."""
    B, L, V = logits.shape
    flat = logits.view(B * L, V)
    ids, lpr, lse = [], [], []
    rank = (1 << 20) - 1 - torch.arange(V, device=logits.device)
    n = max(1, _rows_at_once(V) // 4)
    for s in range(0, B * L, n):
        row = flat[s:s + n]
        i = torch.topk(_ordered(row) * (1 << 20) + rank, K, dim=1).indices
        z = torch.logsumexp(row.double(), 1)
        ids.append(i)
        lse.append(z)
        lpr.append(row.gather(1, i).double() - z[:, None])
    return (torch.cat(ids).view(B, L, K), torch.cat(lpr).view(B, L, K),
            torch.cat(lse).view(B, L))


def _verifier(logits):
    """Argmax (lowest id) and log-partition of the verifier rows."""
    ids, _, lse = _candidates(logits, 1)
    return ids[..., 0], lse


def _pick(scores, mode, u):
    """Select: the rank of the best score, or the inverse-CDF draw with u."""
    if mode == "greedy":
        return scores.argmax(-1)
    cum = torch.exp(scores - scores.amax(-1, keepdim=True)).cumsum(-1)
    hit = cum > u.double()[..., None] * cum[..., -1:]
    return hit.long().argmax(-1)


def _corrector(c, w, b, ids, lpr, base=False):
    """Selections' ranks, refined scores [B, L, K] and the ranks fed forward."""
    B, L, K = ids.shape
    W = {k: v.double() for k, v in w.items() if torch.is_tensor(v) and k not in ("E_in", "E_out")}
    hm = b["hidden"].double() @ W["P_h"].T
    prev = b["x0"].long()
    e = w["E_in"][prev].double() @ W["P_e"].T
    s = torch.tanh(torch.cat([b["h_c"].double() @ W["P_h"].T, e], 1) @ W["W0"].T)
    lq = b["logits_q"]
    refined = torch.empty((B, L, K), dtype=F64, device=ids.device)
    ranks, fed = torch.empty_like(ids[..., 0]), torch.empty_like(ids[..., 0])
    for i in range(L):
        ci = ids[:, i]
        top = lq[:, i].gather(1, ci[:, :4]).double()
        lprev = lq[:, i].gather(1, prev[:, None]).double()[:, 0]
        phi = torch.stack([top[:, 0] - top[:, 1], top[:, 0] - top[:, 3],
                           (prev == ci[:, 0]).double(),
                           (prev[:, None] == ci[:, :4]).any(1).double(), top[:, 0] - lprev], 1)
        e = w["E_in"][prev].double() @ W["P_e"].T
        x = torch.cat([hm[:, i], e, W["pos"][i].expand(B, -1), phi @ W["P_phi"].T], 1)
        z = torch.sigmoid(x @ W["Wz"].T)
        s = (1 - z) * s + z * (x @ W["Wh"].T)
        cand = w["E_out"][ci].double() @ W["W_c"].T
        dot = torch.einsum("bkr,br->bk", cand, s @ W["W_s"].T)
        gate = torch.sigmoid(torch.cat([s, phi], 1) @ W["w_g"] + w["b_g"])
        gate = gate / (1 + math.exp(-w["alpha"]))
        refined[:, i] = lpr[:, i].double() + gate[:, None] * dot
        u = b["u_sel"][:, i]
        ranks[:, i] = _pick(refined[:, i], c["select"], u)
        fed[:, i] = _pick(lpr[:, i].double(), c["select"], u) if base else ranks[:, i]
        prev = ci.gather(1, fed[:, i:i + 1])[:, 0]
    return ranks, refined, fed


def _verified(c, lp, b, sel, ids, refined):
    """Accepted lengths, committed tokens and corrections."""
    B, L, V = lp.shape
    amax, lse = _verifier(lp)
    rank = (ids == sel[..., None]).long().argmax(-1)
    pi = torch.softmax(refined.double(), -1)
    if c["select"] == "greedy":
        pi = torch.zeros_like(pi).scatter_(2, rank[..., None], 1.0)
    if c["verify"] == "greedy":
        ok = sel == amax
    else:
        px = torch.exp(lp.gather(2, sel[..., None])[..., 0].double() - lse)
        ok = b["u_acc"].double() < (px / pi.gather(2, rank[..., None])[..., 0]).clamp(max=1)
    acc = torch.where(ok.all(1), torch.full((B,), L, device=lp.device),
                      (~ok).long().argmax(1))
    corr = torch.full((B,), -1, dtype=torch.long, device=lp.device)
    out = torch.full((B, L), -1, dtype=torch.long, device=lp.device)
    for n, a in enumerate(acc.tolist()):
        out[n, :a] = sel[n, :a]
        if a == L:
            continue
        corr[n] = amax[n, a]
        if c["verify"] == "stochastic":
            res = torch.exp(lp[n, a].double() - lse[n, a])
            res.scatter_add_(0, ids[n, a], -pi[n, a])
            cum = res.clamp_(min=0).cumsum(0)
            if float(cum[-1]) > 1e-6:
                corr[n] = (cum > b["u_res"][n, a].double() * cum[-1]).long().argmax()
        out[n, a] = corr[n]
    return acc, out, corr


def _distilled(c, x):
    B, L, V = x["block"]["logits_p"].shape
    lp = x["block"]["logits_p"].gather(2, x["cand_ids"].long()).double()
    logr = torch.log_softmax(x["refined"].double(), -1)
    logq = torch.log_softmax(x["cand_logprob"].double(), -1)
    p, q = torch.softmax(lp, -1), logq.exp()
    reach = x["accepted"].long().clamp(max=L - 1)[:, None] >= torch.arange(L, device=lp.device)
    n = reach.sum()
    loss = (-(p * logr).sum(-1) + BETA * (q * (logq - logr)).sum(-1))[reach].sum() / n
    grad = ((logr.exp() - p) + BETA * (logr.exp() - q)) * reach[..., None] / n
    return {"loss": loss.view(1), "grad": grad}


def exact(case, seed):
    c = case
    x = _inputs(c, seed)
    b, kind = x["block"], c["kind"]
    if kind == "topk":
        ids, lpr, lse = _candidates(b["logits_q"], c["K"])
        return {"cand_ids": ids, "cand_logprob": lpr, "lse_q": lse}
    if kind == "distill":
        return _distilled(c, x)
    if kind == "verify":
        acc, out, corr = _verified(c, b["logits_p"], b, x["sel"].long(), x["cand_ids"].long(),
                                   x["refined"])
        return {"accepted_len": acc, "out_tokens": out, "correction": corr}
    if kind in ("select", "fold"):
        ids = x["cand_ids"].long()
        ranks, refined, _ = _corrector(c, x["weights"], b, ids, x["cand_logprob"])
        return {"sel_tokens": ids.gather(2, ranks[..., None])[..., 0], "refined": refined}
    ids, lpr, lse = _candidates(b["logits_q"], c["K"])
    ranks, refined, fed = _corrector(c, x["weights"], b, ids, lpr, base=kind == "replay")
    sel = ids.gather(2, ranks[..., None])[..., 0]
    if kind == "replay":
        return {"head_tokens": sel, "flags": None, "first_breaker": None, "refined": refined}
    acc, out, corr = _verified(c, b["logits_p"], b, sel, ids, refined)
    return {"accepted_len": acc, "out_tokens": out, "correction": corr,
            "next_anchor": torch.where(acc < c["L"], corr, sel[:, -1]), "cand_ids": ids,
            "cand_logprob": lpr, "lse_q": lse, "sel_tokens": sel, "refined": refined}
