"""Performance cases of the TreeSpark hot path: what a serving program has the library do, call by call.

A program that decodes with draft trees runs one *round* per step: ``expand_tree`` builds every request's
draft tree from the drafter's base logits, the target model scores the tree (outside this library), and
``verify_tree`` walks it.  Around that stand the batch-wide node budget, the attention inputs and the
calibration statistics (``loop`` cases), and programs with a tree policy of their own call
``score_parents`` on a frontier they keep themselves (``score`` cases).

A case is a plain dict:
  kind    "round" = expand + verify; "loop" = expand, cut to a node budget, attention inputs, verify,
          calibration statistics and refit; "score" = one stand-alone scoring call
  B, V, D, r, K, Nmax, dtype    batch, vocabulary, block depth, Markov rank, sibling cap, node cap, input type
  T, theta                      temperature (0 = greedy) and stop price (>= 1 = the chain member of the ladder)
  logits  "peaked" = base logits as a trained drafter gives them (one planted favourite per depth);
          "flat" = no favourite: trees run into their node cap
  P       (score) number of parents; budget (loop) nodes per request handed out over the batch
Inputs follow the recipes of ``paper_2609_22098_b200.synth`` (same distributions; drawn with torch's
generator on the GPU, because they are made often): U = std * N(0,1) plus the planted favourites,
A ~ N(0, 1/r), W ~ N(0, 1/2), target logits = drafter logits + 0.8 * N(0,1) for every node of the tree
that the library grows from them.
"""
import dataclasses
import math

import torch

from paper_2609_22098_b200 import synth
from paper_2609_22098_b200.binding import TreeSpark

VOCAB = 151936


def _case(name, kind="round", B=32, V=VOCAB, D=8, r=64, K=8, Nmax=64, dtype="bf16", T=1.0, theta=0.1, logits="peaked", **more):
    return dict(name=name, kind=kind, B=B, V=V, D=D, r=r, K=K, Nmax=Nmax, dtype=dtype, T=T, theta=theta, logits=logits, **more)


def listed():
    return [
        # a small model all in fp32, one request: the smallest call, bound by latency and launches
        _case("tiny_f32", B=1, V=32000, D=4, r=16, K=4, Nmax=16, dtype="f32", theta=0.05),
        # interactive decoding of one request, sampled and greedy
        _case("single", B=1),
        _case("single_greedy", B=1, T=0.0),
        # a small odd batch at a price that lets the trees grow, temperature below one
        _case("batch5_t07", B=5, T=0.7, theta=0.08),
        # the ordinary serving batch, sampled
        _case("serve32", B=32),
        # full load: at the fixed price, and on the chain member of the price ladder (one child per node)
        _case("load128", B=128),
        _case("load128_chain", B=128, theta=1.0),
        # wide and deep trees on flat distributions: K = 16 siblings, up to 256 nodes
        _case("wide", B=8, V=128256, D=16, r=128, K=16, Nmax=256, T=0.7, theta=0.01, logits="flat"),
        # a head of rank 256, block of 7, at most 56 nodes
        _case("rank256", B=32, D=7, r=256, Nmax=56),
        # a vocabulary that is no multiple of anything (added tokens), bf16
        _case("ragged_vocab", B=8, V=50257),
        # the whole serving loop around a greedy round: budget, attention inputs, verification, calibration
        _case("loop32_greedy", kind="loop", B=32, V=128256, T=0.0, budget=8),
        # one stand-alone scoring call on a frontier with parents at mixed depths
        _case("score_frontier", kind="score", B=32, P=150),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, lo=32000, hi=VOCAB):
    return _log_int(rng, lo / 8, hi / 8) * 8


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    what = rng.choices(["single", "serve", "load", "wide", "rank256", "f32", "ragged", "loop", "score"],
                       [4, 6, 2, 2, 2, 2, 2, 2, 2])[0]
    T = rng.choice([0.0, 0.7, 1.0, 1.0])
    theta = round(math.exp(rng.uniform(math.log(0.05), math.log(0.4))), 3)
    shape = dict(V=_vocab(rng), D=rng.randint(5, 10), r=rng.choice([32, 48, 64, 64, 96]), K=rng.randint(4, 8),
                 Nmax=rng.randint(32, 80), T=T, theta=theta)
    if what == "single":
        c = _case("", B=rng.randint(1, 4), **shape)
    elif what == "serve":
        c = _case("", B=_log_int(rng, 5, 64), **shape)
    elif what == "load":
        c = _case("", B=rng.randint(65, 128), **dict(shape, D=rng.randint(5, 8), theta=rng.choice([1.0, max(theta, 0.1)]), Nmax=rng.randint(32, 64)))
    elif what == "wide":
        c = _case("", B=rng.randint(1, 8), logits="flat", **dict(shape, V=_vocab(rng, 32000, 128256), D=rng.randint(8, 16), r=rng.choice([64, 128]), K=rng.randint(9, 16),
                                                                Nmax=rng.randint(128, 256), T=rng.choice([0.7, 1.3]), theta=0.01))
    elif what == "rank256":
        c = _case("", B=rng.randint(1, 32), **dict(shape, D=7, r=256, Nmax=56))
    elif what == "f32":
        c = _case("", B=rng.randint(1, 4), dtype="f32", **dict(shape, V=_vocab(rng, 8000, 32000), D=rng.randint(4, 8), r=rng.choice([16, 24, 32]), K=4, Nmax=rng.randint(16, 48)))
    elif what == "ragged":
        c = _case("", B=rng.randint(1, 8), **dict(shape, V=_log_int(rng, 32000, 50256) | 1, r=rng.choice([32, 64])))
    elif what == "loop":
        c = _case("", kind="loop", B=_log_int(rng, 2, 64), budget=rng.randint(4, 16), **shape)
    else:
        c = _case("", kind="score", B=rng.randint(4, 32), P=_log_int(rng, 8, 512), **shape)
    del c["name"]
    return c


def _workload(case):
    base = synth.WORKLOADS["wide" if case["logits"] == "flat" else "serve32"]
    return dataclasses.replace(base, B=case["B"], V=case["V"], D=case["D"], r=case["r"], K=case["K"], Nmax=case["Nmax"],
                               dtype=case["dtype"], theta=case["theta"])


def prepare(case, seed):
    """Head weights, library context with its workspace, output buffers and one step's inputs."""
    wl, dev = _workload(case), "cuda"
    B, V, D, r, T = case["B"], case["V"], case["D"], case["r"], case["T"]
    g = torch.Generator(device=dev).manual_seed(seed)
    dt = wl.torch_dtype
    A = (torch.randn(V, r, generator=g, device=dev) * math.sqrt(1.0 / r)).to(dt)
    W = (torch.randn(r, V, generator=g, device=dev) * math.sqrt(0.5)).to(dt)
    full = torch.empty(B, D + 1, V, dtype=dt, device=dev)   # row D only feeds the target logits
    strength = wl.plant_lo + (wl.plant_hi - wl.plant_lo) * torch.rand(B, generator=g, device=dev)
    favourite = torch.randint(0, V, (B, D + 1), generator=g, device=dev)
    for b in range(B):
        u = torch.randn(D + 1, V, generator=g, device=dev) * wl.u_std
        if wl.plant_hi > 0.0:
            u.scatter_add_(1, favourite[b, :, None], strength[b].expand(D + 1, 1))
        full[b] = u.to(dt)
    anchor = torch.randint(0, V, (B,), generator=g, device=dev, dtype=torch.int32)
    theta = torch.full((B,), case["theta"], dtype=torch.float32, device=dev)
    ts = TreeSpark(V, D, r, case["K"], case["Nmax"], B, dtype=dt, calib_mode=1, calib_table=synth.make_calibration_table(wl, seed, "fit"))
    s = dict(ts=ts, kind=case["kind"], U=full[:, :D].contiguous(), A=A, W=W, anchor=anchor, theta=theta, T=T, round_seed=1000 + seed)
    if case["kind"] == "score":
        P = case["P"]
        s["req"] = torch.randint(0, B, (P,), generator=g, device=dev, dtype=torch.int32)
        s["dep"] = torch.randint(0, D, (P,), generator=g, device=dev, dtype=torch.int32)
        s["tok"] = torch.randint(0, V, (P,), generator=g, device=dev, dtype=torch.int32)
        s["hash"] = torch.randint(0, 2 ** 62, (P,), generator=g, device=dev, dtype=torch.int64)
        s["out"] = ts.alloc_score_outputs(P)
        return s
    s["tree"], s["verdict"] = ts.alloc_tree(B), ts.alloc_verdict(B)
    ts.expand_tree(s["U"], A, W, anchor, theta, T, s["round_seed"], out=s["tree"])
    if case["kind"] == "loop":
        s["budget"] = B * case["budget"]
        s["price"] = torch.zeros(1, dtype=torch.float32, device=dev)
        s["base_pos"] = torch.randint(0, 4096, (B,), generator=g, device=dev, dtype=torch.int32)
        R = case["Nmax"] + 1
        s["attn"] = dict(flat_tok=torch.empty(B, R, dtype=torch.int32, device=dev), pos_ids=torch.empty(B, R, dtype=torch.int32, device=dev),
                         dense_mask=torch.empty(B, R, R, dtype=torch.float32, device=dev))
        s["stats"] = ts.calib_new_stats()
        s["table"] = torch.empty(D, 16, dtype=torch.float32, device=dev)
        s["platt"] = torch.empty(4, dtype=torch.float64, device=dev)
        ts.allocate_budget(s["tree"], s["budget"], s["price"])
    s["Z"], s["zoff"] = _targets(s, full, g)
    return s


def _targets(s, full, g):
    """Target logits of every node of every tree (root first): the drafter's own logits plus noise."""
    tree, A, Wf = s["tree"], s["A"], s["W"].float()
    B, V = full.shape[0], full.shape[2]
    n = tree["n_nodes"].tolist()
    req = torch.cat([torch.full((n[b] + 1,), b) for b in range(B)]).cuda()
    dep = torch.cat([torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), tree["depth"][b, :n[b]].long()]) for b in range(B)])
    tok = torch.cat([torch.cat([s["anchor"][b:b + 1].long(), tree["tok"][b, :n[b]].long()]) for b in range(B)])
    off = torch.zeros(B + 1, dtype=torch.int64)
    off[1:] = torch.cumsum(torch.tensor(n) + 1, 0)
    Z = torch.empty(int(off[-1]), V, dtype=full.dtype, device="cuda")
    for i in range(0, Z.shape[0], 128):
        j = min(i + 128, Z.shape[0])
        z = A[tok[i:j]].float() @ Wf
        z += full[req[i:j], dep[i:j]].float()
        z += 0.8 * torch.randn(j - i, V, generator=g, device="cuda")
        Z[i:j] = z.to(full.dtype)
    return Z, off.cuda()


def run(s):
    """One pass, as the program's step calls it."""
    ts = s["ts"]
    if s["kind"] == "score":
        return ts.score_parents(s["U"], s["A"], s["W"], s["req"], s["dep"], s["tok"], s["hash"], s["T"], s["round_seed"], out=s["out"])
    tree = ts.expand_tree(s["U"], s["A"], s["W"], s["anchor"], s["theta"], s["T"], s["round_seed"], out=s["tree"])
    out = {}
    if s["kind"] == "loop":
        ts.allocate_budget(tree, s["budget"], s["price"])
        out["attn"] = ts.emit_attention_inputs(s["anchor"], tree, s["base_pos"], out=s["attn"])
        out["price"] = s["price"]
    verdict = ts.verify_tree(s["U"], s["A"], s["W"], s["Z"], s["zoff"], s["anchor"], tree, s["T"], s["round_seed"], out=s["verdict"])
    if s["kind"] == "loop":
        ts.calib_accumulate(tree, verdict, s["stats"])
        # (the refit carries the running sums; their units of 2^-24 sit below what fp32 log-sum-exps determine)
        out["table"], out["platt"] = ts.calib_refit(s["stats"], population=0, table=s["table"], platt=s["platt"])
    out["tree"], out["verdict"] = tree, verdict
    return out


def _expected(case):
    """(nodes, scored parents, levels with parents) per request, about: which trees grow depends on the inputs."""
    D, N, K = case["D"], case["Nmax"], case["K"]
    if case["theta"] >= 1.0:
        return min(D, N), min(D, N), D
    if case["logits"] == "flat":
        return (N, 0.6 * N, 4) if case["T"] < 1.0 else (min(N, 110.0), 20.0, 3)
    n = min(N, 13.5 * (0.1 / case["theta"]) ** 0.8)
    return n, (n + 1 if case["T"] == 0.0 else 0.35 * n + 1), min(D, 3)


def work(case):
    es = 2 if case["dtype"] == "bf16" else 4
    B, V, r = case["B"], case["V"], case["r"]
    row = V * es
    if case["kind"] == "score":
        P = case["P"]
        rows = B * case["D"] * (1.0 - (1.0 - 1.0 / (B * case["D"])) ** P)   # distinct base-logit rows among P random parents
        return {"bytes": rows * row + r * row + P * (r * es + 8 * case["K"] * 2 + 28), "flops": 2.0 * r * V * P}
    nodes, parents, levels = _expected(case)
    targets = (min(nodes, case["budget"]) if case["kind"] == "loop" else nodes) + 1
    # every base-logit row with a parent, W, the parents' head rows and every target row once; the trees out
    nbytes = B * levels * row + r * row + B * parents * r * es + B * targets * row + B * nodes * 60.0
    if case["kind"] == "loop":
        nbytes += B * (case["Nmax"] + 1) ** 2 * 4.0
    return {"bytes": nbytes, "flops": 2.0 * r * V * B * parents}


def tolerance(case):
    """Scalars are fp32 log-sum-exps over the vocabulary and differences of them: 1e-5; tokens and tree shapes are the
    same except where two candidates tie within that error."""
    return {"rel": 1e-5, "max": 4e-4, "differ": 0.005}
