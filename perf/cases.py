"""The calls whose speed this library is measured by, through its public entry points.

A parameter server calls one of these once per training round: the whole round
(`aspis_round`), the same round as its four steps (`aspis_check`, `aspis_detect`,
`aspis_select`, `aspis_aggregate`: what a server sharded by coordinates calls), the
round for copies that are not bit-identical, the round from pinned host memory, the
model update that follows, or the clique search alone on a graph of more workers.
Inputs are shaped like the evaluation of the method: K workers, every r-subset of them
holds one file, each file has r copies of its gradient of d fp32 values, q colluding
workers return distorted copies (ALIE, reversed or inner-product gradients).
"""
from __future__ import annotations

import itertools
import math
import random

import torch

import paper_2108_02416_gb300 as ap

TAU, NOISE = 1e-4, 1e-6               # tolerant round: bound and std of the per-copy noise
ETA, MU = 0.05, 0.9                    # model update: step and momentum of the experiments
MOST_BYTES = 61.1e9                    # copies of the largest listed case

# (workers, copies per file) of the evaluation's tables and of the tests, with the largest
# number of adversaries drawn for them (2 q <= K, so that the optimal attack exists)
CLUSTERS = [(7, 3, 3), (15, 3, 6), (21, 3, 8), (24, 3, 8), (15, 5, 6), (15, 2, 5), (10, 4, 4), (12, 4, 5)]


def _round(name, K, r, d, q, attack, distortion, kind="round", padded=True, mode="median"):
    return {"name": name, "kind": kind, "K": K, "r": r, "d": d, "q": q, "attack": attack,
            "distortion": distortion, "padded": padded, "mode": mode}


def listed():
    return [
        # the smallest round in use, a toy model on 7 workers: latency and launches
        _round("round_k7_d4k", 7, 3, 4096, 2, "weak", "alie"),
        # one layer (3x3 convolution, 64 to 64 channels, with its normalisation) aggregated by itself
        _round("round_k15_layer", 15, 3, 36_928, 3, "strong", "alie"),
        # an ordinary round as its four calls, as a server sharded by coordinates issues them
        _round("steps_k15_d1m", 15, 3, 1_048_576, 3, "weak", "reversed", kind="steps"),
        # the headline round: a flattened ResNet-18 gradient on 15 workers, optimal attack
        _round("round_k15_d11m", 15, 3, 11_173_962, 3, "strong", "alie"),
        # the larger cluster of the evaluation: 1,330 files
        _round("round_k21_d2m", 21, 3, 2_097_152, 5, "strong", "alie"),
        # higher redundancy: 3,003 files of five copies
        _round("round_k15_r5_d1m", 15, 5, 1_048_576, 4, "strong", "alie"),
        # copies stacked as they come, an odd length without padding: rows at any 4-byte address
        _round("round_k15_unpadded", 15, 3, 1_000_003, 3, "weak", "alie", padded=False),
        # the mean, the aggregator of Algorithm 1 after a successful detection
        _round("round_k15_mean", 15, 3, 1_048_576, 3, "weak", "reversed", mode="mean"),
        # copies that differ by floating-point effects: closeness, averages, then the median
        _round("tolerant_k15_d1m", 15, 3, 1_048_576, 3, "strong", "alie", kind="tolerant"),
        # copies that arrive in pinned host memory: transfer, round and read-back
        _round("host_k15_d64k", 15, 3, 65_536, 3, "strong", "alie", kind="host"),
        # the model update of a ResNet-18 with momentum
        {"name": "sgd_d11m", "kind": "sgd", "d": 11_173_962, "mu": MU},
        # the clique search on 100 workers under the optimal attack (the method's timing table)
        {"name": "wide_k100", "kind": "wide", "K": 100, "r": 5, "q": 25, "attack": "strong", "all": False},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["round", "steps", "tolerant", "host", "sgd", "wide"], [12, 2, 2, 1, 1, 1])[0]
    if kind == "sgd":
        return {"kind": "sgd", "d": _log_uniform(rng, 1000, 11_173_962), "mu": rng.choice([MU, MU, 0.0])}
    if kind == "wide":
        K = rng.randint(33, 128)
        return {"kind": "wide", "K": K, "r": rng.choice([3, 5]), "q": rng.randint(2, K // 2 - 1),
                "attack": rng.choice(["weak", "strong"]), "all": rng.random() < 0.5}
    K, r, most_q = rng.choice(CLUSTERS)
    cap = {"round": MOST_BYTES, "steps": MOST_BYTES, "tolerant": 6e9, "host": 1e9}[kind]
    lo = 1000 if kind != "host" else 1024
    d = _log_uniform(rng, lo, min(11_173_962, cap / (math.comb(K, r) * r * 4)))
    case = _round("", K, r, d, rng.randint(2, most_q), rng.choice(["weak", "strong"]),
                  rng.choice(["alie", "reversed", "foe"]), kind=kind, padded=rng.random() < 0.7,
                  mode="median" if rng.random() < 0.8 else "mean")
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _sides(case, seed):
    """(A, D): the colluding workers and, for the optimal attack, those they disagree with."""
    perm = list(range(case["K"]))
    random.Random(seed * 7919 + 1).shuffle(perm)
    q = case["q"]
    return set(perm[:q]), set(perm[q: 2 * q]) if case["attack"] == "strong" else set()


def _files(case):
    return list(itertools.combinations(range(case["K"]), case["r"]))


def _distorted_rows(case, seed):
    """Row numbers i*r + s of the copies that adversaries distort."""
    A, D = _sides(case, seed)
    most = (case["r"] + 1) // 2
    rows = []
    for i, ws in enumerate(_files(case)):
        if case["attack"] == "strong" and not (all(w in A or w in D for w in ws) and
                                               sum(w in A for w in ws) >= most):
            continue
        rows += [i * case["r"] + s for s, w in enumerate(ws) if w in A]
    return rows


def _copies(case, seed, dev):
    """fp32 [f, r, ld]: honest file gradients b + 0.001 z per file around a shared b, and the
    adversaries' copies (population mean and std over the files for ALIE)."""
    f, r, d = math.comb(case["K"], case["r"]), case["r"], case["d"]
    ld = (d + 31) // 32 * 32 if case["padded"] else d
    gen = torch.Generator(dev).manual_seed(seed)
    b = 0.01 * torch.randn(d, device=dev, generator=gen)
    copies = torch.empty((f, r, ld), dtype=torch.float32, device=dev)
    if ld > d:
        copies[:, :, d:] = 0.0
    per = max(1, 32_000_000 // d)
    s1 = torch.zeros(d, dtype=torch.float64, device=dev)
    s2 = torch.zeros(d, dtype=torch.float64, device=dev)
    for i in range(0, f, per):
        n = min(per, f - i)
        z = torch.randn((n, d), device=dev, generator=gen).mul_(0.001).add_(b)
        copies[i: i + n, :, :d] = z[:, None, :]
        z = z.double()
        s1 += z.sum(0)
        s2 += (z - b).square_().sum(0)
    mean = s1 / f
    std = (s2 / f - (mean - b).square()).clamp_(min=0).sqrt()
    bad = (mean - std if case["distortion"] == "alie" else -mean).float()
    rows = _distorted_rows(case, seed)
    flat = copies.view(f * r, ld)
    if case["kind"] == "tolerant":
        per = max(1, 32_000_000 // d)
        for i in range(0, f * r, per):
            n = min(per, f * r - i)
            flat[i: i + n, :d] += NOISE * torch.randn((n, d), device=dev, generator=gen)
    for row in rows:
        if case["distortion"] == "reversed":
            flat[row, :d] = -10.0 * flat[row, :d]
        else:
            flat[row, :d] = bad
    return copies


def _graph(case, seed):
    """int32 words [K, 4] of the agreement graph that the attack leaves."""
    A, D = _sides(case, seed)
    K = case["K"]
    words = torch.zeros((K, 4), dtype=torch.int64)
    for j in range(K):
        for k in range(K):
            if j == k:
                continue
            if case["attack"] == "weak":
                apart = (j in A) != (k in A)
            else:
                apart = (j in A and k in D) or (k in A and j in D)
            if not apart:
                words[j, k // 32] |= 1 << (k % 32)
    return torch.where(words >= 2 ** 31, words - 2 ** 32, words).to(torch.int32)


def prepare(case, seed):
    dev, kind = _device(), case["kind"]
    if kind == "sgd":
        gen = torch.Generator(dev).manual_seed(seed)
        g, w, v = (torch.randn(case["d"], device=dev, generator=gen) for _ in range(3))
        return {"case": case, "g": 0.01 * g, "w": w, "v": 0.1 * v}
    if kind == "wide":
        return {"case": case, "adj": _graph(case, seed).to(dev),
                "det": ap.wide_detection_buffer(dev, flags=ap.WIDE_ALL_MAXIMAL if case["all"] else 0)}
    a = ap.aspis_assign(case["K"], case["r"])
    s = {"case": case, "a": a, "copies": _copies(case, seed, dev),
         "mode": ap.MEAN if case["mode"] == "mean" else ap.MEDIAN}
    s["buf"] = (ap.TolerantBuffers if kind == "tolerant" else ap.RoundBuffers)(a, case["d"], dev)
    if kind == "host":
        s["host"] = torch.empty(s["copies"].shape, dtype=torch.float32, pin_memory=True)
        s["host"].copy_(s["copies"])
        s["host_out"] = torch.empty(case["d"], dtype=torch.float32, pin_memory=True)
        s["host_det"] = torch.empty(ap.DETECTION_BYTES, dtype=torch.uint8, pin_memory=True)
    return s


# The record's first six words are the outcome (clique, size, count, success, kept files, status);
# the rest are the search's own input and its diagnostics (nodes visited, coordinates that took the
# median's exact path).
OUTCOME = 24


def run(s):
    case = s["case"]
    kind, d = case["kind"], case["d"] if "d" in case else 0
    if kind == "sgd":
        ap.aspis_sgd(s["g"], s["w"], s["v"] if case["mu"] else None, ETA, case["mu"])
        return {"w": s["w"], "v": s["v"]}
    if kind == "wide":
        ap.aspis_detect_wide(s["adj"], case["K"], s["det"])
        # without the flag the number of maximal cliques is a diagnostic too
        n = 32 if case["all"] else 24
        return {"cliques": s["det"][:n], "outcome": s["det"][40:52]}
    a, b, copies = s["a"], s["buf"], s["copies"]
    if kind == "host":
        ap.aspis_round_host(s["host"], copies, d, a, b.file_neq, b.adj, b.det, b.sel, b.out,
                            s["host_out"], s["host_det"], s["mode"])
        return {"out": s["host_out"], "det": s["host_det"][:OUTCOME], "sel": b.sel, "adj": b.adj}
    got = {"out": b.out, "det": b.det[:OUTCOME], "sel": b.sel, "adj": b.adj, "file_neq": b.file_neq}
    if kind == "tolerant":
        ap.aspis_round_tolerant(copies, d, a, TAU, b.file_neq, b.adj, b.det, b.slot_mask, b.sel,
                                b.means, b.out, s["mode"])
        return dict(got, slot_mask=b.slot_mask, means=b.means)
    if kind == "steps":
        ap.aspis_check(copies, d, a, b.file_neq, b.adj)
        ap.aspis_detect(b.adj, case["K"], b.det)
        ap.aspis_select(b.file_neq, b.det, a, b.sel)
        ap.aspis_aggregate(copies, d, a, b.sel, b.det, b.out, s["mode"])
    else:
        ap.aspis_round(copies, d, a, b.file_neq, b.adj, b.det, b.sel, b.out, s["mode"])
    return got


def work(case):
    if case["kind"] == "sgd":
        return {"bytes": case["d"] * (20 if case["mu"] else 12), "flops": case["d"] * (4 if case["mu"] else 2)}
    if case["kind"] == "wide":
        return {"bytes": case["K"] * 16 + 64, "flops": 0}
    f, r, d = math.comb(case["K"], case["r"]), case["r"], case["d"]
    b = f * r * d * 4 + d * 4 + f * 5                 # every copy once, the aggregate, the per-file words
    if case["kind"] == "tolerant":
        b += f * d * 4                                # the averages are an output
    return {"bytes": b, "flops": 0}


def tolerance(case):
    # medians are elements of the input and the update rounds each result once: the same bits
    if case["kind"] == "tolerant":
        return {"rel": 1.2e-7, "max": 5e-7}           # fp32 averages: 2.9e-8 from 64 bits measured
    if case.get("mode") == "mean":
        return {"rel": 1.2e-7, "max": 5e-7}           # compensated sums rounded once: 2.5e-8 measured
    return "exact"


# ------------------------------------------------------------------ 64 bits


def _max_cliques(K, adj):
    best = []

    def grow(R, P, X):
        if not P and not X:
            best.append(R)
            return
        u = max(P | X, key=lambda w: len(P & adj[w]))
        for w in sorted(P - adj[u]):
            grow(R | {w}, P & adj[w], X & adj[w])
            P, X = P - {w}, X | {w}

    grow(frozenset(), frozenset(range(K)), frozenset())
    omega = max(len(c) for c in best)
    return [c for c in best if len(c) == omega]


def _apart(case, copies, d):
    """bool [f, pairs]: the pair of copies differs (or is not close)."""
    f, r = copies.shape[:2]
    pairs = list(itertools.combinations(range(r), 2))
    out = torch.zeros((f, len(pairs)), dtype=torch.bool)
    per = max(1, 64_000_000 // (d * r))
    for i in range(0, f, per):
        x = copies[i: i + per, :, :d]
        for p, (s, t) in enumerate(pairs):
            if case["kind"] == "tolerant":
                far = ~((x[:, s] - x[:, t]).abs() <= TAU)
            else:
                far = x[:, s].view(torch.int32) != x[:, t].view(torch.int32)
            out[i: i + per, p] = far.any(-1).cpu()
    return out.tolist(), pairs


def _slots(case, copies, d):
    """Per file the slots that enter the aggregate (averaged where several)."""
    K, r, files = case["K"], case["r"], _files(case)
    apart, pairs = _apart(case, copies, d)
    adj = [set(range(K)) - {j} for j in range(K)]
    for ws, row in zip(files, apart):
        for (s, t), no in zip(pairs, row):
            if no:
                adj[ws[s]].discard(ws[t])
                adj[ws[t]].discard(ws[s])
    cliques = _max_cliques(K, [frozenset(x) for x in adj])
    chosen = []
    for ws, row in zip(files, apart):
        if len(cliques) == 1:
            keep = [s for s in range(r) if ws[s] in cliques[0]]
        else:
            near = {s: {s} for s in range(r)}
            for (s, t), no in zip(pairs, row):
                if not no:
                    near[s].add(t)
                    near[t].add(s)
            groups = []
            for s in range(r):
                g, more = {s}, True
                while more:
                    h = set().union(*(near[x] for x in g))
                    more, g = h != g, h
                groups.append(sorted(g))
            keep = max(groups, key=lambda g: (len(g), -g[0]))
        chosen.append(keep if case["kind"] == "tolerant" else keep[:1])
    return chosen


def exact(case, seed):
    if case["kind"] == "wide":
        return None
    if case["kind"] == "sgd":
        s = prepare(case, seed)
        g, w, v = s["g"].double(), s["w"].double(), s["v"].double()
        eta, mu = (float(torch.tensor(x)) for x in (ETA, case["mu"]))       # as the fp32 arguments
        v1 = mu * v + g if case["mu"] else v
        return {"w": w - eta * (v1.float().double() if case["mu"] else g), "v": v1}
    dev, d = _device(), case["d"]
    copies = _copies(case, seed, dev)
    f, r, ld = copies.shape
    if f * d > 6e9:
        return None
    chosen = _slots(case, copies, d)
    kept = [i for i, c in enumerate(chosen) if c]
    n = len(kept)
    first = torch.tensor([i * r + chosen[i][0] for i in kept], device=dev)
    flat = copies.view(f * r, ld)
    weight = torch.zeros((n, r), dtype=torch.float64)
    for k, i in enumerate(kept):
        weight[k, chosen[i]] = 1.0 / len(chosen[i])
    weight, rows = weight.to(dev), torch.tensor(kept, device=dev)
    tolerant = case["kind"] == "tolerant"
    out = torch.empty(d, dtype=torch.float64, device=dev)
    means = torch.zeros((f, (d + 3) // 4 * 4), dtype=torch.float64, device=dev) if tolerant else None
    per = max(1, 60_000_000 // (n * (r if tolerant else 1)))
    for c in range(0, d, per):
        e = min(d, c + per)
        if tolerant:
            x = (copies[rows, :, c:e].double() * weight[:, :, None]).sum(1)
            means[rows, c:e] = x
        else:
            x = flat[:, c:e].index_select(0, first).double()
        if case["mode"] == "mean":
            out[c:e] = x.mean(0)
        else:
            out[c:e] = x.sort(0).values[(n - 1) // 2]
    got = {"out": out, "det": None, "sel": None, "adj": None}
    if case["kind"] != "host":
        got["file_neq"] = None
    return dict(got, slot_mask=None, means=means) if tolerant else got
