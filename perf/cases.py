"""The work whose speed is measured: what programs have this library do, through its public
Python entry points (Graph.sample_and_decode, Graph.decode_batch, Graph.decode_bbp4mf, Multi).

A case is a dict of plain values.  `kind` names the entry point:
  "mc"       Graph.sample_and_decode: one Monte Carlo point of a threshold sweep
  "request"  Graph.decode_batch on host (numpy) buffers: one decoding request of a service
  "batch"    Graph.decode_batch on device-resident syndromes and outputs
  "bbp"      Graph.decode_bbp4mf: B-BP4MF on both Pauli types
  "fused"    Multi.run: several graphs with uneven shot counts in one run
Syndromes are sampled from the case's own noise model (Graph.sample, counter-based), so defect
counts, convergence and ties are those of real use.  Every output is a byte or a whole number
(predicted flips, flags, iteration counts, failure counts).
"""
import math

import numpy as np
import torch

import paper_2603_05381_gb300 as pkg


def _case(kind, model, d, p, shots, iters, **kw):
    c = {"kind": kind, "model": model, "family": "rotated", "d": d, "p": p, "shots": shots, "iters": iters,
         "precision": "fp32", "decoder": "bp4m", "alpha": 1.0, "early_exit": True, "forced": "greedy"}
    c.update(kw)
    return c


def listed():
    cases = [
        # a single syndrome of a small code from the host: the latency a decoding service sees
        # at its lightest, launches and copies only
        _case("request", "circuit", 5, 0.005, 1, 50, name="request_d5_one_shot"),
        # the smallest Monte Carlo point: d = 3 code capacity, 10^4 shots, FP64 messages
        _case("mc", "code_capacity", 3, 0.05, 10000, 50, precision="fp64", name="mc_cc_d3_fp64"),
        # a few shots of a large code from the host: latency of heavy requests (too few shots to
        # fill the device with one block each)
        _case("request", "circuit", 19, 0.005, 7, 50, name="request_d19_few_shots"),
        # a code-capacity sweep point near the threshold, middle distance, T = 2 d: many small
        # factor graphs, sampling and classification beside the decoding
        _case("mc", "code_capacity", 9, 0.10, 1000000, 18, name="mc_cc_d9"),
        # the largest distance of the code-capacity sweep above the threshold: 50 to 90 defects
        _case("mc", "code_capacity", 21, 0.16, 200001, 42, name="mc_cc_d21"),
        # a circuit sweep point below the threshold: most shots have a handful of defects and
        # converge within a few iterations
        _case("mc", "circuit", 7, 0.002, 1000000, 50, name="mc_circuit_d7_low_p"),
        # the benchmark's workload (d = 13, p = 0.005, T = 50): 126 defects a shot on average
        _case("mc", "circuit", 13, 0.005, 300000, 50, name="mc_circuit_d13"),
        # device-resident batch of a larger code: 283 defects a shot, beyond shared memory
        _case("batch", "circuit", 17, 0.005, 3001, 50, name="batch_d17"),
        # the same at 534 defects a shot with 16-bit message storage
        _case("batch", "circuit", 21, 0.005, 801, 50, precision="fp16", name="batch_d21_fp16"),
        # Memory-BP4MF: forced convergence after every iteration, lightest candidate kept
        _case("batch", "circuit", 9, 0.005, 20000, 25, decoder="bp4mf", alpha=0.85, name="batch_d9_memory_bp4mf"),
        # B-BP4MF on the unrotated code: quaternary BP, then BP4MF on reweighted priors
        _case("bbp", "code_capacity", 9, 0.10, 10000, 25, family="unrotated", decoder="bbp4mf", name="bbp4mf_d9"),
        # mixed distances and noise models with uneven shot counts in one fused 16-bit run
        # (d, model and shots of the parts follow from `shots`: _fused_parts)
        _case("fused", "mixed", 17, 0.005, 40000, 50, precision="fp16", name="fused_fp16"),
    ]
    return cases


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges (without a name)."""
    kind = rng.choice(["mc", "mc", "request", "request", "batch", "batch", "bbp", "fused"])
    budget = 4.0e10  # message updates of one pass: well below the largest listed case's
    if kind == "mc":
        if rng.random() < 0.5:
            d = rng.choice([3, 5, 7, 9, 11, 13, 15, 17, 21])
            c = _case(kind, "code_capacity", d, round(rng.uniform(0.05, 0.20), 3), 0, 2 * d)
        else:
            d = rng.choice([3, 5, 7, 9, 11, 13])
            c = _case(kind, "circuit", d, round(rng.uniform(0.001, 0.010), 4), 0, 50)
        if d <= 5 and rng.random() < 0.2:
            c["precision"] = "fp64"
            budget = 2.0e8
        lo, hi = 10000, 1000000
    elif kind == "request":
        d = rng.choice([5, 7, 9, 11, 13, 15, 17, 19])
        c = _case(kind, "circuit", d, 0.005, 0, 50, precision=rng.choice(["fp32", "fp16", "bf16"]))
        lo, hi = 1, 4096
    elif kind == "batch":
        d = rng.choice([5, 7, 9, 11, 13, 15, 17, 19])
        c = _case(kind, "circuit", d, round(rng.uniform(0.002, 0.007), 4), 0, rng.choice([25, 50]),
                  precision=rng.choice(["fp32", "fp32", "fp16", "bf16"]), forced=rng.choice(["greedy", "greedy", "static"]),
                  family=rng.choice(["rotated", "rotated", "unrotated"]))
        if rng.random() < 0.3:
            c.update(decoder="bp4mf", alpha=rng.choice([1.0, 0.85]))
            budget = 4.0e9
        elif rng.random() < 0.25:
            c["early_exit"] = False
        lo, hi = 50, 100000
    elif kind == "bbp":
        d = rng.choice([3, 5, 7, 9, 11, 13])
        c = _case(kind, "code_capacity", d, round(rng.uniform(0.05, 0.15), 3), 0, 25, decoder="bbp4mf",
                  family=rng.choice(["rotated", "unrotated"]))
        budget = 2.0e8
        lo, hi = 100, 10000
    else:
        c = _case(kind, "mixed", rng.choice([13, 17]), 0.005, 0, 50, precision=rng.choice(["fp32", "fp16", "bf16"]))
        lo, hi = 2000, 40000
    c["shots"] = 1
    c["shots"] = max(1, min(_log_int(rng, lo, hi), int(budget / max(1.0, _updates(c)))))
    return c


# ---- the parts of a fused run: (model, d, p, Pauli type, shots)
def _fused_parts(case):
    n = case["shots"]
    parts = [("circuit", 5, 0.005, 0, n), ("code_capacity", 5, 0.10, 1, n // 2 + 1), ("circuit", 9, 0.005, 0, n // 4 + 1),
             ("code_capacity", 13, 0.10, 0, n // 2 + 1), ("circuit", 13, 0.005, 0, n // 8 + 1)]
    if case["d"] >= 17:
        parts += [("circuit", 17, 0.005, 0, n // 50 + 1), ("code_capacity", 17, 0.10, 1, n // 8 + 1)]
    return parts


def _graph(model, d, p, family="rotated"):
    return pkg.Graph(d, model, p, family=family)


def _sample(g, shots, seed):
    """Device syndromes of every Pauli type: one flat int32 tensor and its per-type views."""
    info = g.info()
    synd = torch.empty((shots * sum(info["n_words"]),), dtype=torch.int32, device="cuda")
    obs = torch.empty((info["n_types"], shots), dtype=torch.uint8, device="cuda")
    g.sample(synd, obs, first_shot=0, seed=seed)
    views, off = [], 0
    for nw in info["n_words"]:
        views.append(synd[off:off + shots * nw].view(shots, nw))
        off += shots * nw
    return synd, views


def _opts(case, type=0):
    return pkg.make_opts(precision=case["precision"], early_exit=case["early_exit"], decoder=case["decoder"],
                         alpha=case["alpha"], type=type, forced=case["forced"])


def prepare(case, seed):
    n, kind = case["shots"], case["kind"]
    if kind == "fused":
        parts = _fused_parts(case)
        graphs = [_graph(m, d, p) for (m, d, p, _, _) in parts]
        types = [ty for (_, _, _, ty, _) in parts]
        shots = [k for (_, _, _, _, k) in parts]
        synd = [_sample(g, k, seed + j)[1][ty].cpu().numpy().view(np.uint32)
                for j, (g, ty, k) in enumerate(zip(graphs, types, shots))]
        obs = [np.zeros(k, dtype=np.uint8) for k in shots]
        conv = [np.zeros(k, dtype=np.uint8) for k in shots]
        multi = pkg.Multi(graphs, shots, case["iters"], _opts(case), types=types, max_defects=448)
        multi.run(synd, obs, conv)  # the plan's own first run, on which it tunes itself
        return {"kind": kind, "graphs": graphs, "multi": multi, "synd": synd, "obs": obs, "conv": conv}
    g = _graph(case["model"], case["d"], case["p"], case["family"])
    s = {"kind": kind, "g": g, "shots": n, "iters": case["iters"], "opts": _opts(case), "seed": seed}
    if kind == "mc":
        return s
    flat, views = _sample(g, n, seed)
    if kind == "bbp":
        s["synd"] = flat
        s["obs"] = torch.zeros((2, n), dtype=torch.uint8, device="cuda")
        s["flags"] = torch.zeros((2, n), dtype=torch.uint8, device="cuda")
    elif kind == "batch":
        s["synd"] = views[0]
        s["obs"] = torch.zeros((n,), dtype=torch.uint8, device="cuda")
        s["conv"] = torch.zeros((n,), dtype=torch.uint8, device="cuda")
        s["its"] = torch.zeros((n,), dtype=torch.int16, device="cuda")
    else:
        s["synd"] = views[0].cpu().numpy().view(np.uint32)
        s["obs"] = np.zeros(n, dtype=np.uint8)
        s["conv"] = np.zeros(n, dtype=np.uint8)
        s["its"] = np.zeros(n, dtype=np.int16)
    return s


def run(state):
    s = state
    if s["kind"] == "fused":
        s["multi"].run(s["synd"], s["obs"], s["conv"])
        return {"obs": s["obs"], "converged": s["conv"]}
    if s["kind"] == "mc":
        return s["g"].sample_and_decode(s["shots"], s["seed"], s["iters"], s["opts"])
    if s["kind"] == "bbp":
        s["g"].decode_bbp4mf(s["synd"], s["iters"], s["opts"], s["obs"], s["flags"])
        return {"obs": s["obs"], "flags": s["flags"]}
    s["g"].decode_batch(s["synd"], s["iters"], s["opts"], s["obs"], s["conv"], s["its"])
    return {"obs": s["obs"], "converged": s["conv"], "iters": s["its"]}


def exact(case, seed):
    """No output is a computed real number: every one is a byte or a count."""
    return None


# ---- work of one pass

_info = {}


def _graph_info(model, d, p, family):
    key = (model, d, p, family)
    if key not in _info:
        g = _graph(model, d, p, family)
        _info[key] = g.info()
        g.close()
    return _info[key]


def _part_updates(model, d, p, family, iters, all_iters):
    """Expected message updates of one shot and type: s^2 per iteration.  A shot that converges
    does so within about four iterations; the fraction that never does was fitted to this
    library's sweep tables (1 - exp(-kappa p s))."""
    info = _graph_info(model, d, p, family)
    m = sum(info["mean_defects"]) / info["n_types"]
    never = 1.0 - math.exp(-(5.3 if model == "circuit" else 0.5) * p * m)
    its = iters if all_iters else never * iters + (1.0 - never) * min(4, iters)
    return (m * m + m) * its, info


def _updates(case):
    if case["kind"] == "fused":
        return sum(k * _part_updates(m, d, p, "rotated", case["iters"], False)[0] for (m, d, p, _, k) in _fused_parts(case))
    all_iters = case["decoder"] == "bp4mf" or not case["early_exit"]
    u, info = _part_updates(case["model"], case["d"], case["p"], case["family"], case["iters"], all_iters)
    types = info["n_types"] if case["kind"] in ("mc", "bbp") else 1
    return case["shots"] * u * types


def work(case):
    """Bytes: the syndromes read once and the outputs written once (a Monte Carlo point makes its
    syndromes itself and returns counts only).  Flops: one exponential, one logarithm and ten
    additions, maxima and multiplications per message update; ten rounds of Philox (about 60
    operations) per four sampler draws."""
    flops = 12.0 * _updates(case)
    if case["kind"] == "fused":
        byts = sum(k * (4 * _graph_info(m, d, p, "rotated")["n_words"][ty] + 2) for (m, d, p, ty, k) in _fused_parts(case))
        return {"bytes": float(byts), "flops": flops}
    info = _graph_info(case["model"], case["d"], case["p"], case["family"])
    n = case["shots"]
    if case["kind"] == "mc":
        return {"bytes": 200.0, "flops": flops + 15.0 * n * info["n_units"]}
    if case["kind"] == "bbp":
        return {"bytes": float(n * (4 * sum(info["n_words"]) + 4)), "flops": flops}
    return {"bytes": float(n * (4 * info["n_words"][0] + 4)), "flops": flops}
