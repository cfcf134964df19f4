"""The calls that users of this library make, at the sizes they make them: one list of performance cases.

A case is a dict of plain values; ``prepare`` builds its inputs on the GPU (or in pinned host memory, for
the host-buffer call), ``run`` makes one pass through the public entry points of ``binding``.

Shapes: vocabularies from 1000 to 262144 (also ones that leave rows unaligned), batches from 1 to 128,
draft trees with a trunk of ``L1`` nodes and ``K`` branches of ``L2`` nodes, bf16 and fp32 logits,
temperatures from 0.2 to 1.2, top-p from 0.9 to 0.99, top-k of 20 to 200.
"""
from __future__ import annotations

import math

import torch

from paper_2602_16994_b200 import binding, synth

DEFAULTS = dict(call="specinfer", api="plain", B=8, V=128256, dtype="bf16", K=4, L1=2, L2=4, sigma=1.0,
                sigma_per_depth=0.0, temperature=1.0, top_k=0, top_p=1.0, features=False, diagnostics=False)


def _case(name, **kw):
    return dict(DEFAULTS, name=name, **kw)


def listed():
    return [
        # the smallest call: a toy vocabulary, one sequence; launches and host work are all of it
        _case("specinfer_tiny_f32", B=1, V=1000, dtype="f32", K=2, L1=0, L2=3),
        # interactive decoding, one user: latency of one sequence at a full-size vocabulary
        _case("traversal_one_sequence", call="traversal", B=1),
        # the benchmark's batch, both verifiers: a decoding loop that reuses its buffers, so the call is prepared once
        _case("specinfer_b8", api="prepared"),
        _case("traversal_b8", call="traversal", api="prepared"),
        # a wide tree under nucleus sampling, the usual setting of a served model
        _case("specinfer_top_p_b32", B=32, V=151936, K=8, L1=0, L2=5, sigma=0.7, temperature=0.6, top_p=0.95),
        # T = 1 with top-p 0.99: the widest nucleus among the usual settings, hundreds to thousands of tokens
        _case("traversal_wide_nucleus_b8", call="traversal", top_p=0.99),
        # the largest vocabulary, divergence growing with depth
        _case("traversal_v262144_b16", call="traversal", B=16, V=262144, sigma=0.5, sigma_per_depth=0.25),
        # a serving batch at low temperature with top-k and the selector's features
        _case("specinfer_top_k_features_b128", B=128, K=8, L2=6, sigma=1.2, temperature=0.3, top_k=50, features=True),
        # fp32 logits, rows that start on no 16-byte boundary, every threshold and the residual law wanted
        # (evaluation of draft models, training of a selector)
        _case("traversal_diagnostics_f32", call="traversal", B=6, V=50257, dtype="f32", K=3, L1=1, L2=3, temperature=0.8,
              diagnostics=True),
        # distributions of every node written out, and one token drawn from each (sampling without a tree)
        _case("probs_and_draw", call="probs", B=4, temperature=0.8, top_p=0.9),
        # acceptance rates, divergences, branching probabilities and block efficiency of the benchmark's batch
        _case("analysis_b8", call="analysis"),
        # logits in pinned host memory: copies in, verification, decisions back
        _case("host_specinfer_b8", call="host"),
    ]


# most bytes of logits in a drawn case, by call: none costs more than the largest listed case
_CAP = dict(specinfer=3.0e9, traversal=4.0e8, probs=1.5e8, analysis=7.0e7, host=7.5e7)


def draw(rng):
    """One more case: the call, the tree, the batch and the sampling parameters over their whole ranges."""
    c = dict(DEFAULTS)
    c["call"] = rng.choice(["specinfer", "specinfer", "specinfer", "traversal", "traversal", "traversal", "probs", "analysis",
                            "host"])
    c["V"] = int(round(math.exp(rng.uniform(math.log(1000), math.log(262144)))))
    if rng.random() < 0.5:                       # a row length that keeps rows aligned, as model vocabularies mostly do
        c["V"] = max(1024, c["V"] // 64 * 64)
    c["B"] = int(round(math.exp(rng.uniform(0.0, math.log(128)))))
    c["dtype"] = rng.choice(["bf16", "bf16", "f32"])
    c["K"], c["L1"], c["L2"] = rng.randint(1, 8), rng.randint(0, 4), rng.randint(1, 6)
    c["sigma"] = round(rng.uniform(0.5, 1.2), 3)
    c["temperature"] = round(rng.uniform(0.2, 1.2), 3)
    kind = rng.choice(["none", "none", "top_p", "top_k", "both"])
    if kind in ("top_p", "both"):
        c["top_p"] = round(rng.uniform(0.9, 0.99), 3)
    if kind in ("top_k", "both"):
        c["top_k"] = rng.randint(20, 200)
    if c["call"] in ("specinfer", "traversal"):
        c["api"] = rng.choice(["plain", "prepared"])
        c["features"] = rng.random() < 0.2
        c["diagnostics"] = rng.random() < 0.15
    cap = _CAP[c["call"]]
    if c["diagnostics"] or c["top_p"] < 1.0:
        cap = min(cap, 1.0e8)
    while _logit_bytes(c) > cap:
        if c["B"] > 1:
            c["B"] = (c["B"] + 1) // 2
        elif c["K"] > 1:
            c["K"] -= 1
        else:
            c["L2"] = max(1, c["L2"] - 1)
            c["L1"] = max(0, c["L1"] - 1)
    return c


def _workload(case):
    return synth.Workload("perf_case", case["B"], case["V"], case["dtype"], case["K"], case["L1"], case["L2"],
                          case["sigma"], case["sigma_per_depth"], case["temperature"], case["top_k"], case["top_p"])


def _rows(case):
    """(nodes, nodes with children) per sequence."""
    parent, _ = _workload(case).tree
    return len(parent), len({int(p) for p in parent[1:]})


def _logit_bytes(case):
    """Logits that a pass has to read: target rows of all nodes and draft rows of the nodes with children (a
    verification), both rows of the nodes with children (the analysis), one side's rows (distributions)."""
    n, internal = _rows(case)
    rows = {"analysis": 2 * internal, "probs": n}.get(case["call"], n + internal)
    return case["B"] * rows * case["V"] * (4 if case["dtype"] == "f32" else 2)


def work(case):
    B, V = case["B"], case["V"]
    n, _ = _rows(case)
    read = _logit_bytes(case)
    logits = read // (4 if case["dtype"] == "f32" else 2)
    written = B * (4 * 4 + 4 * n)
    if case["call"] == "probs":
        written = B * n * (4 * V + 6 * 4 + 4)
    if case["call"] == "analysis":
        written = 4 * B * (17 * n + 5)
    written += 16 * B * n * case["features"] + 4 * B * (V + n) * case["diagnostics"]
    # per logit: scale, subtract the reference, exponential, add
    return {"bytes": read + written, "flops": 4 * logits}


def tolerance(case):
    # distributions, thresholds, rates and features are fp32 values of fp32 / fp64 sums over 1e3 to 1e5 terms; a token
    # drawn by inverse CDF may be the neighbour where a uniform falls within rounding of a boundary
    return {"rel": 1e-5, "differ": 0.01}


def prepare(case, seed):
    w = _workload(case)
    b = synth.make_batch(w, seed=seed, device="cuda")
    args = (b.target_logits, b.draft_logits, b.parent, b.token, b.u_accept, b.u_bonus)
    sampling = dict(temperature=case["temperature"], top_k=case["top_k"], top_p=case["top_p"])
    extra = dict(residual=case["diagnostics"], node_thr=case["diagnostics"], features=case["features"])
    call = case["call"]
    if call == "host":
        verifier = binding.HostVerifier(w.B, w.N, w.V, b.target_logits.dtype, "cuda", "specinfer")
        host = tuple(t.cpu().pin_memory() for t in args)
        return call, lambda: verifier.run(*host, **sampling)
    if call == "analysis":
        return call, lambda: binding.tree_analysis(*args, **sampling)
    if call == "probs":
        u = b.u_bonus.reshape(-1)

        def probs_and_draw():
            probs, stats = binding.tree_probs(b.target_logits, **sampling)
            return probs, stats, binding.sample_bonus(probs.view(-1, w.V), u)
        return call, probs_and_draw
    if case["api"] == "prepared":
        return call, binding.PreparedVerify(call, *args, **sampling, **extra).launch
    verify = binding.verify_specinfer if call == "specinfer" else binding.verify_traversal
    return call, lambda: verify(*args, **sampling, **extra)


def run(state):
    call, one_pass = state
    out = one_pass()
    if call == "probs" or isinstance(out, dict):
        return out
    return {k: v for k, v in vars(out).items() if isinstance(v, torch.Tensor)}
