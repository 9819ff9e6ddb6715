"""Workloads of the verify / commit entry points, for timing them over the range they are used in.

A case is a dict of plain values:

    kind      which calls one pass makes
                verify    gdn_tree_verify
                separate  gdn_tree_verify, then gdn_tree_commit of the accepted path of the same trees
                step      gdn_tree_commit_verify: the previous step's accepted path, then the new trees
                padded    gdn_tree_commit_verify_padded: the same step in the dense layout, trees shared by layer slots
                planned   gdn_tree_plan once, then per layer gdn_tree_commit_padded + gdn_tree_verify_planned
    slots     (sequence, layer) pairs; for `planned` the layers, each a call of its own with `trees` sequences
    trees     different trees among them; slot s carries tree s % trees
    lo, hi    nodes of a tree (drawn uniformly from lo..hi by `sizes`, the seed of the sizes)
    shape     how a tree grows: geo (breadth-first, geometric child counts), bestfirst (deep, narrow), chain
    accepted  nodes of the accepted path (cut to the depth of the tree; -1: uniform over 0..16, per tree)
    h_qk, h_v, d, in_dtype, out_dtype, raw_gates

Sizes are those of the benchmark configurations of ``synth`` (16 / 32 heads of 128 components, 48 layer slots, trees of
8 to 512 nodes, root paths of at most 16 nodes) and of the tests (fp32 inputs, smaller heads).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_06763_b200 as gdn
from paper_2607_06763_b200 import synth

_CODES = {"f32": 0, "bf16": 1}
_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(name, kind, slots, trees, lo, hi, shape="geo", accepted=7, h_qk=16, h_v=32, d=128, in_dtype="bf16",
          out_dtype="bf16", raw_gates=False, sizes=1):
    c = dict(kind=kind, slots=slots, trees=trees, lo=lo, hi=hi, shape=shape, accepted=accepted, h_qk=h_qk, h_v=h_v, d=d,
             in_dtype=in_dtype, out_dtype=out_dtype, raw_gates=raw_gates, sizes=sizes)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a smoke-size model in fp32: the cost of a call itself, on the general path
        _case("tiny_f32_T8", "separate", 1, 1, 8, 8, accepted=3, h_qk=2, h_v=4, d=32, in_dtype="f32", out_dtype="f32"),
        # one layer of a decode step at batch 1: the first step behind a prefill (nothing to commit yet)
        _case("layer_T64_verify", "verify", 1, 1, 64, 64),
        # one layer of a later step: commit and verification in one call
        _case("layer_T64_step", "step", 1, 1, 64, 64),
        # the largest tree budget of the tree-size sweep, one layer
        _case("layer_T512_verify", "verify", 1, 1, 512, 512),
        # a decode step layer by layer in the dense layout: the tree's plan once, two calls for each of 48 layers
        _case("layers48_T121_planned", "planned", 48, 1, 121, 121, raw_gates=True),
        # a decode step over all the heads of a 48-layer stack at once (the headline workload)
        _case("stack48_T64_step", "step", 48, 1, 64, 64),
        # the same in the dense layout, with the deep trees of a best-first builder, an odd node count and raw gates
        _case("stack48_T61_padded", "padded", 48, 1, 61, 61, shape="bestfirst", accepted=12, raw_gates=True),
        # the same as two calls: verification, then the commit once the acceptance is known
        _case("stack48_T64_separate", "separate", 48, 1, 64, 64),
        # the stack with a large tree (the most work of the list)
        _case("stack48_T256_step", "step", 48, 1, 256, 256, accepted=5),
        # a serving batch: 32 sequences with trees of all sizes
        _case("ragged32_step", "step", 32, 32, 16, 256, accepted=4, sizes=3),
        # linear drafts at a large batch, anything from none to all of a draft accepted
        _case("chains64x16_step", "step", 64, 64, 16, 16, shape="chain", accepted=-1),
        # an accuracy run in fp32 on a small batch (general path)
        _case("batch8_f32", "separate", 8, 8, 9, 64, accepted=5, in_dtype="f32", out_dtype="f32", sizes=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above (at most the bytes of the largest listed one; fp32 at most ``batch8_f32``)."""
    while True:
        kind = rng.choice(["verify", "step", "step", "padded", "separate", "planned", "general"])
        shape = rng.choice(["geo", "geo", "bestfirst", "chain"])
        hi = _log(rng, 1, 512)
        if kind == "padded":
            hi = _log(rng, 8, 64)
        if shape == "chain":
            hi = min(hi, 16)
        lo = rng.choice([hi, max(1, hi // 8)])
        slots = _log(rng, 1, 64)
        trees = slots if lo < hi or rng.random() < 0.3 else 1
        accepted = rng.choice([-1, 0, 1, 3, 5, 7, 10, 16])
        out_dtype = rng.choice(["bf16", "bf16", "f32"])
        h_qk, h_v = rng.choice([(16, 32), (16, 32), (8, 16), (2, 4), (16, 48)])
        c = _case(None, kind, slots, trees, lo, hi, shape=shape, accepted=accepted, h_qk=h_qk, h_v=h_v,
                  out_dtype=out_dtype, sizes=rng.randrange(1 << 20))
        if kind in ("padded", "planned"):
            c["raw_gates"] = rng.random() < 0.5
            c["trees"] = rng.choice([n for n in (1, 2, 3, 4) if kind == "planned" or slots % n == 0])
        if kind == "general":
            c.update(kind=rng.choice(["separate", "step", "verify"]), d=rng.choice([32, 64, 128]))
            c["in_dtype"] = rng.choice(["f32", "f32", "bf16"]) if c["d"] < 128 else "f32"
            c["slots"] = _log(rng, 1, 8)
            c["trees"] = c["slots"]
            c["hi"] = min(c["hi"], 64)
            c["lo"] = min(c["lo"], c["hi"])
            c["out_dtype"] = rng.choice(["f32", "bf16"])
            if c["d"] * c["h_v"] > 32 * 128:
                continue
        big = listed()[8]
        if work(c)["bytes"] <= work(big)["bytes"]:
            return c


# ------------------------------------------------------------------------------------------------ sizes and work
def _tree_sizes(c):
    return np.random.Generator(np.random.PCG64(c["sizes"])).integers(c["lo"], c["hi"] + 1, size=c["trees"])


def _nodes(c):
    """Nodes over all slots."""
    n = _tree_sizes(c)
    if c["kind"] == "planned":
        return c["slots"] * int(n.sum())
    return int(sum(n[s % c["trees"]] for s in range(c["slots"])))


def work(case):
    """State read once (and written once where a path is committed), every node's q, k, v, gates and output once; two
    products with the state per node (S k, S q), two per node of an accepted path."""
    c = case
    isz, osz = (4 if c["in_dtype"] == "f32" else 2), (4 if c["out_dtype"] == "f32" else 2)
    n, d = _nodes(c), c["d"]
    slots = c["slots"] * (c["trees"] if c["kind"] == "planned" else 1)
    state = slots * c["h_v"] * d * d * 4
    commits = c["kind"] != "verify" and c["accepted"] != 0
    acc = 0 if not commits else slots * (8 if c["accepted"] < 0 else c["accepted"])
    nodes = n * (2 * c["h_qk"] * d * isz + c["h_v"] * (d * (isz + osz) + 2 * isz))
    path = acc * (c["h_qk"] + c["h_v"]) * d * isz if c["kind"] != "separate" else 0
    return {"bytes": state * (2 if commits else 1) + nodes + path, "flops": 4 * d * d * c["h_v"] * (n + acc)}


def tolerance(case):
    """About four times what the path differs by from itself in 64 bits: a bf16 output by its own rounding (1.7e-3 in the
    norm, 2^-8 of a value at most), an fp32 output of the tensor-core path (bf16 inputs, 128 components) by the bf16
    pairs that carry the state and the solve (4.2e-6, 4e-5), fp32 sums otherwise (1e-7, 9e-7; more on deep trees)."""
    if case["out_dtype"] == "bf16":
        return {"rel": 6e-3, "max": 1.6e-2}
    if case["in_dtype"] == "bf16" and case["d"] == 128:
        return {"rel": 2e-5, "max": 2e-4}
    return {"rel": 1e-6, "max": 1e-5}


# ------------------------------------------------------------------------------------------------ inputs
def _one_tree(rng, c, n):
    if c["shape"] == "chain":
        return synth.tree_chain(n)
    if c["shape"] == "bestfirst" and n > 1:
        return synth.tree_bestfirst(rng, n, concentration=0.1)
    return synth.tree_geo(rng, n)


def _trees_and_paths(rng, c):
    trees = [_one_tree(rng, c, int(n)) for n in _tree_sizes(c)]
    want = rng.integers(0, 17, size=len(trees)) if c["accepted"] < 0 else [c["accepted"]] * len(trees)
    return trees, [synth.longest_path(t)[: int(a)] for t, a in zip(trees, want)]


def _tensors(gen, c, n):
    """q, k, v, g, beta of n nodes: unit q and k, v ~ N(0,1), decays and strengths of N(0,1) gate inputs."""
    dt, dev = _TORCH[c["in_dtype"]], "cuda"

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    q, k = (torch.nn.functional.normalize(normal(n, c["h_qk"], c["d"]), dim=-1).to(dt) for _ in range(2))
    v, a, b = normal(n, c["h_v"], c["d"]).to(dt), normal(n, c["h_v"]), normal(n, c["h_v"])
    if not c["raw_gates"]:
        a, b = -torch.nn.functional.softplus(a), torch.sigmoid(b)
    return [q, k, v, a.to(dt), b.to(dt)]


def _i32(x):
    a = np.ascontiguousarray(x, dtype=np.int32)
    return torch.from_numpy(a if a.size else np.zeros(1, np.int32)).cuda()


def _offsets(sizes):
    return np.concatenate([[0], np.cumsum(sizes)])


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    prev_trees, prev_paths = _trees_and_paths(rng, c)
    trees, paths = _trees_and_paths(rng, c)
    s = {"case": c, "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    dense = c["kind"] in ("padded", "planned")
    n_seq = c["trees"] if c["kind"] == "planned" else c["slots"]
    layers = c["slots"] if c["kind"] == "planned" else 1
    t_pad = max(1, c["hi"])
    if dense:
        total = n_seq * t_pad
    else:
        slot_trees = [trees[i % c["trees"]] for i in range(n_seq)]
        total = sum(len(t) for t in slot_trees)
    s["shape"] = gdn.GdnShape(n_seq, c["h_qk"], c["h_v"], c["d"], c["d"], _CODES[c["in_dtype"]], _CODES[c["out_dtype"]],
                              16, total, t_pad, 1.0 / math.sqrt(c["d"]))
    # the layers' states, inputs and outputs each in one tensor, as a model keeps them; a layer's call gets its slice
    S = 0.1 * torch.randn((layers, n_seq, c["h_v"], c["d"], c["d"]), generator=gen, device="cuda")
    o = torch.zeros((layers, total, c["h_v"], c["d"]), dtype=_TORCH[c["out_dtype"]], device="cuda")
    new, prev = _tensors(gen, c, layers * total), _tensors(gen, c, layers * total)
    s["S"], s["o"] = S, o
    s["layers"] = [{"S": S[i], "o": o[i], "new": [x[i * total:(i + 1) * total] for x in new],
                    "prev": [x[i * total:(i + 1) * total] for x in prev]} for i in range(layers)]
    if dense:
        for key, ts, ps in (("tree", trees, paths), ("prev_tree", prev_trees, prev_paths)):
            parent, path = np.full((len(ts), t_pad), -1, np.int32), np.zeros((len(ts), 16), np.int32)
            for i, (t, p) in enumerate(zip(ts, ps)):
                parent[i, : len(t)] = t
                path[i, : len(p)] = p
            s[key] = [_i32(parent), _i32([len(t) for t in ts]), _i32(path), _i32([len(p) for p in ps])]
        if c["kind"] == "planned":
            s["plan"] = torch.zeros(gdn.gdn_tree_plan_bytes(s["shape"], c["trees"]), dtype=torch.uint8, device="cuda")
        return s
    for key, ts, ps in (("tree", trees, paths), ("prev_tree", prev_trees, prev_paths)):
        ts, ps = [ts[i % c["trees"]] for i in range(n_seq)], [ps[i % c["trees"]] for i in range(n_seq)]
        s[key] = [_i32(np.concatenate(ts)), _i32(_offsets([len(t) for t in ts])), _i32(np.concatenate(ps)),
                  _i32(_offsets([len(p) for p in ps]))]
    s["ws_bytes"] = gdn.gdn_tree_workspace_bytes(s["shape"])
    s["ws"] = torch.zeros(max(256, s["ws_bytes"]), dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ one pass
def _check(rc):
    if rc != 0:
        raise RuntimeError(gdn.gdn_status_string(rc))


def run(state):
    s, c = state, state["case"]
    shape, status = s["shape"], s["status"]
    stream = torch.cuda.current_stream()
    first = s["layers"][0]
    q, k, v, g, beta = first["new"]
    _, kp, vp, gp, bp = first["prev"]
    parent, offsets, path, path_offsets = s["tree"]
    pparent, poffsets, ppath, ppath_offsets = s["prev_tree"]
    S, o = first["S"], first["o"]
    if c["kind"] in ("verify", "separate"):
        _check(gdn.gdn_tree_verify(shape, S, q, k, v, g, beta, parent, offsets, o, s["ws"], s["ws_bytes"], status, stream))
        if c["kind"] == "verify":
            return {"o": s["o"]}
        _check(gdn.gdn_tree_commit(shape, S, k, v, g, beta, parent, offsets, path, path_offsets, status, stream))
        return {"o": s["o"], "S": s["S"]}
    if c["kind"] == "step":
        _check(gdn.gdn_tree_commit_verify(shape, S, kp, vp, gp, bp, pparent, poffsets, ppath, ppath_offsets, q, k, v, g,
                                          beta, parent, offsets, o, s["ws"], s["ws_bytes"], status, stream))
        return {"o": s["o"], "S": s["S"]}
    raw, n_trees = c["raw_gates"], c["trees"]
    if c["kind"] == "padded":
        _check(gdn.gdn_tree_commit_verify_padded(shape, n_trees, raw, S, shape.max_tree_nodes, kp, vp, gp, bp, pparent,
                                                 poffsets, ppath, ppath_offsets, q, k, v, g, beta, parent, offsets, o,
                                                 status, stream))
        return {"o": s["o"], "S": s["S"]}
    _check(gdn.gdn_tree_plan(shape, n_trees, parent, offsets, s["plan"], status, stream))
    for layer in s["layers"]:
        _, kp, vp, gp, bp = layer["prev"]
        q, k, v, g, beta = layer["new"]
        _check(gdn.gdn_tree_commit_padded(shape, n_trees, raw, layer["S"], kp, vp, gp, bp, pparent, poffsets, ppath,
                                          ppath_offsets, status, stream))
        _check(gdn.gdn_tree_verify_planned(shape, n_trees, raw, layer["S"], q, k, v, g, beta, s["plan"], layer["o"],
                                           status, stream))
    return {"o": s["o"], "S": s["S"]}
