"""The calls this library is measured on, through its public entry points.

Every case is one pass of a program a user builds with the package: a batch of integer recursions
(`Graph.eval_int`), the forward pass of a tree network (`Graph.eval_trees`) or its training step
(`Graph.grad_trees`).  Sizes and distributions are those of the workloads this repository generates for
its benchmark and tests, and sizes between and below them.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the inputs, parameters, buffers and the graph that a program holds before the call
    run(state)           one pass; its outputs
    work(case)           bytes and operations the pass cannot do without
    tolerance(case)      how far two correct implementations may be apart
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

import paper_2410_20225_b200 as rdf

CLASSES = 5
FIB_MAX = 18                    # 2-bit labels in a packed path tag: 19 nested calls
TAK_Y, TAK_Z, TAK_MAX = 12, 6, 18
TOPDOWN_BIAS = -0.3             # gate bias of the top-down workload; a node is then expanded with probability ~5/8
TOPDOWN_GROWTH = 1.25           # so a level is about 1.25 times as wide as the one above it


# ------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # A handful of calls: the latency of one evaluation, launches and host path included.
        {"name": "fib_8_calls", "program": "fib", "B": 8, "n_hi": 10},
        # The benchmark's integer workload: 1024 concurrent calls of fib(n), n ~ U{0..18}.
        {"name": "fib_1024_calls", "program": "fib", "B": 1024, "n_hi": 18},
        # The same calls at a batch that fills the device: throughput of tags, tokens and the hash store.
        {"name": "fib_131072_calls", "program": "fib", "B": 131072, "n_hi": 18},
        # Three parameters, arguments that are calls themselves: frame tags and the dense store.
        {"name": "tak_200_calls", "program": "tak", "B": 200},
        # Inference on short random trees in fp32 (the benchmark's small tree workload).
        {"name": "rnn_infer_f32_512", "program": "rnn", "train": False, "bf16": False, "repro": False, "B": 512,
         "leaves": "uniform", "H": 64, "V": 1000},
        # Inference on one small request batch of sentences in bf16: latency of a served model.
        {"name": "rnn_infer_bf16_48", "program": "rnn", "train": False, "bf16": True, "repro": False, "B": 48,
         "leaves": "lognormal", "H": 300, "V": 21000},
        # The headline: a training step over 8192 sentence-sized trees, per-node loss, bf16 contractions.
        {"name": "rnn_train_bf16_8192", "program": "rnn", "train": True, "bf16": True, "repro": False, "B": 8192,
         "leaves": "lognormal", "H": 300, "V": 21000},
        # A training step whose sums have to be the same bits on every run, at an ordinary batch.
        {"name": "rnn_train_bf16_repro_1000", "program": "rnn", "train": True, "bf16": True, "repro": True, "B": 1000,
         "leaves": "lognormal", "H": 256, "V": 21000},
        # The heavier cell: a TreeLSTM training step over the same sentences.
        {"name": "lstm_train_bf16_8192", "program": "lstm", "train": True, "bf16": True, "repro": False, "B": 8192,
         "leaves": "lognormal", "H": 300, "V": 21000},
        # TreeLSTM inference in fp32 at an odd batch and a hidden size that is no multiple of a tile.
        {"name": "lstm_infer_f32_601", "program": "lstm", "train": False, "bf16": False, "repro": False, "B": 601,
         "leaves": "lognormal", "H": 148, "V": 21000},
        # Depth stress, fp32 training: degenerate chains (long dependent sequences) with large perfect trees (wide waves).
        {"name": "deep_train_f32", "program": "deep", "chains": 64, "depth": 4096, "perfect": 16, "height": 16,
         "H": 256, "V": 50000},
        # Generation: trees grown top-down, the values deciding where they stop.
        {"name": "topdown_8192_seeds", "program": "topdown", "B": 8192, "H": 128, "V": 21000, "D": 10},
    ]


# (the library takes hidden sizes that are multiples of 4)
def _between(rng, lo, hi):
    """A size between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["fib", "tak", "rnn", "rnn", "rnn", "lstm", "lstm", "deep", "topdown"])
    if kind == "fib":
        return {"program": "fib", "B": _between(rng, 1, 131072), "n_hi": rng.randint(2, FIB_MAX)}
    if kind == "tak":
        return {"program": "tak", "B": _between(rng, 1, 200)}
    if kind == "deep":
        return {"program": "deep", "chains": _between(rng, 1, 64), "depth": _between(rng, 65, 4096),
                "perfect": _between(rng, 1, 16), "height": rng.randint(2, 16), "H": 4 * rng.randint(8, 64),
                "V": _between(rng, 100, 50000)}
    if kind == "topdown":
        return {"program": "topdown", "B": _between(rng, 1, 8192), "H": 4 * rng.randint(4, 32), "V": _between(rng, 100, 21000),
                "D": rng.randint(2, 10)}
    bf16, train = rng.random() < 0.6, rng.random() < 0.6
    most = 8192 if bf16 or kind == "rnn" else 1024
    return {"program": kind, "train": train, "bf16": bf16, "repro": train and bf16 and rng.random() < 0.25,
            "B": _between(rng, 1, most), "leaves": rng.choice(["uniform", "lognormal"]), "H": 4 * rng.randint(8, 80),
            "V": _between(rng, 100, 21000)}


# ------------------------------------------------------------------------------------------------ inputs
@lru_cache(maxsize=None)
def _fib_calls(n):
    """Invocations of fib(n)."""
    return 1 if n < 2 else 1 + _fib_calls(n - 1) + _fib_calls(n - 2)


@lru_cache(maxsize=None)
def _tak(x, y, z):
    """(value, invocations) of tak(x, y, z)."""
    if y >= x:
        return z, 1
    parts = [_tak(x - 1, y, z), _tak(y - 1, z, x), _tak(z - 1, x, y)]
    value, calls = _tak(*(p[0] for p in parts))
    return value, 1 + calls + sum(p[1] for p in parts)


def _arguments(case, rng):
    """Arguments of the integer calls and the number of invocations they cause."""
    if case["program"] == "fib":
        x = rng.integers(0, case["n_hi"] + 1, size=case["B"], dtype=np.int64)
        calls = np.array([_fib_calls(n) for n in range(case["n_hi"] + 1)])
    else:
        x = rng.integers(0, TAK_MAX + 1, size=case["B"], dtype=np.int64)
        calls = np.array([_tak(n, TAK_Y, TAK_Z)[1] for n in range(TAK_MAX + 1)])
    return x, int(calls[x].sum())


def _leaf_counts(case, rng):
    """Leaves of every tree: short trees, or sentence lengths (median 18, at most 56)."""
    if case["leaves"] == "uniform":
        return rng.integers(2, 33, size=case["B"])
    return np.clip(np.rint(np.exp(rng.normal(math.log(18.0), 0.5, size=case["B"]))), 1, 56).astype(np.int64)


def _random_trees(leaves, rng):
    """Full binary trees by uniform recursive splits, nodes in pre-order, stored one after another."""
    size = 2 * leaves - 1
    root = np.concatenate([[0], np.cumsum(size)[:-1]])
    left = np.full(int(size.sum()), -1, dtype=np.int64)
    right = left.copy()
    node, below = root[leaves > 1], leaves[leaves > 1]
    while node.size:
        k = rng.integers(1, below)
        left[node], right[node] = node + 1, node + 2 * k
        node = np.concatenate([node + 1, node + 2 * k])
        below = np.concatenate([k, below - k])
        node, below = node[below > 1], below[below > 1]
    return root, left, right


def _deep_trees(case):
    """Left-degenerate chains (every cell has a leaf on its right), then perfect trees in heap order."""
    depth, height = case["depth"], case["height"]
    shapes = []
    i = np.arange(depth)
    left = np.full(2 * depth + 1, -1, dtype=np.int64)
    right = left.copy()
    left[2 * i], right[2 * i] = 2 * i + 2, 2 * i + 1
    shapes += [(left, right)] * case["chains"]
    i = np.arange(2 ** height - 1)
    left = np.full(2 ** (height + 1) - 1, -1, dtype=np.int64)
    right = left.copy()
    left[i], right[i] = 2 * i + 1, 2 * i + 2
    shapes += [(left, right)] * case["perfect"]
    root = np.concatenate([[0], np.cumsum([s[0].size for s in shapes])[:-1]])
    cat = [np.concatenate([np.where(s[k] >= 0, s[k] + o, -1) for s, o in zip(shapes, root)]) for k in (0, 1)]
    return root, cat[0], cat[1]


def _tree_tensors(root, left, right, vocab, rng):
    tok = np.where(left < 0, rng.integers(0, vocab, size=left.size), -1)
    label = rng.integers(0, CLASSES, size=left.size)
    arrays = {"tree_root": root, "left": left, "right": right, "tok": tok, "label": label}
    return {k: torch.from_numpy(v.astype(np.int32)).cuda() for k, v in arrays.items()}


def _parameters(case, seed):
    """Embedding rows ~ N(0, 0.1^2), Xavier-uniform weights, zero biases; bf16 models hold bf16-representable values."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    H, V, topdown = case["H"], case["V"], case["program"] == "topdown"

    def xavier(rows, cols, scale=1.0):
        bound = scale * math.sqrt(6.0 / (rows + cols))
        return (torch.rand(rows, cols, device="cuda", generator=gen) * 2 - 1) * bound

    gates = 5 if case["program"] == "lstm" else 1
    p = {"E": torch.randn(V, H, device="cuda", generator=gen) * (1.0 if topdown else 0.1),
         "W": xavier(gates * H, 2 * H, 2.0 if topdown else 1.0), "b": torch.zeros(gates * H, device="cuda"),
         "W_s": xavier(CLASSES, H), "b_s": torch.zeros(CLASSES, device="cuda")}
    if gates == 5:
        p["W_x"], p["b_x"] = xavier(3 * H, H), torch.zeros(3 * H, device="cuda")
    if topdown:
        p["b_s"][0] = TOPDOWN_BIAS
    if case.get("bf16"):
        p = {k: v.bfloat16().float() for k, v in p.items()}
    return p


def prepare(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    program = case["program"]
    if program in ("fib", "tak"):
        x, calls = _arguments(case, rng)
        functions, result = rdf.fib_program() if program == "fib" else rdf.tak_program(TAK_Y, TAK_Z)
        graph = rdf.Graph(functions, result, rdf.TAGS_PATH if program == "fib" else rdf.TAGS_FRAME)
        return {"call": "eval_int", "graph": graph, "x": torch.from_numpy(x).cuda(), "max_invocations": calls,
                "y": torch.empty(case["B"], dtype=torch.int64, device="cuda")}

    if program == "deep":
        trees = _tree_tensors(*_deep_trees(case), case["V"], rng)
    elif program == "topdown":
        single = np.full(case["B"], -1, dtype=np.int64)          # a seed is a tree of one node whose token selects its row
        trees = _tree_tensors(np.arange(case["B"]), single, single, case["V"], rng)
    else:
        trees = _tree_tensors(*_random_trees(_leaf_counts(case, rng), rng), case["V"], rng)
    params = _parameters(case, seed)
    train = case.get("train", program == "deep")
    if program == "topdown":
        functions, result = rdf.topdown_program(case["D"])
    else:
        functions, result = rdf.tree_net_program("lstm" if program == "lstm" else "rnn", with_loss=train)
    state = {"call": "grad_trees" if train else "eval_trees", "graph": rdf.Graph(functions, result, rdf.TAGS_FRAME),
             "trees": trees, "params": params, "compute": rdf.BF16 if case.get("bf16") else rdf.F32,
             "h_root": torch.empty(trees["tree_root"].numel(), case["H"], device="cuda"), "max_invocations": None}
    if program == "topdown":
        # few seeds: every tree may be full (2^(D+1) - 1 expansions and as many child states); many seeds: far above the mean
        full = 4 * 2 ** case["D"]
        state["max_invocations"] = case["B"] * (full if case["B"] < 256 else min(full, 256))
    if train:
        state["repro"] = case.get("repro", False)
        state["loss"] = torch.zeros(1, device="cuda")
        state["grads"] = {k: torch.empty_like(v) for k, v in params.items()}
    return state


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    graph = state["graph"]
    if state["call"] == "eval_int":
        y, _ = graph.eval_int(state["x"], state["max_invocations"], check=False, y=state["y"])
        return y
    if state["call"] == "eval_trees":
        h, _ = graph.eval_trees(state["trees"], state["params"], state["compute"], check=False, h_root=state["h_root"],
                                max_invocations=state["max_invocations"])
        return h
    loss, h, grads = graph.grad_trees(state["trees"], state["params"], state["compute"], check=False, grads=state["grads"],
                                      loss=state["loss"], h_root=state["h_root"], reproducible=state["repro"])
    return {"loss": loss, "h_root": h, **{"d" + k: v for k, v in grads.items()}}


# ------------------------------------------------------------------------------------------------ work and tolerance
def work(case):
    program = case["program"]
    rng = np.random.Generator(np.random.PCG64(0))
    if program in ("fib", "tak"):
        # argument in, result out; a comparison, the argument subtractions and the combining addition of every invocation
        calls = _arguments(case, rng)[1]
        return {"bytes": 16 * case["B"], "flops": (4 if program == "fib" else 3) * calls}
    H, V = case["H"], case["V"]
    if program == "topdown":
        B = case["B"]
        expands = B * sum(TOPDOWN_GROWTH ** d for d in range(case["D"] + 1))
        cells = (expands - B) / 2                                # every pair of expansions below a seed has one parent cell
        flops = expands * 2 * H + (expands - B) * 2 * H * H + cells * 4 * H * H
        return {"bytes": 4 * (B * 2 + min(V, B) * H + 2 * H * H + 2 * H + B * H), "flops": flops}
    if program == "deep":
        B = case["chains"] + case["perfect"]
        leaves = case["chains"] * (case["depth"] + 1) + case["perfect"] * 2 ** case["height"]
    else:
        B = case["B"]
        leaves = int(_leaf_counts(case, rng).sum())
    cells, nodes = leaves - B, 2 * leaves - B
    gates, train = (5 if program == "lstm" else 1), case.get("train", program == "deep")
    flops = cells * gates * 4 * H * H + (leaves * 6 * H * H if gates == 5 else 0)
    weights = gates * (2 * H * H + H) + (3 * (H * H + H) if gates == 5 else 0)
    words = B + 3 * nodes + min(V, leaves) * H + weights + B * H
    if train:                                                    # the loss at every node, two more contractions each, gradients out
        flops = 3 * (flops + nodes * 2 * CLASSES * H)
        head = CLASSES * (H + 1)
        words += nodes + head + (V * H + weights + head) + 1
    return {"bytes": 4 * words, "flops": flops}


def tolerance(case):
    """Measured against the same networks in 64 bits, over the listed cases and drawn ones: bf16 states and operands are off
    by up to 3.6e-3 (root states, bias gradients), fp32 results by up to 1.7e-6 and up to 3.8e-6 with their sums in another
    order (the deep recursion)."""
    if case["program"] in ("fib", "tak"):
        return "exact"
    return {"rel": 1.4e-2 if case.get("bf16") else 1.5e-5}
