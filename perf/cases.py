"""The work users of this library have it do, as measurable cases.

A case is one call pattern on one batch of trees:

  call   "serve"    forest in pinned host memory in, root states in pinned host memory out (forward_host)
         "forward"  device-resident forest, states of every node and the schedule out (forward)
         "train"    forward that keeps its activations, then loss and every gradient (backward)
  cell   "treelstm", "treernn" or "rntn", the three models of the paper's evaluation
  dtype  "bf16" or "fp32": precision of the gate contraction (TreeRNN and RNTN are fp32)
  shape  "moderate" (uniform random splits), "linear" (left chains), "balanced" (a power of two leaves)
  ids    "postorder" as a parser numbers its nodes, or "shuffled" (the library asks for no order)

Sizes are those of the repository's own workloads: H = 256 and 150 with E = 300 and a vocabulary of 20000
for TreeLSTM, H = 128 for TreeRNN, H = 32 for RNTN, sentences of 2 to 56 words, chains of 64 and balanced
trees of 1024 leaves, batches from one tree to a thousand, five classes.
"""
import math

import numpy as np
import torch

from paper_1809_00832_b200 import binding
from paper_1809_00832_b200 import forests

VOCAB = 20000
CLASSES = 5


def _case(call, cell, dtype, H, E, trees, lo, hi, shape="moderate", ids="postorder"):
    return dict(call=call, cell=cell, dtype=dtype, H=H, E=E, trees=trees, min_leaves=lo, max_leaves=hi, shape=shape, ids=ids)


def listed():
    cases = {
        # one sentence at a time, as an interactive service has it: latency and launches are everything
        "serve_1_tree_bf16": _case("serve", "treelstm", "bf16", 256, 300, 1, 30, 30),
        # a service that batches its requests, at the benchmark's batch; the copies are part of the call
        "serve_256_trees_bf16": _case("serve", "treelstm", "bf16", 256, 300, 256, 2, 56),
        # the paper's largest batch on the smaller model (no size a multiple of a tile), nodes in no order
        "forward_25_trees_bf16": _case("forward", "treelstm", "bf16", 150, 300, 25, 2, 56, ids="shuffled"),
        # the benchmark's own workload
        "forward_256_trees_bf16": _case("forward", "treelstm", "bf16", 256, 300, 256, 2, 56),
        # bulk evaluation of a corpus: the largest batches a user submits in one call
        "forward_1000_trees_bf16": _case("forward", "treelstm", "bf16", 256, 300, 1000, 2, 56),
        # deepest usual forest: every wavefront 64 nodes wide
        "forward_chains64_bf16": _case("forward", "treelstm", "bf16", 256, 300, 64, 64, 64, "linear"),
        # shallowest usual forest: wide wavefronts
        "forward_balanced1024_bf16": _case("forward", "treelstm", "bf16", 256, 300, 16, 1024, 1024, "balanced"),
        # full-precision evaluation at the paper's largest batch
        "forward_25_trees_fp32": _case("forward", "treelstm", "fp32", 150, 300, 25, 2, 56),
        # the paper's training step
        "train_25_trees_fp32": _case("train", "treelstm", "fp32", 150, 300, 25, 2, 56),
        # a training step at a batch that fills the GPU, bf16 forward
        "train_256_trees_bf16": _case("train", "treelstm", "bf16", 256, 300, 256, 2, 56),
        # training steps of the paper's other two models
        "train_25_trees_treernn": _case("train", "treernn", "fp32", 128, 128, 25, 2, 56),
        "train_25_trees_rntn": _case("train", "rntn", "fp32", 32, 32, 25, 2, 56),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    cell = rng.choice(["treelstm"] * 4 + ["treernn", "rntn"])
    if cell == "treelstm":
        call = rng.choice(["serve", "forward", "forward", "train"])
        dtype = rng.choice(["bf16", "bf16", "fp32"])
        H, E = rng.randint(100, 256), rng.randint(100, 300)
        trees = _log_int(rng, 1, 1000 if dtype == "bf16" and call != "train" else 256)
    else:
        call, dtype = rng.choice(["forward", "train"]), "fp32"
        H = rng.randint(64, 128) if cell == "treernn" else rng.randint(16, 32)
        E, trees = H, _log_int(rng, 1, 100 if cell == "treernn" else 25)
    shape = rng.choice(["moderate", "moderate", "linear", "balanced"])
    if shape == "moderate":
        lo = rng.randint(1, 24)
        hi = rng.randint(lo + 1, 56)
    elif shape == "linear":
        lo = rng.randint(2, 16)
        hi = rng.randint(lo, 64 if cell == "treelstm" else 16)
    else:
        lo = hi = 2 ** rng.randint(3, 10 if cell == "treelstm" else 6)
    case = _case(call, cell, dtype, H, E, trees, lo, hi, shape, rng.choice(["postorder", "postorder", "shuffled"]))
    # no more nodes than the largest listed case of its kind has
    most = 29000 if cell == "treelstm" and dtype == "bf16" and call != "train" else 7500 if cell == "treelstm" else 2900
    case["trees"] = max(1, min(case["trees"], int(most / _leaves_per_tree(case))))
    return case


def _leaves_per_tree(case):
    return (case["min_leaves"] + case["max_leaves"]) / 2


def _lengths(case):
    """Sentence lengths spread evenly over the case's range: every forest of a case has the same number of nodes."""
    span = case["max_leaves"] - case["min_leaves"] + 1
    return [case["min_leaves"] + (2 * i + 1) * span // (2 * case["trees"]) for i in range(case["trees"])]


def _forest(case, rng):
    shape_of = {"moderate": lambda n: forests.random_split_shape(rng, n), "linear": forests.left_chain_shape,
                "balanced": forests.balanced_shape}[case["shape"]]
    lengths = rng.permutation(_lengths(case))
    f = forests.forest_from_shapes([shape_of(int(n)) for n in lengths], rng, VOCAB)
    # words come with the frequencies of a natural language (Zipf): the logarithm of a word's rank is uniform.  The ranks
    # are those of the case and their places and ids those of the seed, so that as many different words occur every time.
    leaf = f.left < 0
    rank = np.exp(np.random.default_rng(0).uniform(0.0, math.log(VOCAB + 1), size=int(leaf.sum())))
    word = np.minimum(rank.astype(np.int32) - 1, VOCAB - 1)
    f.token[leaf] = rng.permutation(VOCAB).astype(np.int32)[rng.permutation(word)]
    if case["ids"] == "shuffled":
        f, _ = forests.permute_node_ids(f, rng)
    return f


def _model(case, gen):
    """The parameters a trained or freshly initialised model has, in the distributions of the repository's workloads."""
    H, E = case["H"], case["E"]

    def uniform(shape, scale):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(-scale, scale, generator=gen)

    if case["cell"] == "treelstm":
        emb = torch.empty((VOCAB, E), dtype=torch.float32, device="cuda").normal_(0.0, 0.1, generator=gen)
        precision = binding.BF16 if case["dtype"] == "bf16" else binding.FP32
        model = binding.TreeLSTM(H, E, VOCAB, emb, uniform((E + 2 * H, 5 * H), 0.05), uniform((5 * H,), 0.05), precision)
    else:
        tensor = case["cell"] == "rntn"
        scale = 1.0 / math.sqrt(2 * H)
        model = binding.TreeLSTM.recursive(binding.CELL_RNTN if tensor else binding.CELL_TREERNN, H, VOCAB, uniform((VOCAB, H), 0.5),
                                           uniform((2 * H, H), scale), uniform((H,), scale),
                                           uniform((H, 2 * H, 2 * H), 1.0 / (2 * H)) if tensor else None)
    if case["call"] == "train":
        model.set_classifier(uniform((H, CLASSES), 0.05), uniform((CLASSES,), 0.05))
    return model


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = _forest(case, rng)
    n, H = f.n_nodes, case["H"]
    state = dict(call=case["call"], cell=case["cell"], model=_model(case, gen), trees=case["trees"])
    if case["call"] == "serve":
        # a service keeps its pinned buffers; the roots' ids, h and c share one, as forward_host lays them out
        m = case["trees"]
        pack = torch.empty(4 * m * (1 + 2 * H), dtype=torch.uint8, pin_memory=True)
        state["forest"] = binding.pack_forest_host(f.left, f.right, f.token)
        state["out"] = dict(n_levels=torch.zeros(1, dtype=torch.int32, pin_memory=True),
                            n_roots=torch.zeros(1, dtype=torch.int32, pin_memory=True),
                            root_ids=pack[:4 * m].view(torch.int32),
                            root_h=pack[4 * m:4 * m * (1 + H)].view(torch.float32).view(m, H),
                            root_c=pack[4 * m * (1 + H):].view(torch.float32).view(m, H))
        return state
    state["forest"] = tuple(torch.from_numpy(a).cuda() for a in (f.left, f.right, f.token))
    whole = dict(dtype=torch.int32, device="cuda")
    state["out"] = dict(h=torch.empty((n, H), dtype=torch.float32, device="cuda"),
                        c=torch.empty((n, H), dtype=torch.float32, device="cuda") if case["cell"] == "treelstm" else None,
                        level=torch.empty(n, **whole), order=torch.empty(n, **whole),
                        level_offset=torch.empty(n + 2, **whole), n_levels=torch.zeros(1, **whole))
    if case["call"] == "train":
        state["labels"] = torch.from_numpy(rng.integers(0, CLASSES, size=n, dtype=np.int32)).cuda()
        state["leaves"] = f.n_leaves
        state["words"] = int(np.unique(f.token[f.left < 0]).size)   # rows of the embedding gradient past these are unspecified
    return state


def run(state):
    model = state["model"]
    if state["call"] == "serve":
        return dict(model.forward_host(*state["forest"], max_roots=state["trees"], out=state["out"]))
    # calls follow one another on the stream; the status is read where the program next waits for the device
    flags = binding.PERSISTENT | (binding.SAVE_FOR_BACKWARD if state["call"] == "train" else 0)
    out = model.forward(*state["forest"], flags=flags, out=state["out"], check=False)
    result = {k: out[k] for k in ("h", "c", "level", "order", "n_levels")}   # level_offset is unspecified past n_levels
    if state["call"] == "train":
        backward = model.backward if state["cell"] == "treelstm" else model.backward_recursive
        grads = dict(backward(state["labels"], state["leaves"]))
        for k in ("touched_ids", "dEmb_rows"):
            grads[k] = grads[k][:state["words"]]
        result.update(grads)
    return result


def work(case):
    """Inputs once (forest, embedding rows of the leaves, weights in the precision of the contraction) and outputs once;
    the forest the case draws on average; the multiply-adds of the cells, twice more of them in a training step."""
    H, E, T = case["H"], case["E"], case["trees"]
    leaves = T * _leaves_per_tree(case)
    internal = leaves - T
    n = leaves + internal
    wide = 2 if case["dtype"] == "bf16" else 4
    if case["cell"] == "treelstm":
        weights = 3 * H * E + 10 * H * H
        flops = 2 * leaves * E * 3 * H + 2 * internal * 2 * H * 5 * H
        states = 8 * H
    else:
        weights = 2 * H * H + (4 * H ** 3 if case["cell"] == "rntn" else 0)
        flops = 2 * internal * weights
        states = 4 * H
    nbytes = 12 * n + leaves * 4 * E + weights * wide
    nbytes += T * (states + 4) if case["call"] == "serve" else n * (states + 8)
    if case["call"] == "train":
        all_weights = (E + 2 * H) * 5 * H if case["cell"] == "treelstm" else weights
        nbytes += 4 * n + 4 * all_weights + 4 * H * CLASSES * 2 + leaves * 4 * E
        flops = 3 * flops + 3 * 2 * n * H * CLASSES
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """bf16 operands and hardware tanh against another order of the sums: states that round to the neighbouring bf16 value.
    fp32: the order of 32-bit sums, over up to 64 cells in a row.  The schedule is whole numbers and stays the same."""
    if case["dtype"] == "bf16":
        return {"rel": 5e-3, "max": 5e-2, "differ": 0.0}
    return {"rel": 1e-5, "max": 4e-4, "differ": 0.0}
