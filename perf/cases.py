"""What a user of this framework has it do, as measured cases: training epochs and forward-only passes of the model
families the library builds (multi-layer perceptron, list RNN, binary tree RNN, Tree-LSTM, gated graph network), from one
small request to data sets of the benchmark's shape, through the package's Engine.

A pass is one call as a user's loop makes it: one asynchronous training epoch (parameters move on from pass to pass), one
evaluation of a loaded split, or one request (load a handful of new instances, evaluate them).  Data are synthetic, with the
shapes of the repository's own workloads: dense rows U[0,1], digit lists with an operator token, random binary trees with
Zipf leaf tokens, molecule-like typed graphs.
"""
import math

import numpy as np
import torch

import paper_1705_09786_b200 as amp

LINEAR, LOOKUP, GRUCELL = 1, 2, 3           # parameterised node types of the IR tables
ACT_TANH = 2
KIND_DENSE, KIND_LISTS, KIND_TREES, KIND_GRAPHS = range(4)
TREE_FAMILIES = ("tree", "tree_lstm")
DEFAULTS = {"family": "", "pass": "train", "n": 0, "mak": 1, "muf": 1, "lr": 0.01, "dim": 0, "emb": 0, "hidden": 0,
            "classes": 5, "vocab": 0, "min_size": 1, "max_size": 1, "steps": 4, "bf16": False, "optimizer": "sgd"}


def _case(name, **kw):
    return dict(DEFAULTS, name=name, **kw)


def listed():
    # The learning rates are those of a run that has settled: sums over a tree's or a graph's nodes make large gradients, and a
    # run that diverges has no result to compare.
    return [
        # training a small dense classifier, four instances in flight: the smallest model of the benchmark set
        _case("mlp_train", family="mlp", n=2048, mak=4, muf=32, lr=0.005, dim=784, hidden=256, classes=10),
        # training the list-reduction RNN: variable-length sequences, a loop per token
        _case("rnn_train", family="rnn", n=20000, mak=16, muf=50, lr=0.01, hidden=128, classes=10, vocab=14, max_size=10),
        # training the tree RNN over the whole sentiment-treebank-sized set, a loss at every tree node
        _case("tree_train", family="tree", n=8544, mak=64, muf=100, lr=0.002, emb=300, hidden=150, vocab=20000, min_size=2, max_size=50),
        # training the graph network over a prefix of the molecule set: matrix messages, four propagation steps, regression
        _case("ggnn_train", family="ggnn", n=8000, mak=128, muf=200, lr=0.000002, hidden=100, vocab=15, min_size=9, max_size=29),
        # training the Tree-LSTM sentiment model (leaf and branch cells) on the same kind of trees
        _case("tree_lstm_train", family="tree_lstm", n=2000, mak=64, muf=100, lr=0.005, emb=300, hidden=150, vocab=20000, min_size=2, max_size=50),
        # the throughput configuration: wide cells, large trees, bfloat16 messages
        _case("tree_wide_bf16_train", family="tree", n=400, mak=64, muf=64, lr=0.0001, emb=512, hidden=512, vocab=20000, min_size=64, max_size=512, bf16=True),
        # many keys in flight with Adam: the setting of a user who wants throughput from a small recurrent model
        _case("rnn_train_adam_256", family="rnn", n=20000, mak=256, muf=200, lr=0.00002, hidden=128, classes=10, vocab=14, max_size=10, optimizer="adam"),
        # plain SGD, one instance at a time and an update per gradient, odd widths: a first run on a few rows
        _case("mlp_train_sgd", family="mlp", n=64, mak=1, muf=1, lr=0.002, dim=61, hidden=37, classes=3),
        # validation accuracy after an epoch: forward-only pass over the loaded trees
        _case("tree_eval", family="tree", **{"pass": "eval"}, n=8544, mak=64, emb=300, hidden=150, vocab=20000, min_size=2, max_size=50),
        # validation loss of the graph network
        _case("ggnn_eval", family="ggnn", **{"pass": "eval"}, n=8000, mak=128, hidden=100, vocab=15, min_size=9, max_size=29),
        # one request of a service: eight new lists are loaded and evaluated
        _case("rnn_request", family="rnn", **{"pass": "request"}, n=8, mak=8, hidden=128, classes=10, vocab=14, max_size=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _most_work(case):
    """The case's multiply-adds and its longest chain of dependent messages, against what the largest listed cases have."""
    serial = _messages(case) / case["mak"] + _messages(case) / 64.0
    return max(work(case)["flops"] / 4.0e11, serial / 2.0e4)


def draw(rng):
    """One more case: family, pass, option and every size over the range that the listed ones span."""
    family = rng.choice(["mlp", "rnn", "rnn", "tree", "tree", "ggnn", "ggnn", "tree_lstm", "tree_bf16"])
    c = dict(DEFAULTS)
    c["pass"] = rng.choice(["train", "train", "train", "eval", "request"])
    c["mak"] = _log_int(rng, 1, 256)
    c["muf"] = _log_int(rng, 8, 300)
    c["optimizer"] = rng.choice(["sgd", "sgd", "sgd", "momentum", "adam"])
    if family == "mlp":
        c.update(family="mlp", n=_log_int(rng, 16, 4096), dim=_log_int(rng, 16, 784), hidden=_log_int(rng, 16, 256), classes=rng.randint(2, 10))
    elif family == "rnn":
        c.update(family="rnn", n=_log_int(rng, 8, 20000), hidden=rng.randint(32, 160), classes=10, vocab=14, max_size=rng.randint(2, 12))
    elif family == "ggnn":
        c.update(family="ggnn", n=_log_int(rng, 16, 8000), hidden=rng.randint(24, 100), vocab=15, min_size=rng.randint(2, 9), max_size=rng.randint(10, 29), steps=rng.randint(2, 4))
    else:
        low = rng.randint(2, 64) if family == "tree_bf16" else 2
        c.update(family="tree_lstm" if family == "tree_lstm" else "tree", n=_log_int(rng, 8, 8544), emb=rng.randint(32, 300), hidden=rng.randint(32, 150),
                 vocab=_log_int(rng, 500, 20000), min_size=low, max_size=rng.randint(low, 512 if family == "tree_bf16" else 50))
        if family == "tree_bf16":
            c.update(bf16=True, emb=64 * rng.randint(2, 8))
            c["hidden"] = c["emb"]
    c["lr"] = {"mlp": 2e-3, "rnn": 2e-3, "tree": 5e-4, "tree_lstm": 5e-4, "tree_bf16": 5e-5, "ggnn": 1e-6}[family] * (0.1 if c["optimizer"] == "momentum" else 1.0)
    if c["optimizer"] == "adam":
        c["lr"] = 2e-5
    if c["pass"] == "request":
        c["n"] = min(c["n"], 64)
    if c["pass"] != "train":
        c.update(muf=1, lr=0.0, optimizer="sgd")
    c["mak"] = min(c["mak"], c["n"])
    while c["n"] > 8 and _most_work(c) > 1.0:           # no dearer than the largest listed case
        c["n"] = max(8, int(c["n"] * 0.7))
        c["mak"] = min(c["mak"], c["n"])
    while _most_work(c) > 1.0 and c["max_size"] > 2:    # (one key in flight on large trees)
        c["max_size"] = max(2, c["max_size"] // 2)
        c["min_size"] = min(c["min_size"], c["max_size"])
    return c


# ---- models and data ---------------------------------------------------------------------------------------
class _Graph:
    """The IR tables of a model family, from the library's builders, in the form Engine takes."""

    def __init__(self, case):
        f = case["family"]
        args = {"mlp": ([case["dim"], case["hidden"], case["hidden"], case["classes"]],),
                "rnn": (case["vocab"], case["hidden"], case["hidden"], case["classes"], ACT_TANH),
                "tree": (case["vocab"], case["emb"], case["hidden"], case["classes"]),
                "tree_lstm": (case["vocab"], case["emb"], case["hidden"], case["classes"]),
                "ggnn": (case["vocab"], case["hidden"], case["steps"], 4, case["hidden"])}[f]
        self.nodes, self.edges = amp.ir_tables(f, *args)

    def ppt_nodes(self):
        return [i for i, n in enumerate(self.nodes) if n[0] in (LINEAR, LOOKUP, GRUCELL)]

    def param_shapes(self, i):
        t, din, dout = (int(v) for v in self.nodes[i][:3])
        if t == LINEAR:
            return [(0, (dout, din)), (1, (dout,))]
        if t == LOOKUP:
            return [(0, (din, dout))]
        return [(k, (dout, din)) for k in range(3)] + [(k, (dout,)) for k in range(3, 6)]


class _Instances:
    def __init__(self, kind, n):
        self.kind, self.n = kind, n
        for k in ("offsets", "tokens", "left", "right", "edge_offsets", "edge_src", "edge_dst", "edge_type", "dense", "labels_i", "labels_f"):
            setattr(self, k, None)


def _offsets(sizes):
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _dense_rows(case, rng):
    x = rng.random((case["n"], case["dim"]), dtype=np.float32)
    teacher = np.random.default_rng(11).standard_normal((case["dim"], case["classes"])).astype(np.float32)
    out = _Instances(KIND_DENSE, case["n"])
    out.dense, out.labels_i = x, np.argmax((x - 0.5) @ teacher, axis=1).astype(np.int32)
    return out


def _lists(case, rng):
    n = case["n"]
    length = rng.integers(1, case["max_size"] + 1, size=n)
    op = rng.integers(0, 4, size=n)
    off = _offsets(length + 1)
    tokens = rng.integers(0, 10, size=int(off[-1])).astype(np.int32)
    tokens[off[:-1]] = 0
    first = off[:-1] + 1
    sums = np.add.reduceat(tokens, off[:-1]) % 10
    most = np.maximum.reduceat(tokens, off[:-1])
    tokens[off[:-1]] = 9                                        # not below any digit, for the minimum
    least = np.minimum.reduceat(tokens, off[:-1])
    label = np.choose(op, [sums, most, least, tokens[first]])
    tokens[off[:-1]] = 10 + op                                  # vocabulary: ten digits, four operators
    out = _Instances(KIND_LISTS, n)
    out.offsets, out.tokens, out.labels_i = off, tokens, label.astype(np.int32)
    return out


def _trees(case, rng):
    """Random binary trees by recursive uniform splits, in post-order (children precede parents), all trees level by level:
    a subtree with k leaves fills 2k - 1 consecutive positions, its root last."""
    n = case["n"]
    leaves = rng.integers(case["min_size"], case["max_size"] + 1, size=n)
    off = _offsets(2 * leaves - 1)
    total = int(off[-1])
    left, right = np.full(total, -1, np.int32), np.full(total, -1, np.int32)
    k, start, base = leaves.copy(), off[:-1].copy(), off[:-1].copy()      # open subtrees: leaves, first position, tree's base
    while len(k):
        inner = k > 1
        k, start, base = k[inner], start[inner], base[inner]
        kl = rng.integers(1, np.maximum(k, 2))
        root = start + 2 * k - 2
        left[root], right[root] = start + 2 * kl - 2 - base, root - 1 - base
        k, start, base = np.concatenate([kl, k - kl]), np.concatenate([start, start + 2 * kl - 1]), np.concatenate([base, base])
    is_leaf = left < 0
    p = np.arange(1, case["vocab"] + 1, dtype=np.float64) ** -1.1
    words = np.minimum(np.searchsorted(np.cumsum(p / p.sum()), rng.random(int(is_leaf.sum()))), case["vocab"] - 1)
    tokens = np.full(total, -1, np.int32)
    tokens[is_leaf] = words
    # label of a node: the class of its subtree's mean word score (a stand-in for sentiment)
    score = np.zeros(total + 1)
    score[1:][is_leaf] = np.random.default_rng(12).standard_normal(case["vocab"])[words]
    size = np.ones(total, np.int64)                              # positions of the subtree: 1 at a leaf, else back to its leftmost leaf
    pos = np.arange(total)
    tree_base = np.repeat(off[:-1], np.diff(off))
    first = pos.copy()
    inner = np.nonzero(~is_leaf)[0]
    for _ in range(64):                                          # pointer jumping along left children
        nxt = first[tree_base[inner] + left[inner]]
        if np.array_equal(nxt, first[inner]):
            break
        first[inner] = nxt
    size = pos - first + 1
    csum = np.cumsum(score)
    mean = (csum[pos + 1] - csum[first]) / ((size + 1) / 2)
    edges = np.quantile(mean, np.linspace(0, 1, case["classes"] + 1)[1:-1])
    out = _Instances(KIND_TREES, n)
    out.offsets, out.left, out.right, out.tokens = off, left, right, tokens
    out.labels_i = np.searchsorted(edges, mean).astype(np.int32)
    return out


def _graphs(case, rng):
    """Molecule-like graphs: a random spanning tree and a few ring-closing bonds, every bond two directed edges of one of four
    types; the target follows the composition."""
    n = case["n"]
    size = rng.integers(case["min_size"], case["max_size"] + 1, size=n)
    off = _offsets(size)
    total = int(off[-1])
    gid = np.repeat(np.arange(n), size)
    local = np.arange(total) - off[gid]
    p = np.arange(1, case["vocab"] + 1, dtype=np.float64) ** -1.5
    tokens = np.minimum(np.searchsorted(np.cumsum(p / p.sum()), rng.random(total)), case["vocab"] - 1).astype(np.int32)
    v = np.nonzero(local > 0)[0]
    pairs = [np.stack([gid[v], (rng.random(len(v)) * local[v]).astype(np.int64), local[v]], 1)]
    extra = np.repeat(np.arange(n), np.maximum(0, np.rint(1.05 * size).astype(np.int64) - size + 1))
    extra = extra[size[extra] > 3]
    a = (rng.random(len(extra)) * size[extra]).astype(np.int64)
    b = (a + 1 + (rng.random(len(extra)) * (size[extra] - 1)).astype(np.int64)) % size[extra]
    pairs.append(np.stack([extra, np.minimum(a, b), np.maximum(a, b)], 1))
    pairs = np.unique(np.concatenate(pairs), axis=0)            # no bond twice; sorted by graph
    bond = np.minimum(np.searchsorted(np.cumsum([0.75, 0.12, 0.03, 0.10]), rng.random(len(pairs))), 3)
    out = _Instances(KIND_GRAPHS, n)
    out.offsets, out.tokens = off, tokens
    out.edge_offsets = _offsets(2 * np.bincount(pairs[:, 0], minlength=n))
    out.edge_src = pairs[:, [1, 2]].astype(np.int32).reshape(-1)
    out.edge_dst = pairs[:, [2, 1]].astype(np.int32).reshape(-1)
    out.edge_type = np.repeat(bond.astype(np.int32), 2)
    w = np.random.default_rng(13).standard_normal(case["vocab"])
    y = np.add.reduceat(w[tokens], off[:-1])
    out.labels_f = ((y - y.mean()) / (y.std() + 1e-6)).astype(np.float32)
    return out


def _parameters(graph, rng):
    """Matrices U(+-sqrt(6 / (in + out))), biases U(+-1 / sqrt(in)), embeddings N(0, 0.1)."""
    out = {}
    for i in graph.ppt_nodes():
        t, din, dout = (int(v) for v in graph.nodes[i][:3])
        for which, shape in graph.param_shapes(i):
            if t == LOOKUP:
                out[(i, which)] = 0.1 * rng.standard_normal(shape, dtype=np.float32)
            else:
                lim = math.sqrt(6.0 / (din + dout)) if len(shape) == 2 else 1.0 / math.sqrt(din)
                out[(i, which)] = ((2.0 * rng.random(shape, dtype=np.float32) - 1.0) * lim).astype(np.float32)
    return out


def _data(case, seed):
    rng = np.random.default_rng([20170509, seed])
    make = {"mlp": _dense_rows, "rnn": _lists, "tree": _trees, "tree_lstm": _trees, "ggnn": _graphs}[case["family"]]
    return make(case, rng)


def prepare(case, seed):
    """The engine with its weights and its loaded data set; a request comes as host arrays."""
    graph = _Graph(case)
    engine = amp.Engine(graph, payload_bf16=case["bf16"])
    engine.set_params(_parameters(graph, np.random.default_rng([7, seed])))
    inst = _data(case, seed)
    state = {"case": case, "engine": engine, "instances": inst}
    if case["pass"] == "train":
        engine.load_instances(inst)
        if case["optimizer"] != "sgd":
            engine.set_optimizer(case["optimizer"])
        state["params"] = {"%d.%d" % k: v for k, v in engine.param_tensors().items()}
    elif case["pass"] == "eval":
        engine.load_instances(inst, split=1)
    return state


def run(state):
    case, engine = state["case"], state["engine"]
    if case["pass"] == "train":
        st, loss = engine.run_epoch(mak=case["mak"], muf=case["muf"], lr=case["lr"])
        return {"loss": loss, "mean_loss": st.mean_loss, "instances": st.instances, "node_messages": st.node_messages, "params": state["params"]}
    if case["pass"] == "request":
        engine.load_instances(state["instances"], split=1)
    mean_loss, accuracy, loss = engine.eval(split=1, mak=case["mak"])
    return {"loss": loss, "mean_loss": mean_loss, "accuracy": accuracy}


# ---- what a pass cannot do without -----------------------------------------------------------------------------
def _mean_size(case):
    return 0.5 * (case["min_size"] + case["max_size"])


def _messages(case):
    """Parameterised-node messages of a pass, about (forward; training answers each with a backward one)."""
    m = {"mlp": 3.0, "rnn": 2 * (_mean_size(case) + 1) + 1, "tree": 5 * _mean_size(case), "tree_lstm": 5 * _mean_size(case),
         "ggnn": 5.0 * case["steps"] + 3}[case["family"]]
    return case["n"] * m * (2 if case["pass"] == "train" else 1)


def _linear_rows(case):
    """[(rows per instance, in, out, has input gradient)] of the dense layers of one instance."""
    h, s = case["hidden"], _mean_size(case)
    f = case["family"]
    if f == "mlp":
        return [(1, case["dim"], h, False), (1, h, h, True), (1, h, case["classes"], True)]
    if f == "rnn":
        return [(s + 1, 2 * h, h, True), (1, h, case["classes"], True)]
    if f == "tree":
        return [(s, case["emb"], h, True), (s - 1, 2 * h, h, True), (2 * s - 1, h, case["classes"], True)]
    if f == "tree_lstm":
        return [(s, case["emb"], 3 * h, True), (s - 1, 2 * h, 5 * h, True), (2 * s - 1, h, case["classes"], True)]
    edges = 2 * max(s - 1, 1.05 * s)
    return [(case["steps"] * edges, h, h, True), (case["steps"] * s, 2 * h, 3 * h, True), (1, h, h, True), (1, h, 1, True)]


def work(case):
    n, s, train = case["n"], _mean_size(case), case["pass"] == "train"
    rows = _linear_rows(case)
    flops = sum(n * r * 2.0 * i * o * ((3 if dx else 2) if train else 1) for r, i, o, dx in rows)
    weights = sum((i + 1.0) * o * (4 if case["family"] == "ggnn" and k == 0 else 1) for k, (_, i, o, _) in enumerate(rows))
    if case["family"] in TREE_FAMILIES:
        touched, width, structure = min(case["vocab"], n * s), case["emb"], (2 * s - 1) * 16.0 + 8
    elif case["family"] == "rnn":
        touched, width, structure = min(case["vocab"], n * s), case["hidden"], (s + 1) * 4.0 + 12
    elif case["family"] == "ggnn":
        touched, width, structure = min(case["vocab"], n * s), case["hidden"], s * 4.0 + 2.1 * s * 12.0 + 20
    else:
        touched, width, structure = 0, 0, case["dim"] * 4.0 + 4
    params = 4.0 * (weights + touched * width)
    states = {"sgd": 1, "momentum": 2, "adam": 3}[case["optimizer"]]
    return {"bytes": n * (structure + 4.0) + params * (2 * states if train else 1), "flops": flops}


def tolerance(case):
    if case["pass"] != "train":
        # forward values: single-precision sums, or bfloat16 payloads that may round either way
        return {"rel": 2e-2, "max": 0.2, "differ": 0.0} if case["bf16"] else {"rel": 1e-5, "max": 1e-3, "differ": 0.0}
    # An asynchronous epoch has no one schedule: which update a message sees depends on what else is in flight (staleness up to
    # max_active_keys instances), so losses and parameters of two correct runs differ by about an update's worth.
    return {"rel": 1e-2, "max": 0.3, "differ": 0.0}
