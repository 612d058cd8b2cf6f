"""The work that a user has the framework do, as cases that can be timed and checked.

A case is one mutation-testing call, or one whole job (prefix cache, then the mutant table), on
one of the network families that the library takes: the fully connected network, LeNet-5, the
VGG-style network, ResNet-20, ResNet-10 (projection shortcuts), the MobileNetV2-style network
(depthwise layers) and the recurrent models (embedding and LSTM layers, 2 and 90 classes).
Sizes are those of the named workloads, or parts of them: tens of inputs and a handful of mutants
(a developer trying a test), a thousand inputs, the 10,000 of a whole test set.

Fields of a case: `net` the network; `mode` "memo" (the cache is kept from earlier: another table
on the same inputs), "job" (the cache is built in the pass) or "vanilla" (every mutant end to
end, the comparison that soundness is checked with); `n_in` and `n_mut`; `ratio` the selection
ratio; `wide` the neurons of a mutant drawn over the whole model instead of one layer; `ops` the
operators in rotation (the paper's set has WS, the named workloads' has NS); `precision`;
`labels` (kills counted against given labels); `logits` (every mutant's logits are asked for);
`skip` (the exact elimination of unchanged rows); `device` (outputs left on the GPU).
"""
import math
import random

import numpy as np
import torch

from paper_2607_18582_gb300 import mure
from paper_2607_18582_gb300 import workloads as wl

CONFIG = "GF,NEB,NAI,NS"     # the named workloads' rotation
PAPER = "GF,NAI,WS,NEB"      # the operator set of the paper's Sec. 3.1


def _case(net, mode, n_in, n_mut, **more):
    c = {"net": net, "mode": mode, "n_in": n_in, "n_mut": n_mut, "ratio": 0.01, "wide": False, "ops": CONFIG,
         "precision": "tf32x3", "labels": False, "logits": True, "skip": False, "device": True}
    c.update(more)
    return c


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # a developer trying a few mutants on a few inputs: latency and launches
        named("mlp_few", "mlp", "memo", 50, 8, device=False),
        # the fully connected workload, whole: 1,000 inputs x 200 mutants with its cache
        named("mlp_job", "mlp", "job", 1000, 200, ops=PAPER, labels=True, logits=False, device=False),
        # LeNet-5 on a whole test set, kill matrix and scores only
        named("lenet5_job", "lenet5", "job", 10000, 1000, logits=False),
        # the paper's 3 % model-wide selection: mutants over several layers
        named("lenet5_modelwide", "lenet5", "memo", 2500, 397, ratio=0.03, wide=True),
        # the vanilla comparison that a memoized run is checked against
        named("lenet5_vanilla", "lenet5", "vanilla", 1200, 90, labels=True),
        # plain fp32 arithmetic, as the CPU drift comparison wants it
        named("lenet5_fp32", "lenet5", "job", 1500, 150, precision="fp32"),
        # the benchmark's network: one table slice on a tenth of its inputs, the largest work here
        named("vgg_job", "vgg", "job", 1000, 250, ratio=0.02),
        # ResNet-20: residual adds, option-A shortcuts, global average pooling
        named("resnet20_job", "resnet20", "job", 600, 60),
        # ResNet-10 at reduced precision with the unchanged rows dropped: a quick screening run
        named("resnet10_screen", "resnet10", "memo", 333, 45, precision="tf32", skip=True),
        # MobileNetV2 blocks: 1x1 and depthwise convolutions, ReLU6
        named("mobilenetv2_job", "mobilenetv2_tiny", "job", 500, 41, ops=PAPER),
        # sentiment model: embedding and two LSTM layers, 80 steps
        named("rnn_imdb_job", "rnn_imdb", "job", 500, 40, ops=PAPER),
        # topic model of 90 classes, an odd number of documents on a kept cache
        named("rnn_reuters_odd", "rnn_reuters", "memo", 201, 23, labels=True),
    ]


# a drawn case: inputs and mutants over these ranges (log-uniform); the product is bounded per
# network so that no drawn case costs more than the VGG job above
_RANGE = {"mlp": ((30, 5000), (4, 800), 4e6), "lenet5": ((40, 10000), (6, 2000), 5e6), "vgg": ((20, 1500), (4, 300), 6e4),
          "resnet20": ((20, 1500), (4, 200), 6e4), "resnet10": ((20, 1500), (4, 200), 6e4),
          "mobilenetv2_tiny": ((20, 2000), (4, 200), 6e4), "rnn_imdb": ((20, 1500), (4, 150), 3e4),
          "rnn_reuters": ((20, 1500), (4, 150), 3e4)}


def draw(rng: random.Random):
    net = rng.choice(sorted(_RANGE))
    (a, b), (c, d), most = _RANGE[net]
    mode = rng.choice(["job", "job", "memo", "memo", "vanilla"])
    precision = rng.choice(["tf32x3", "tf32x3", "tf32x3", "tf32", "fp32"])
    if mode == "vanilla":
        most /= 4
    if precision == "fp32" and not net.startswith("rnn"):
        most /= 16 if net in ("vgg", "resnet20", "resnet10") else 4
    wide = net not in ("rnn_imdb", "rnn_reuters") and rng.random() < 0.2
    if wide:
        most /= 2
    n_in = int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    n_mut = int(round(math.exp(rng.uniform(math.log(c), math.log(d)))))
    n_mut = max(1, min(n_mut, int(most / n_in)))
    return _case(net, mode, n_in, n_mut, ratio=rng.choice([0.005, 0.01, 0.01, 0.02, 0.05]), wide=wide,
                 ops=rng.choice([CONFIG, CONFIG, PAPER]), precision=precision, labels=rng.random() < 0.4,
                 logits=rng.random() < 0.6, skip=mode != "vanilla" and rng.random() < 0.15,
                 device=rng.random() < 0.7)


# ------------------------------------------------------------------------- one pass

def _data(case, seed):
    """The network (the user's own: fixed weights), inputs, labels and mutant table of a seed."""
    net = wl.MODELS[case["net"]](0)
    X = wl.inputs(net, case["n_in"], seed=2 * seed + 1)
    ops = tuple(case["ops"].split(","))
    if case["wide"]:
        table = wl.modelwide_mutants(net, case["n_mut"], seed=2 * seed + 2, ratio=case["ratio"], ops=ops)
    else:
        table = wl.mutants(net, case["n_mut"], seed=2 * seed + 2, ratios=(case["ratio"],), ops=ops)
    labels = np.random.default_rng(seed).integers(0, net.n_classes, case["n_in"]).astype(np.int32) if case["labels"] else None
    return net, X, labels, table


_context = []


def _ctx():
    """A program's one library context."""
    if not _context:
        _context.append(mure.mure_create(0))
    return _context[0]


def prepare(case, seed):
    net, X, labels, table = _data(case, seed)
    model = mure.mure_model_load(_ctx(), net, precision=case["precision"])
    state = {"case": case, "model": model, "X": torch.from_numpy(X).cuda(), "table": table,
             "labels": None if labels is None else torch.from_numpy(labels).cuda(), "arrays": mure.table_array(table)}
    if case["mode"] == "memo":
        state["cache"] = mure.mure_build_prefix_cache(model, state["X"], state["labels"])
    return state


def run(state):
    c = state["case"]
    how = {"logits": c["logits"], "outputs_on_device": c["device"]}
    out = {}
    if c["mode"] == "vanilla":
        r = mure.mure_eval_vanilla(state["model"], state["X"], state["table"], state["labels"], **how)
    else:
        cache = state["cache"] if c["mode"] == "memo" else mure.mure_build_prefix_cache(state["model"], state["X"],
                                                                                         state["labels"])
        r = mure.mure_eval_mutants(cache, state["table"], arrays=state["arrays"], skip_unchanged=c["skip"], **how)
        if c["mode"] == "job":
            out["original_logits"], out["original_predictions"] = mure.mure_cache_outputs(cache)
            cache.free()
    out["kill_bits"] = r["kill_bits"]
    out["scores"] = np.array([r["scoreA"], r["scoreB"]])
    if c["logits"]:
        out["logits"] = r["logits"]
    return out


# ------------------------------------------------------------------- work and tolerance

def work(case):
    """Lemma 4's count: a forward pass for the cache, then for every mutant (layer uniform) the
    mutated neurons' own products and the layers after it; vanilla: every layer for every mutant.
    A mutated LSTM layer is recomputed whole.  Bytes: inputs and weights in, results out."""
    net = wl.MODELS[case["net"]](0)
    L = net.n_layers()
    macs = [net.layer_macs(l) for l in range(L)]
    full = float(sum(macs))
    widths = [net.layer_width(l) for l in range(L)]
    ops = case["ops"].split(",")
    dots = sum(o in ("GF", "WS") for o in ops) / len(ops)
    first = np.ones(L) / L
    if case["wide"]:   # P(smallest mutated layer = l) for k neurons drawn over the model
        k = max(1, int(case["ratio"] * sum(widths) + 0.5))
        tail = [(sum(widths[l:]) / sum(widths)) ** k for l in range(L)] + [0.0]
        first = np.array([tail[l] - tail[l + 1] for l in range(L)])
    rows = float(case["n_in"]) * case["n_mut"]
    per = 0.0
    for l in range(L):
        lstm = net.nodes[net.layers()[l]].kind == "lstm"
        k = max(1, int(case["ratio"] * widths[l] + 0.5))
        own = macs[l] if lstm else dots * macs[l] * k / widths[l]
        per += first[l] * (own + sum(macs[l + 1:]))
    macs_all = {"vanilla": full * (rows + case["n_in"]), "job": rows * per + full * case["n_in"], "memo": rows * per}
    size_x = float(np.prod(net.in_shape)) * 4
    weights = sum(float(n.W.size) * 4 for n in net.nodes if n.W is not None)
    out = case["n_mut"] * math.ceil(case["n_in"] / 64) * 8.0
    if case["logits"]:
        out += rows * net.n_classes * 4
    return {"bytes": case["n_in"] * size_x + weights + out, "flops": 2 * macs_all[case["mode"]]}


#: relative error of the logits against 64 bits as measured, times about four: three TF32 products
#: per product summed by the tensor cores (it grows with the fan-in and the depth), the layers that
#: run in plain fp32 (the recurrent models at every precision), one TF32 product
_REL = {"mlp": 3e-5, "lenet5": 2e-5, "vgg": 2.5e-4, "resnet20": 6e-5, "resnet10": 6e-5, "mobilenetv2_tiny": 5e-6}
_REL_FP32, _REL_TF32 = 2e-6, 2e-3


def tolerance(case):
    """A kill word (64 inputs) differs where one of its rows is a near tie."""
    rel = _REL_FP32 if case["precision"] == "fp32" else _REL_TF32 if case["precision"] == "tf32" else _REL.get(case["net"], _REL_FP32)
    if case["net"].startswith("rnn"):
        rel = _REL_FP32
    return {"rel": rel, "differ": 0.01 if rel == _REL_TF32 else 0.002}


# ---------------------------------------------------------------- the same in 64 bits

_M64 = (1 << 64) - 1


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _draws(seed, n):
    """Outputs 0 .. n-1 of SplitMix64 seeded `seed`, as the top 53 bits."""
    with np.errstate(over="ignore"):
        i = np.arange(1, n + 1, dtype=np.uint64)
        return _mix(np.uint64(seed) + i * np.uint64(0x9E3779B97F4A7C15))


def _fuzz(seed, q, fan, sigma):
    """Gaussian fuzzing's weight noise of neuron slot q (Box-Muller, rounded to fp32)."""
    u = _draws(int(_draws(seed, q + 1)[q]), 2 * ((fan + 1) // 2)) >> np.uint64(11)
    u1, u2 = (u[0::2].astype(np.float64) + 1) * 2.0 ** -53, (u[1::2].astype(np.float64) + 1) * 2.0 ** -53
    r, t = np.sqrt(-2 * np.log(u1)), 2 * math.pi * u2
    return (sigma * np.stack([r * np.cos(t), r * np.sin(t)], 1).reshape(-1)[:fan]).astype(np.float32).astype(np.float64)


def _shuffle(seed, q, fan):
    """Weight shuffling's permutation of neuron slot q (Fisher-Yates from the last down)."""
    u = (_draws(int(_draws(seed, q + 1)[q]), fan) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    p = list(range(fan))
    for i in range(fan - 1, 0, -1):
        j = min(int(u[fan - 1 - i] * (i + 1)), i)
        p[i], p[j] = p[j], p[i]
    return np.array(p)


def _act(name, v):
    return v.clamp(min=0) if name == "relu" else v.clamp(0, 6) if name == "relu6" else v


def _node(n, W, b, zero, ins):
    """One node on inputs in NHWC, all in 64 bits; `zero`: neurons held at 0."""
    x = ins[0]
    if n.kind in ("conv", "dwconv"):
        w = W.reshape(n.cout, n.kh, n.kw, -1).permute(0, 3, 1, 2)
        y = torch.nn.functional.conv2d(x.permute(0, 3, 1, 2), w, b, n.stride, n.pad, 1, n.cout if n.kind == "dwconv" else 1)
        y = y.permute(0, 2, 3, 1)
    elif n.kind == "dense":
        y = (x.reshape(len(x), -1) @ W.reshape(n.cout, -1).T + b).reshape(len(x), 1, 1, -1)
    elif n.kind == "embed":
        y = W.T[x[:, 0, :, 0].long()][:, None]
    elif n.kind == "lstm":
        N, _, T, C = x.shape
        H, live = n.cout, torch.ones(n.cout, dtype=x.dtype, device=x.device)
        if zero:
            live[zero] = 0
        W4 = W.reshape(H, 4, C + H)
        wx, wh, bb = W4[:, :, :C].reshape(4 * H, C).T, W4[:, :, C:].reshape(4 * H, H).T, b.reshape(4 * H)
        pre = x[:, 0] @ wx + bb
        h = c = torch.zeros(N, H, dtype=x.dtype, device=x.device)
        hs = []
        for t in range(T):
            i, f, g, o = (pre[:, t] + h @ wh).reshape(N, H, 4).unbind(2)
            c = f.sigmoid() * c + i.sigmoid() * g.tanh()
            h = o.sigmoid() * c.tanh() * live
            hs.append(h)
        return torch.stack(hs, 1)[:, None] if n.kh else h[:, None, None]
    elif n.kind == "maxpool":
        return torch.nn.functional.max_pool2d(x.permute(0, 3, 1, 2), (n.kh, n.kw), n.stride).permute(0, 2, 3, 1)
    elif n.kind == "flatten":
        return x.reshape(len(x), 1, 1, -1)
    elif n.kind == "add":
        return _act(n.act, x + ins[1])
    elif n.kind == "gap":
        return x.mean((1, 2), keepdim=True)
    else:   # option-A shortcut: subsample, append zero channels
        return torch.nn.functional.pad(x[:, ::n.stride, ::n.stride], (0, n.cout - x.shape[3]))
    y = _act(n.act, y)
    if zero:
        y = y.clone()
        y[..., zero] = 0
    return y


def _mutated(net, table, i):
    """{node: (W, b, neurons held at 0)} of mutant i, in 64 bits (numpy)."""
    nodes, op, seed = net.layers(), wl.OPS[int(table.op[i])], int(table.seed[i])
    pool = table.pool[int(table.neuron_off[i]):int(table.neuron_off[i]) + int(table.n_neurons[i])]
    spots = [(int(e) >> 20, int(e) & 0xFFFFF) if table.tagged is not None and table.tagged[i] else (int(table.layer[i]), int(e))
             for e in pool]
    out = {}
    for q, (l, j) in enumerate(spots):
        n = net.nodes[nodes[l]]
        if nodes[l] not in out:
            W = n.W.astype(np.float64).reshape(n.cout, -1)
            out[nodes[l]] = (W.copy(), np.zeros((n.cout, 1)) if n.b is None else n.b.astype(np.float64).reshape(n.cout, -1).copy(), [])
        W, b, zero = out[nodes[l]]
        W0 = n.W.astype(np.float64).reshape(n.cout, -1)
        b0 = np.zeros((n.cout, 1)) if n.b is None else n.b.astype(np.float64).reshape(n.cout, -1)
        if op == "GF":
            W[j] += _fuzz(seed, q, W.shape[1], float(np.float32(table.param[i])) * float(W0.std()))
        elif op == "WS":
            W[j] = W0[j][_shuffle(seed, q, W.shape[1])]
        elif op == "NAI":
            W[j], b[j] = -W0[j], -b0[j]
        elif op == "NS":
            m = spots[q ^ 1][1]
            W[j], b[j] = W0[m], b0[m]
        elif op == "NEB":
            zero.append(j)
    return out


#: 64-bit operations that take about 20 seconds here (matrix products and convolutions in fp64)
_MOST_FLOPS = 2.5e12


def exact(case, seed):
    net, X, _, table = _data(case, seed)
    forward = 2.0 * sum(net.layer_macs(l) for l in range(net.n_layers())) * case["n_in"]
    if forward > _MOST_FLOPS:
        return None
    many = work(dict(case, mode="memo"))["flops"] > _MOST_FLOPS
    if many and case["mode"] != "job":
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    x = up(X).double()
    W = {v: up(n.W.astype(np.float64)) for v, n in enumerate(net.nodes) if n.W is not None}
    b = {v: up(n.b.astype(np.float64)) for v, n in enumerate(net.nodes) if n.b is not None}

    def go(base, changed):
        """Every node's output: those that a changed node feeds anew, the others from base."""
        vals, dirty = {-1: x}, set()
        for v, n in enumerate(net.nodes):
            if base is not None and v not in changed and not any(u in dirty for u in n.inputs):
                vals[v] = base[v]
                continue
            dirty.add(v)
            w, bb, zero = W.get(v), b.get(v), None
            if v in changed:
                w, bb, zero = up(changed[v][0]), up(changed[v][1]), changed[v][2]
            vals[v] = _node(n, w, None if bb is None else bb.reshape(-1), zero, [vals[u] for u in n.inputs])
        return vals

    plain = go(None, {})
    last = len(net.nodes) - 1
    out = {"kill_bits": None, "scores": None}
    if case["mode"] == "job":
        out["original_logits"], out["original_predictions"] = plain[last].reshape(len(X), -1), None
    if case["logits"]:
        out["logits"] = None if many else torch.stack(
            [go(plain, _mutated(net, table, i))[last].reshape(len(X), -1) for i in range(len(table))])
    return out
