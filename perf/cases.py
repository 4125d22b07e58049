"""The work a user of this library has it do, as measurable cases.

Sizes are those of the paper's node-classification workloads (its dataset, cost and entropy tables, and the recipes
in ``synth``) and their neighbourhood: citation graphs of a few thousand nodes, where a whole forward is a handful of
short launches, up to co-purchase graphs of millions of nodes, where it is bound by the gathers of the aggregation.
Every case draws a graph, features and weights from its seed alone, through the library's own synthetic recipes, and
sets up what a program keeps: the normalised adjacency, the packed weights, the frozen batch-norm constants.

Kinds of case

  forward    ``BiGCN.forward`` / ``forward_packed`` of the whole network (inference)
  pipeline   consecutive forwards of host-resident inputs through ``open_pipeline``, copies included
  sage       the Bi-GraphSAGE stack: pack the features, then ``sage_layer_forward`` per layer
  backward   ``layer_backward`` of one layer (Algorithm 1), with or without the gradient of its input
  train      one training step: the forward layer by layer, every layer's input normalised with the batch's own
             statistics, then ``layer_backward`` from the last layer to the first
  entropy    ``entropy_bins`` over a matrix of activations (the capacity analysis)
"""
import math

import torch

from paper_2210_13149_b200 import binding, synth


def _net(name, kind, n, edges, dims, features, density=1.0, packed=False, steps=1):
    return {"name": name, "kind": kind, "n": n, "edges": edges, "dims": dims, "features": features,
            "density": density, "packed": packed, "steps": steps}


def listed():
    return [
        # Citation graph with bag-of-words features: the smallest network, all latency and launches.
        _net("citation_forward", "forward", 2_708, 10_556, "1433-64-7", "bernoulli", 0.013),
        # The same kind with the widest features, loaded already binary (1 bit per element and a scalar per node).
        _net("citation_packed", "forward", 3_327, 9_104, "3703-64-6", "bernoulli", 0.0085, packed=True),
        # TF-IDF features on a mid-sized citation graph.
        _net("tfidf_forward", "forward", 19_717, 88_648, "500-64-3", "tfidf", 0.10),
        # One training step on it.
        _net("tfidf_train", "train", 19_717, 88_648, "500-64-3", "tfidf", 0.10),
        # Inductive image graph (the paper's Flickr sizes) with the mean aggregator.
        _net("image_sage", "sage", 89_250, 899_756, "500-256-7", "normal"),
        # Paper-citation graph of the OGB setups: three layers.
        _net("papers_forward", "forward", 169_343, 2_332_486, "128-256-256-40", "normal"),
        # Dense social graph, rows of about 490 stored entries.
        _net("social_forward", "forward", 232_965, 114_600_000, "602-256-41", "normal"),
        # Co-purchase graph: the largest network, the benchmark's own configuration.
        _net("products_forward", "forward", 2_449_029, 123_700_000, "100-256-256-47", "normal"),
        # The same graph with Bi-GraphSAGE layers.
        _net("products_sage", "sage", 2_449_029, 123_700_000, "100-256-256-47", "normal"),
        # Back-propagation through its widest layer.
        {"name": "products_backward", "kind": "backward", "n": 2_449_029, "edges": 123_700_000, "dims": "256-256", "input_gradient": True},
        # A tenth of it served from host memory: eight binary inputs in, eight sets of logits out, three slots.
        _net("served_pipeline", "pipeline", 244_903, 12_370_000, "100-256-256-47", "normal", packed=True, steps=8),
        # Entropy of a hidden layer of the largest network (largest row of the paper's entropy table).
        {"name": "products_entropy", "kind": "entropy", "n": 2_449_029, "d": 128, "bins": 1000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: sizes spread over their logarithm, widths round and odd."""
    kind = rng.choice(["forward", "forward", "forward", "sage", "backward", "train", "entropy", "pipeline"])
    if kind == "entropy":
        n = _log_int(rng, 2_000, 2_449_029)
        return {"kind": kind, "n": n, "d": min(_log_int(rng, 16, 512), 300_000_000 // n), "bins": _log_int(rng, 50, 2_000)}
    n = _log_int(rng, 2_000, 250_000 if kind in ("pipeline", "train") else 2_449_029)
    degree = math.exp(rng.uniform(math.log(3), math.log(500)))
    edges = int(min(n * degree, n * (n - 1) * 0.05, 30_000_000))
    hidden = rng.choice([64, 128, 256] if kind == "train" else [16, 32, 64, 64, 128, 256, 256, _log_int(rng, 16, 256)])
    if kind == "backward":
        return {"kind": kind, "n": n, "edges": edges, "dims": "%d-%d" % (rng.choice([hidden, _log_int(rng, 50, 700)]), hidden),
                "input_gradient": rng.random() < 0.5}
    d0 = min(_log_int(rng, 50, 3_703), 245_000_000 // n)
    layers = 2 if kind == "train" else rng.choice([2, 2, 3])
    features = rng.choice(["bernoulli", "tfidf", "normal"])
    case = _net("", kind, n, edges, "-".join(map(str, [d0] + [hidden] * (layers - 1) + [rng.randint(2, 50)])), features,
                round(rng.uniform(0.01, 0.2), 3) if features != "normal" else 1.0)
    del case["name"]
    if kind == "forward":
        case["packed"] = rng.random() < 0.3
    if kind == "pipeline":
        case["packed"], case["steps"] = rng.random() < 0.5, rng.randint(3, 8)
    return case


def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _seed(seed):
    return seed % 1_000_003 + 17


def _frozen_constants(H, hidden):
    """Batch-norm constants of a layer's input: 1 / std of every column, and a shift at its mean -- for a hidden layer at
    the middle of the widest gap between two of the column's values next to the mean.  A hidden activation is the SIGN of
    an fp32 sum minus its shift: with no sum within rounding of the shift, every correct implementation takes the same
    signs, and outputs can be compared as closely as fp32 sums can."""
    n, d = H.shape
    mean, var = torch.empty(d, dtype=torch.float64, device=H.device), torch.empty(d, dtype=torch.float64, device=H.device)
    for a in range(0, d, 32):
        block = H[:, a:a + 32].double()
        mean[a:a + 32], var[a:a + 32] = block.mean(0), block.var(0, unbiased=False)
    if hidden:
        near = var.sqrt() * (0.02 if n > 100_000 else 0.1)
        for j in range(d):
            column = H[:, j].double()
            column = column[(column - mean[j]).abs() <= near[j]].sort().values
            if column.numel() > 1 and column[0] < column[-1]:
                k = column.diff().argmax()
                mean[j] = (column[k] + column[k + 1]) / 2
            else:
                mean[j] -= near[j] + 1e-3
    return mean.float(), (var + 1e-5).rsqrt().float()


def prepare(case, seed):
    seed, dev, ctx = _seed(seed), "cuda", binding.BiGCN(0)
    s = {"case": case, "ctx": ctx}
    gen = torch.Generator(device=dev).manual_seed(seed)
    if case["kind"] == "entropy":
        # Activations with a spread of their own per neuron, every fourth neuron rectified.
        n, d = case["n"], case["d"]
        H = torch.randn((n, d), device=dev, generator=gen) * (torch.rand(d, device=dev, generator=gen) * 3.8 + 0.2)
        H[:, ::4].clamp_(min=0)
        s["H"] = H
        return s
    n, dims = case["n"], _dims(case)
    rowptr, colidx = synth.power_law_graph(n, case["edges"], seed, device=dev)
    s["W"] = W = synth.weights(dims, seed, dev)
    if case["kind"] == "backward":
        s["graph"] = ctx.normalize_adjacency(rowptr, colidx)
        s["layer"] = ctx.prepare_layers(W)[0]
        s["bits"], s["beta"] = ctx.pack_features(torch.randn((n, dims[0]), device=dev, generator=gen))
        s["g_out"] = torch.randn((n, dims[1]), device=dev, generator=gen) * 0.02
        return s
    X = synth.features(case["features"], n, dims[0], seed, case["density"], dev)
    L = len(dims) - 1
    s["X"] = X
    if case["kind"] == "sage":
        s["graph"] = G = ctx.mean_adjacency(rowptr, colidx)
        W_nbr = synth.weights(dims, seed + 7, dev)
        nbr = ctx.prepare_layers(W_nbr)
    else:
        s["graph"] = G = ctx.normalize_adjacency(rowptr, colidx)
    if case["kind"] == "train":
        s["g_out"] = torch.randn((n, dims[-1]), device=dev, generator=gen) * 0.02
        return s
    # The batch-norm constants of every layer, frozen from the network's own activations; a served network sees three
    # inputs, its nodes' features in another order each.
    inputs, layers = [X.roll(k, 0) for k in range(3)] if case["kind"] == "pipeline" else [X], []
    H = inputs
    for l in range(L):
        shift, scale = _frozen_constants(H[0] if len(H) == 1 else torch.cat(H), l > 0)
        packed = [ctx.pack_features(h, shift, scale) for h in H]
        if l == 0:
            s["bits"], s["beta"] = packed[0]
            first = packed
        layers += ctx.prepare_layers([W[l]], [shift], [scale])
        if case["kind"] == "sage":
            H = [ctx.sage_layer_forward(G, layers[l], nbr[l], *p)["h"] for p in packed if l + 1 < L]
        else:
            H = [ctx.layer_forward(G, layers[l], *p)["h"] for p in packed if l + 1 < L]
    s["layers"] = layers
    if case["kind"] == "sage":
        s["pairs"] = list(zip(layers, nbr))
    if case["kind"] == "pipeline":
        s["inputs"] = [[t.cpu().pin_memory() for t in (p if case["packed"] else [x])] for x, p in zip(inputs, first)]
        s["logits"] = [torch.empty((n, dims[-1]), dtype=torch.float32, pin_memory=True) for _ in range(case["steps"])]
        s["pipe"] = ctx.open_pipeline(G, layers, slots=3)
    return s


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "forward":
        if case["packed"]:
            return ctx.forward_packed(s["graph"], s["layers"], s["bits"], s["beta"])
        return ctx.forward(s["graph"], s["layers"], s["X"])
    if kind == "pipeline":
        pipe = s["pipe"]
        for k, out in enumerate(s["logits"]):
            if k >= 3:
                pipe.wait()
            (pipe.submit_packed if case["packed"] else pipe.submit)(*s["inputs"][k % 3], out)
        while pipe.wait() is not None:
            pass
        return s["logits"]
    if kind == "sage":
        pairs = s["pairs"]
        bits, beta = ctx.pack_features(s["X"], pairs[0][0].in_shift, pairs[0][0].in_scale)
        for l, (own, nbr) in enumerate(pairs):
            last = l + 1 == len(pairs)
            out = ctx.sage_layer_forward(s["graph"], own, nbr, bits, beta, want_h=last,
                                         next_layer=None if last else pairs[l + 1][0])
            bits, beta = out["next_bits"], out["next_beta"]
        return out["h"]
    if kind == "backward":
        return ctx.layer_backward(s["graph"], s["layer"], s["W"][0], s["bits"], s["beta"], s["g_out"],
                                  want_g_in=case["input_gradient"])
    if kind == "train":
        # The weights change every step, so a step packs them; a layer's input is normalised with this step's statistics.
        H, saved = s["X"], []
        for W in s["W"]:
            shift, scale = ctx.col_stats(H)
            layer = ctx.prepare_layers([W], [shift], [scale])[0]
            bits, beta = ctx.pack_features(H, shift, scale)
            H = ctx.layer_forward(s["graph"], layer, bits, beta)["h"]
            saved.append((layer, W, bits, beta))
        grads, g = [], s["g_out"]
        for l in range(len(saved) - 1, -1, -1):
            layer, W, bits, beta = saved[l]
            g, g_w = ctx.layer_backward(s["graph"], layer, W, bits, beta, g, want_g_in=l > 0)
            grads.append(g_w)
        return H, grads
    return ctx.entropy_bins(s["H"], case["bins"])


def work(case):
    """Bytes: every input read once, every result written once.  Operations: the contraction of every layer (its binary
    multiply-adds) and its aggregation over the narrower of its two sides."""
    n = case["n"]
    if case["kind"] == "entropy":
        d, M = case["d"], case["bins"]
        return {"bytes": 4 * n * d + 4 * d * M + 16 * d, "flops": 4 * n * d}
    dims, nnz = _dims(case), case["edges"] + n
    csr = 8 * nnz + 8 * (n + 1)
    weights = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
    layer_flops = sum(2 * n * a * b + 2 * nnz * min(a, b) for a, b in zip(dims[:-1], dims[1:]))
    x_bits = n * (dims[0] / 8 + 4)
    if case["kind"] == "backward":
        g_in = n * dims[0] if case["input_gradient"] else 0
        return {"bytes": csr + x_bits + 4 * (n * dims[1] + g_in + 2 * weights),
                "flops": layer_flops + (2 * g_in * dims[1])}
    if case["kind"] == "train":
        return {"bytes": csr + 4 * (n * dims[0] + 2 * n * dims[-1] + 2 * weights), "flops": 3 * layer_flops}
    x = x_bits if case["packed"] else 4 * n * dims[0]
    one = {"bytes": x + 4 * n * dims[-1], "flops": layer_flops}
    if case["kind"] == "sage":
        one["flops"] += sum(2 * n * a * b for a, b in zip(dims[:-1], dims[1:]))
    steps = case["steps"]
    return {"bytes": csr + weights / 8 + steps * one["bytes"], "flops": steps * one["flops"]}


def tolerance(case):
    """Sums are fp32 (entropies are double sums over exact counts).  In a training step the thresholds are the batch's own
    means, so single hidden activations lie within rounding of them: correct implementations differ in such a bit, which
    moves the integer dots of its node by 2, of a spread of sqrt(width) >= 7, and more where few terms are averaged."""
    if case["kind"] == "entropy":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    if case["kind"] == "train":
        return {"rel": 1e-2, "max": 0.9}
    return {"rel": 1e-5, "max": 5e-4}
