"""The work a user of this library has it do, as measurable cases.

Placeto (arXiv 1906.08879) evaluates a graph-embedding policy on batches of
placement states of one computation graph, rolls whole episodes out, trains the
policy by REINFORCE and simulates the run time of the placements it finds. A
case names one of these calls (`path`), a synthetic graph (`graph`, `size`,
`graph_seed`) and the policy's dimensions:

    d       embedding width            m       devices (F = m + 4 raw features)
    layers  layers of f and g: 2 in the workload configurations, 1 in the paper (Appendix A.7)
    batch   states, episodes or placements of one call

Paths:

    forward     placeto_policy_forward: a batch of states -> logits and probabilities
    host        placeto_policy_forward_host: the same from and to page-locked host buffers
    embeddings  placeto_build_features, placeto_embed_forward, placeto_policy_logits called one by
                one, which also hands the caller the features and the node embeddings
    rollout     placeto_episode_rollout: sampled episodes, every node placed once
    train       features, embeddings and placeto_policy_gradient of one batch of visited states
    simulate    placeto_simulate_placements: run time, peak memory and penalised run time

The sizes are those of the repository's workload configurations (32 nodes at
d = 8, about 300 to 1000 nodes at d = 32, about 2000 nodes at d = 64, batches of
16 to 992 states), of the paper's device counts (2, 4, 8) and, in `draw`, ragged
ones between and below them.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

import paper_1906_08879_b200 as placeto


def listed():
    return [
        # The smallest call: a 32-node graph on two devices, a handful of states. Launches and latency.
        dict(name="forward_tiny", path="forward", graph="layered", size=8, graph_seed=1, d=8, m=2, layers=2, batch=16),
        # One placement decision served from host memory (a scheduler asking for the next device).
        dict(name="host_one_state", path="host", graph="modules", size=11, graph_seed=2, d=32, m=4, layers=2, batch=1),
        # The Inception-shaped workload: a narrow, deep graph and a batch of placement states.
        dict(name="forward_modules", path="forward", graph="modules", size=11, graph_seed=2, d=32, m=4, layers=2, batch=256),
        # The paper's own networks (single-layer f and g) on two devices, a ragged batch.
        dict(name="forward_paper_2gpu", path="forward", graph="modules", size=11, graph_seed=2, d=32, m=2, layers=1, batch=250),
        # The NMT-shaped workload, step by step, for a caller that keeps the node embeddings.
        dict(name="embeddings_unrolled", path="embeddings", graph="unrolled", size=40, graph_seed=3, d=32, m=4, layers=2, batch=256),
        # The NASNet-shaped workload: the largest graph, d = 64, eight devices.
        dict(name="forward_cells_d64", path="forward", graph="cells", size=18, graph_seed=4, d=64, m=8, layers=2, batch=512),
        # All the states of one episode of a large recurrent graph, in one batch.
        dict(name="forward_episode_states", path="forward", graph="recurrent", size=990, graph_seed=1063, d=32, m=8, layers=2, batch=992),
        # A few sampled episodes on a small convolutional graph: one policy evaluation after another.
        dict(name="rollout_few", path="rollout", graph="conv", size=150, graph_seed=1010, d=32, m=8, layers=2, batch=16),
        # A training iteration's worth of sampled episodes on the Inception-shaped graph.
        dict(name="rollout_many", path="rollout", graph="modules", size=11, graph_seed=2, d=32, m=4, layers=2, batch=256),
        # The policy gradient of a batch of visited states, Inception-shaped graph.
        dict(name="train_modules", path="train", graph="modules", size=11, graph_seed=2, d=32, m=4, layers=2, batch=256),
        # The same at d = 64 on a stack of a few NAS cells, eight devices, a ragged batch.
        dict(name="train_cells_d64", path="train", graph="cells", size=5, graph_seed=4, d=64, m=8, layers=2, batch=100),
        # Scoring the placements of many episodes with the event-based simulator.
        dict(name="simulate", path="simulate", graph="modules", size=11, graph_seed=2, d=32, m=4, layers=2, batch=4096),
    ]


_SIZES = {"layered": (4, 40), "modules": (2, 11), "unrolled": (5, 40), "cells": (2, 18), "conv": (100, 1000), "recurrent": (100, 1000)}
_LARGEST = 2130 * 512 * 64 * 64      # nodes x states x d^2 of the largest batch of states that is evaluated at once


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case: any path on any of the graph shapes, sizes spread over their logarithm."""
    path = rng.choice(("forward", "forward", "host", "embeddings", "rollout", "train", "simulate"))
    graph = rng.choice(sorted(_SIZES))
    case = dict(path=path, graph=graph, size=_log_uniform(rng, *_SIZES[graph]), graph_seed=rng.randrange(1, 1000),
                d=rng.choice((32, 32, 64)), m=rng.choice((2, 3, 4, 5, 8)), layers=rng.choice((2, 2, 1)))
    if graph == "layered" and rng.random() < 0.5:
        case["d"] = 8
    if path == "rollout":            # as many steps as nodes: smaller graphs
        while _shape(case)[0] > 200 and case["size"] > 1:
            case["size"] = case["size"] * 2 // 3
    n = _shape(case)[0]
    most = {"forward": 1024, "embeddings": 1024, "host": 256, "rollout": 128, "train": 256, "simulate": 8192}[path]
    room = _LARGEST // (n * case["d"] ** 2)
    if path == "train":
        room //= 8                   # forward, backward and the rows kept between them
    if path == "rollout":
        room //= n
    if path == "simulate":
        room = most
    case["batch"] = max(1, min(_log_uniform(rng, 64 if path == "simulate" else 1, most), room))
    return case


# ------------------------------------------------------------------ graphs --

class _Edges:
    def __init__(self):
        self.n, self.src, self.dst = 0, [], []

    def node(self, *parents):
        self.src += parents
        self.dst += [self.n] * len(parents)
        self.n += 1
        return self.n - 1

    def chain(self, at, length):
        for _ in range(length):
            at = self.node(at)
        return at


def _layered(e, rng, levels, width=4):
    """`levels` x `width` nodes, one to three parents in the two levels above."""
    rows = []
    for lv in range(levels):
        above = [v for row in rows[-2:] for v in row]
        rows.append([e.node(*rng.sample(above, min(len(above), rng.randint(1, 3)))) if above else e.node() for _ in range(width)])


def _modules(e, rng, modules):
    """A stem chain, then modules of four parallel branches of short unit chains joined by one node."""
    join = e.chain(e.node(), 19)
    for _ in range(modules):
        join = e.node(*[e.chain(join, sum(rng.randint(2, 3) for _ in range(rng.randint(1, 4)))) for _ in range(4)])


def _unrolled(e, rng, steps, layers=2):
    """Encoder and decoder LSTM stacks unrolled over time, an attention node per decoder step over all encoder outputs."""
    def stack(h, c):
        below = e.node()
        for k in range(layers):
            gates = [e.node(*([below] + ([h[k]] if h[k] is not None else []))) for _ in range(4)]
            c[k] = e.node(*(gates + ([c[k]] if c[k] is not None else [])))
            h[k] = below = e.node(*gates)
        return below
    h, c = [None] * layers, [None] * layers
    top = [stack(h, c) for _ in range(steps)]
    for _ in range(steps):
        e.node(*top, stack(h, c))


def _cells(e, rng, cells, blocks=5):
    """A stack of NAS cells: adapters on the two previous cells, blocks that add two op chains, a concat of the loose ends."""
    before = e.node()
    last = e.node(before)
    for _ in range(cells):
        outs = [e.chain(last, 4), e.chain(before, 4)]
        loose = set()
        for _ in range(blocks):
            ends = []
            for _ in range(2):
                pick = rng.randrange(len(outs))
                loose.discard(pick)
                ends.append(e.chain(outs[pick], rng.choice((1, 3, 16, 16, 16, 4))))
            outs.append(e.node(*ends))
            loose.add(len(outs) - 1)
        before, last = last, e.node(*[outs[k] for k in sorted(loose)])


def _conv(e, rng, target):
    """Random convolutional cells of six to twelve nodes with one or two inputs each, until `target` nodes."""
    before = e.node()
    last = e.node(before)
    while e.n < target:
        pool, used = [last, before], {0, 1}
        for _ in range(rng.randint(6, 12)):
            picks = rng.sample(range(len(pool)), rng.randint(1, 2))
            used.update(picks)
            pool.append(e.node(*[pool[k] for k in picks]))
        before, last = last, e.node(*[v for k, v in enumerate(pool) if k not in used])


def _recurrent(e, rng, target):
    """One random recurrent cell unrolled 25 to 40 steps, about `target` nodes."""
    steps = rng.randint(25, 40)
    inside = max(2, round(target / steps) - 2)
    picks = [rng.randint(0, j) for j in range(inside - 1)]
    out = None
    for _ in range(steps):
        x = e.node()
        nodes = [e.node(x) if out is None else e.node(x, out)]
        for p in picks:
            nodes.append(e.node(nodes[p]))
        out = e.node(*[v for k, v in enumerate(nodes) if k not in picks])


@functools.lru_cache(maxsize=64)
def _graph(graph, size, graph_seed):
    e = _Edges()
    {"layered": _layered, "modules": _modules, "unrolled": _unrolled, "cells": _cells, "conv": _conv,
     "recurrent": _recurrent}[graph](e, random.Random(graph_seed), size)
    return e.n, np.asarray(e.src, dtype=np.int32), np.asarray(e.dst, dtype=np.int32)


def _shape(case):
    """Nodes and edges of a case's graph. Every recipe numbers its nodes in a topological order."""
    n, src, _ = _graph(case["graph"], case["size"], case["graph_seed"])
    return n, len(src)


# ------------------------------------------------------------------ inputs --

def _network(rng, sizes, final_act, scale=1.0):
    """Xavier-uniform weights W[in][out] and small biases of a one- or two-layer network, as placeto.Weights takes them."""
    net = {"n_layers": len(sizes) - 1, "in_dim": sizes[0], "hidden_dim": sizes[1], "out_dim": sizes[-1], "act": 0,
           "final_act": final_act, "W2": None, "b2": None}
    for k in range(len(sizes) - 1):
        bound = math.sqrt(6.0 / (sizes[k] + sizes[k + 1])) * (scale if k == len(sizes) - 2 else 1.0)
        net["W%d" % (k + 1)] = rng.uniform(-bound, bound, (sizes[k], sizes[k + 1])).astype(np.float32)
        net["b%d" % (k + 1)] = rng.uniform(-0.1, 0.1, sizes[k + 1]).astype(np.float32)
    return net


def _policy(rng, n, edges, d, m, layers):
    """All networks of a policy at the start of training. Messages are sums over a node's neighbours and the pooled sums
    grow with the graph; g and the output layer are scaled down by that, so that the embeddings neither grow nor vanish with
    the depth, the logits are of order one and the policy explores, as REINFORCE needs it to."""
    F = m + 4
    w = {"d": d, "F": F, "m": m}
    for way in ("down", "up"):
        w["f_" + way] = _network(rng, [d + F] + [d] * layers, 1)
        w["g_" + way] = _network(rng, [d] + [d] * layers, 1, min(1.0, n / max(edges, 1)))
    w["l"] = [_network(rng, [2 * d + F, d], 1) for _ in range(3)]
    w["h"] = [_network(rng, [d, d], 1) for _ in range(3)]
    z = 5 * d + F
    w["head"] = _network(rng, [z, z, m], 0, 8.0 / n)
    return w


def prepare(case, seed):
    path, d, m, batch = case["path"], case["d"], case["m"], case["batch"]
    n, src, dst = _graph(case["graph"], case["size"], case["graph_seed"])
    rng = np.random.default_rng(seed)
    gen = torch.Generator("cuda").manual_seed(seed)

    def on_gpu(a):
        return torch.from_numpy(a).cuda()

    # operation times ~ lognormal(0, 1) ms, output sizes ~ lognormal(10, 2) bytes, both relative to their mean
    cost, size = rng.lognormal(0.0, 1.0, n), rng.lognormal(10.0, 2.0, n)
    s = {"path": path, "m": m, "graph": placeto.Graph(n, src, dst),
         "cost": on_gpu((cost / cost.mean()).astype(np.float32)), "bytes": on_gpu((size / size.mean()).astype(np.float32)),
         "dev": torch.randint(0, m, (batch, n), dtype=torch.uint8, device="cuda", generator=gen)}
    if path == "simulate":
        # a bus moves the average tensor in the time of an average operation; memory for half of all outputs per device
        s.update(bandwidth=1.0, limit=0.5 * n, scale=2.0)
        return s
    weights = _policy(rng, n, len(src), d, m, case["layers"])
    s["weights"] = placeto.Weights(weights)
    g, w = s["graph"], s["weights"]
    if path == "rollout":
        s.update(order=torch.arange(n, dtype=torch.int32, device="cuda"), first=s["dev"].clone(),
                 uniforms=torch.rand((batch, n), device="cuda", generator=gen),
                 actions=torch.empty((batch, n), dtype=torch.uint8, device="cuda"),
                 logp=torch.empty((batch, n), device="cuda"), ws=placeto.workspace(g, w, batch, placeto.CALL_EPISODE))
        return s
    # states of episodes that visit the nodes in order: the nodes before the current one are placed
    s["cur"] = torch.randint(0, n, (batch,), dtype=torch.int32, device="cuda", generator=gen)
    s["placed"] = (torch.arange(n, device="cuda").view(1, n) < s["cur"].view(batch, 1)).to(torch.uint8)
    if path == "host":
        for k in ("cost", "bytes", "dev", "cur", "placed"):
            s[k] = s[k].cpu().pin_memory()
        s.update(logits=torch.empty((batch, m), pin_memory=True), probs=torch.empty((batch, m), pin_memory=True),
                 ws=placeto.workspace(g, w, batch, placeto.CALL_FORWARD_HOST))
        return s
    s.update(logits=torch.empty((batch, m), device="cuda"), probs=torch.empty((batch, m), device="cuda"))
    if path == "forward":
        s["ws"] = placeto.workspace(g, w, batch, placeto.CALL_FORWARD)
        return s
    s.update(X=torch.empty((n, batch, m + 4), device="cuda"), H_down=torch.empty((n, batch, d), device="cuda"),
             H_up=torch.empty((n, batch, d), device="cuda"), ws=placeto.workspace(g, w, batch, placeto.CALL_EMBED))
    if path == "embeddings":
        s["ws_logits"] = placeto.workspace(g, w, batch, placeto.CALL_LOGITS)
        return s
    s.update(actions=torch.randint(0, m, (batch,), dtype=torch.int32, device="cuda", generator=gen),
             advantages=torch.randn((batch,), device="cuda", generator=gen), grads=placeto.binding.zero_gradients(weights),
             ws_grad=placeto.workspace(g, w, batch, placeto.CALL_GRADIENT))
    return s


def run(s):
    path, g = s["path"], s["graph"]
    if path == "simulate":
        return placeto.placeto_simulate_placements(g, s["cost"], s["bytes"], s["dev"], s["m"], s["bandwidth"], s["limit"], s["scale"])
    w = s["weights"]
    if path == "forward":
        return placeto.placeto_policy_forward(g, w, s["cost"], s["bytes"], s["dev"], s["cur"], s["placed"], s["logits"], s["probs"], s["ws"])
    if path == "host":
        return placeto.placeto_policy_forward_host(g, w, s["cost"], s["bytes"], s["dev"], s["cur"], s["placed"], s["logits"], s["probs"], s["ws"])
    if path == "rollout":
        s["dev"].copy_(s["first"])       # the call leaves the final placement in place of the initial one
        return placeto.placeto_episode_rollout(g, w, s["cost"], s["bytes"], s["order"], s["dev"], s["uniforms"], s["actions"], s["logp"], s["ws"])
    X = placeto.placeto_build_features(g, s["cost"], s["bytes"], s["dev"], s["cur"], s["placed"], s["m"], s["X"])
    H_down, H_up = placeto.placeto_embed_forward(g, w, X, s["H_down"], s["H_up"], s["ws"])
    if path == "embeddings":
        logits, probs = placeto.placeto_policy_logits(g, w, X, H_down, H_up, s["cur"], s["logits"], s["probs"], s["ws_logits"])
        return X, H_down, H_up, logits, probs
    grads = placeto.placeto_policy_gradient(g, w, X, H_down, H_up, s["cur"], s["actions"], s["advantages"], 0.01, s["grads"], s["ws_grad"])
    return {"%s.%s.%s" % k: t for k, t in grads.tensors.items()}


# ---------------------------------------------------------------- the work --

def work(case):
    """Every input read once and every output written once; the arithmetic of the networks (a pooling network once per node
    and state), three times that with its gradient. A rollout evaluates the policy once per node."""
    path, d, m, batch, layers = (case[k] for k in ("path", "d", "m", "batch", "layers"))
    n, edges = _shape(case)
    F = m + 4
    z = 5 * d + F
    if path == "simulate":
        # an addition per operation and transfer, a comparison and a counter per edge
        return {"bytes": batch * (n + 8 * (m + 2)) + 8 * n + 4 * edges, "flops": batch * (2 * n + 3 * edges)}
    sweep = 2 * ((d + F) * d + d * d + (2 * d * d if layers == 2 else 0))
    weights = sweep + 3 * ((2 * d + F) * d + d * d) + z * z + z * m
    one = n * (2 * sweep + 2 * (2 * d + F) * d) + 2 * (3 * d * d + z * z + z * m)
    read = 8 * n + 4 * weights
    if path == "rollout":
        return {"bytes": read + batch * n * (1 + 1 + 1 + 4 + 4), "flops": batch * n * one}
    read += batch * (2 * n + 4)
    if path == "train":
        return {"bytes": read + batch * 8 + 4 * weights, "flops": 3 * batch * one}
    out = 8 * batch * m + (4 * batch * n * (F + 2 * d) if path == "embeddings" else 0)
    return {"bytes": read + out, "flops": batch * one}


def tolerance(case):
    """Four times what the outputs differ by from the same path in 64 bits, over the listed cases: 5e-7 for logits,
    probabilities and embeddings. A gradient also differs where rounding flips the sign of a pre-activation, whose ReLU then
    passes or stops that row's share: 5e-5 (single entries 8e-4) at d = 64. A rollout's choices differ only where a uniform
    number falls within rounding of an interval's boundary: at most a few of the 1e5 choices of the largest case, each of
    which changes that step's log-probability and hardly the steps after it. The simulator adds its doubles in a stated order."""
    if case["path"] == "simulate":
        return "exact"
    if case["path"] == "rollout":
        return {"rel": 5e-3, "max": 0.5, "differ": 1e-3}
    if case["path"] == "train":
        return {"rel": 2e-4, "max": 3e-3}
    return {"rel": 2e-6, "max": 2e-5}
