"""GPU parity of placeto_policy_gradient against the CPU checker (PyTorch fp64
reverse-mode differentiation of the restated forward, pinned to the C checker).
Every gradient array must agree normwise: max |gpu - ref| <= TOL * max |ref| of
that array (fp32 sums over up to n * B rows; the forward's own normwise
tolerance is 2e-5 per row)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_1906_08879_b200 as placeto
from gen import configs, states
from oracle import gradient
from tests.helpers import random_dag, rng

pytestmark = pytest.mark.gpu

TOL = 2e-4


def dev_t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def gpu_gradient(cfg, actions, adv, beta):
    g = placeto.Graph(cfg["n"], cfg["src"], cfg["dst"])
    w = placeto.Weights(cfg["weights"])
    cur = dev_t(cfg["cur"])
    X = placeto.placeto_build_features(g, dev_t(cfg["cost"]), dev_t(cfg["bytes"]), dev_t(cfg["dev"]),
                                       cur, dev_t(cfg["placed"]), cfg["m"])
    Hd, Hu = placeto.placeto_embed_forward(g, w, X)
    grads = placeto.binding.zero_gradients(cfg["weights"])
    placeto.placeto_policy_gradient(g, w, X, Hd, Hu, cur, dev_t(actions.astype(np.int32)),
                                    dev_t(adv.astype(np.float32)), beta, grads)
    torch.cuda.synchronize()
    return grads


def compare(cfg, grads, ref):
    worst = 0.0
    for (name, idx, key), t in grads.tensors.items():
        want = ref[name][key] if idx is None else ref[name][idx][key]
        got = t.cpu().numpy().astype(np.float64)
        assert got.shape == want.shape and np.isfinite(got).all(), (name, idx, key)
        scale = np.abs(want).max()
        err = np.abs(got - want).max()
        assert err <= TOL * max(scale, 1e-6), "%s[%s].%s: error %.3g against scale %.3g" % (name, idx, key, err, scale)
        worst = max(worst, err / max(scale, 1e-30))
    return worst


def small_case(seed, n, m, d, B, p=0.2):
    r = rng(seed)
    src, dst = random_dag(r, n, p)
    cfg = {"n": n, "src": src, "dst": dst, "m": m, "d": d, "F": m + 4}
    cfg["cost"], cfg["bytes"] = states.node_costs(r, n, normalise=True)
    cfg["dev"], cfg["cur"], cfg["placed"] = states.random_states(r, n, m, B)
    cfg["weights"] = states.policy_weights(r, d, m + 4, m, 2, 0, 0.2)
    return cfg, r.integers(0, m, B), r.normal(size=B)


@pytest.mark.parametrize("d,m,B,beta", [(4, 3, 5, 0.0), (8, 2, 33, 0.5), (32, 4, 20, 0.1), (64, 8, 9, 0.0)])
def test_small_graphs(d, m, B, beta):
    cfg, actions, adv = small_case(10 * d + m, n=18, m=m, d=d, B=B)
    adv32 = adv.astype(np.float32).astype(np.float64)
    grads = gpu_gradient(cfg, actions, adv32, beta)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv32, beta))


def test_degenerate_graphs_and_entropy_only():
    e = np.zeros(0, np.int32)
    for n, src, dst in ((1, e, e), (4, e, e), (6, np.arange(5, dtype=np.int32), np.arange(1, 6, dtype=np.int32))):
        r = rng(n)
        m, d, B = 3, 8, 6
        cfg = {"n": n, "src": src, "dst": dst, "m": m, "d": d, "F": m + 4}
        cfg["cost"], cfg["bytes"] = states.node_costs(r, n, normalise=True)
        cfg["dev"], cfg["cur"], cfg["placed"] = states.random_states(r, n, m, B)
        cfg["weights"] = states.policy_weights(r, d, m + 4, m, 2, 0, 0.2)
        actions = r.integers(0, m, B)
        zero = np.zeros(B)
        grads = gpu_gradient(cfg, actions, zero, 1.0)
        compare(cfg, grads, gradient.gradient(cfg, actions, zero, 1.0))


def test_inception_shaped_graph():
    cfg = configs.make("inception", B=12, normalise=True)
    r = rng(4)
    actions = r.integers(0, cfg["m"], 12)
    adv = r.normal(size=12).astype(np.float32).astype(np.float64)
    grads = gpu_gradient(cfg, actions, adv, 0.05)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.05))


def test_accumulating_over_two_halves_of_the_batch():
    cfg, actions, adv = small_case(12, n=16, m=4, d=32, B=24)
    adv = adv.astype(np.float32).astype(np.float64)
    g = placeto.Graph(cfg["n"], cfg["src"], cfg["dst"])
    w = placeto.Weights(cfg["weights"])
    grads = placeto.binding.zero_gradients(cfg["weights"])
    for k, sel in enumerate((slice(0, 10), slice(10, 24))):
        cur = dev_t(cfg["cur"][sel])
        X = placeto.placeto_build_features(g, dev_t(cfg["cost"]), dev_t(cfg["bytes"]), dev_t(cfg["dev"][sel]),
                                           cur, dev_t(cfg["placed"][sel]), cfg["m"])
        Hd, Hu = placeto.placeto_embed_forward(g, w, X)
        placeto.placeto_policy_gradient(g, w, X, Hd, Hu, cur, dev_t(actions[sel].astype(np.int32)),
                                        dev_t(adv[sel].astype(np.float32)), 0.2, grads, accumulate=k > 0)
    torch.cuda.synchronize()
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.2))


def test_reproducible_and_unsupported_shapes():
    cfg, actions, adv = small_case(3, n=14, m=4, d=32, B=17)
    a = gpu_gradient(cfg, actions, adv, 0.1)
    b = gpu_gradient(cfg, actions, adv, 0.1)
    for key, t in a.tensors.items():
        assert torch.equal(t, b.tensors[key]), key
    # identity activations are not differentiated
    r = rng(6)
    cfg["weights"] = states.policy_weights(r, 32, 8, 4, 2, 1, 0.2)
    with pytest.raises(placeto.PlacetoError) as e:
        gpu_gradient(cfg, actions, adv, 0.0)
    assert e.value.status == 4


@pytest.mark.parametrize("d,m", [(8, 3), (32, 4)])
def test_single_layer_networks_as_in_the_paper(d, m):
    """Appendix A.7: f and g are single layers. Every gradient array against the checker."""
    cfg, actions, adv = small_case(21 + d, n=15, m=m, d=d, B=19)
    r = rng(d)
    cfg["weights"] = states.policy_weights(r, d, m + 4, m, 1, 0, 0.2)
    grads = gpu_gradient(cfg, actions, adv, 0.05)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.05))


@pytest.mark.parametrize("d,m,B,layers", [(32, 4, 1, 2), (32, 2, 160, 2), (32, 12, 75, 1), (64, 3, 1, 2), (64, 8, 155, 2), (64, 5, 76, 1)])
def test_split_sweep_over_tiles(d, m, B, layers):
    """The tensor-core reverse sweep: one state per block, levels of one partial tile and of more tiles than groups of
    warps, a ragged last slice, nodes of many consumers, feature widths that are no multiple of 4."""
    cfg, actions, adv = small_case(7 * d + B, n=33, m=m, d=d, B=B, p=0.12)
    r = rng(B)
    cfg["weights"] = states.policy_weights(r, d, m + 4, m, layers, 0, 0.2)
    adv = adv.astype(np.float32).astype(np.float64)
    grads = gpu_gradient(cfg, actions, adv, 0.1)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.1))


@pytest.mark.parametrize("d,m,n,B", [(32, 3, 150, 2), (64, 8, 140, 3), (64, 4, 300, 1)])
def test_pooling_passes_over_chunks_of_nodes(d, m, n, B):
    """More chunks of nodes than one (few states), sets of fewer rows than a warp's batch and of many batches, states
    whose current node lies in each chunk."""
    cfg, actions, adv = small_case(d + n, n=n, m=m, d=d, B=B, p=0.02)
    cfg["cur"] = np.linspace(0, n - 1, B).astype(np.int32)
    adv = adv.astype(np.float32).astype(np.float64)
    grads = gpu_gradient(cfg, actions, adv, 0.1)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.1))


@pytest.mark.parametrize("d,m,n,B", [(32, 4, 3, 52500), (64, 5, 4, 1025), (32, 2, 5, 2079)])
def test_pooling_weights_of_large_batches(d, m, n, B):
    """The rows of a node are listed a part of the batch at a time: more states than a list in shared memory could hold,
    parts of one state, remainders of a stage carried from part to part and from node to node."""
    cfg, actions, adv = small_case(n + B, n=n, m=m, d=d, B=B, p=0.7)
    adv = adv.astype(np.float32).astype(np.float64)
    grads = gpu_gradient(cfg, actions, adv, 0.1)
    compare(cfg, grads, gradient.gradient(cfg, actions, adv, 0.1))


def cancelling(W, rows):
    """The first `rows` rows of W, the second half of them the first negated: over inputs whose halves agree the exact sum is
    zero, and what a kernel finds is what its order of summation leaves."""
    W = W.copy()
    W[rows // 2:rows] = -W[:rows // 2]
    W[rows:] = 0
    return W


@pytest.mark.parametrize("nets", ["g", "f and l"])
@pytest.mark.parametrize("d,m,n,B,p", [(32, 4, 60, 303, 0.05), (32, 3, 25, 1200, 0.15), (32, 4, 12, 1, 0.3), (64, 8, 40, 155, 0.06), (64, 3, 70, 500, 0.03)])
def test_masks_are_those_of_the_general_kernels(d, m, n, B, p, nets):
    """A ReLU's mask is the sign of a recomputed sum, so the kernels for d = 32 and 64 add up in the order of the general
    ones. Here the sums before the first ReLU of g (of f and l_i) are nothing but rounding; one hidden unit of weight zero more
    in f sends the same problem to the general kernels. One mask that differs moves an array by 1e-3 of its norm and more;
    without, sums of at most n B = 35,000 terms and a few levels differ by rounding, 1e-6 (bound: 2e-5). Levels of one
    row up to more than a pass of 64, last passes short and long, ragged last slices."""
    cfg, actions, adv = small_case(d + n, n=n, m=m, d=d, B=B, p=p)
    r = rng(d + B)
    half = r.uniform(0.1, 1.0, (2, n, B, d // 2)).astype(np.float32)
    H = np.concatenate([half, half], axis=-1)
    w = cfg["weights"]
    for way in ("down", "up"):
        f, g = w["f_" + way], w["g_" + way]
        if nets == "g":
            g["W1"], g["b1"] = cancelling(g["W1"], d), np.zeros(d, np.float32)
            f["W2"][:, d // 2:], f["b2"][d // 2:] = f["W2"][:, :d // 2], f["b2"][:d // 2]      # messages: two equal halves
        else:
            f["W1"], f["b1"] = cancelling(f["W1"], d), np.zeros(d, np.float32)
    for l in w["l"] if nets != "g" else []:
        l["W1"][:d], l["W1"][d:2 * d] = cancelling(l["W1"][:d], d), cancelling(l["W1"][d:2 * d], d)
        l["W1"][2 * d:], l["b1"] = 0, np.zeros(d, np.float32)

    def gradient_of(weights):
        graph = placeto.Graph(cfg["n"], cfg["src"], cfg["dst"])
        cur = dev_t(cfg["cur"])
        X = placeto.placeto_build_features(graph, dev_t(cfg["cost"]), dev_t(cfg["bytes"]), dev_t(cfg["dev"]), cur,
                                           dev_t(cfg["placed"]), m)
        grads = placeto.binding.zero_gradients(weights)
        placeto.placeto_policy_gradient(graph, placeto.Weights(weights), X, dev_t(H[0]), dev_t(H[1]), cur,
                                        dev_t(actions.astype(np.int32)), dev_t(adv.astype(np.float32)), 0.1, grads)
        return {k: t.cpu().numpy().astype(np.float64) for k, t in grads.tensors.items()}

    got = gradient_of(w)
    f = w["f_down"]
    wider = dict(f, hidden_dim=d + 1, W1=np.pad(f["W1"], ((0, 0), (0, 1))), b1=np.pad(f["b1"], (0, 1)), W2=np.pad(f["W2"], ((0, 1), (0, 0))))
    want = gradient_of(dict(w, f_down=wider))
    for (name, idx, key), a in got.items():
        if nets == "g" and name in ("f_down", "f_up") and key in ("W1", "b1"):
            continue               # equal halves of messages, negated halves of g's weights: f's hidden layer has no gradient but rounding
        b = want[name, idx, key][tuple(slice(0, k) for k in a.shape)]
        assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b), (name, idx, key, np.linalg.norm(a - b), np.linalg.norm(b))
