"""Two host threads, each with its own stream and buffers, on a small and a large graph: a kernel's shared-memory limit belongs to
the process, so a call must not lower it under the other thread's launch."""
from __future__ import annotations

import threading

import numpy as np
import pytest
import torch

import paper_1906_08879_b200 as placeto
from gen import graphs, states
from tests.helpers import rng

pytestmark = pytest.mark.gpu


def _work(levels, P, times, errors):
    try:
        r = rng(levels)
        n, src, dst = graphs.layered_dag(seed=levels, levels=levels, width=5)
        g = placeto.Graph(n, src, dst)
        w = placeto.Weights(states.policy_weights(r, 32, 8, 4, 2, 0, 0.1))
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        cost, size = [t(a) for a in states.node_costs(r, n, True)]
        dev = t(r.integers(0, 4, (P, n)).astype(np.uint8))
        X = torch.rand((n, P, 8), device="cuda")
        ws = placeto.workspace(g, w, P, placeto.CALL_EMBED)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            first = None
            for _ in range(times):
                out = list(placeto.placeto_simulate_placements(g, cost, size, dev, 4, 1.0, 1.0, 1.0)) + list(placeto.placeto_embed_forward(g, w, X, ws=ws))
                stream.synchronize()
                if first is None:
                    first = [o.clone() for o in out]
                assert all(torch.equal(a, b) for a, b in zip(out, first))
    except Exception as e:      # noqa: BLE001 (reported by the test's own thread)
        errors.append(repr(e))


def test_small_and_large_graphs_from_two_threads():
    errors: list = []
    threads = [threading.Thread(target=_work, args=(levels, P, 400, errors)) for levels, P in ((4, 64), (60, 300))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
