"""Systems that advance together (batch engine and serving loop, sparse form)
against the oracle: rows of every expand form in one call (up to and beyond 128
neurons, whole 16-byte units and not), frontiers around the 32 rows and 8 rows
a work item holds, caps a pass overshoots, passes of the caller's size."""
import numpy as np
import pytest

import oracle
import snp_synth

MS = [1, 3, 16, 31, 64, 127, 128, 129, 131, 200, 300, 516]


def systems():
    return [snp_synth.random_system(900 + m, m, (1, 4), (min(2, m - 1), min(8, m - 1)), (0, 6), "sparse") for m in MS]


def same(h, x, depth, cap, budget):
    e = oracle.Oracle(x).explore(depth, cap=cap, budget=budget)
    got = h.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.candidates, d.truncated) for d in h.depth_stats()] == \
        [(d.new, d.examined, d.candidates, d.truncated) for d in e.depths]


@pytest.mark.gpu
@pytest.mark.parametrize("depth,cap,budget,chunk", [(4, 1, 0, 0), (4, 31, 500, 0), (3, 32, 0, 0), (4, 33, 3000, 0),
                                                    (3, 300, 5000, 0), (2, 5000, 40000, 0), (3, 300, 5000, 7)])
def test_batch_of_mixed_forms(gpu, depth, cap, budget, chunk):
    xs = systems()
    hs = [gpu.System(x) for x in xs]
    assert (gpu.explore_batch(hs, depth, cap=cap, budget=budget, chunk=chunk) == 0).all()
    for h, x in zip(hs, xs):
        same(h, x, depth, cap, budget)


@pytest.mark.gpu
def test_served_mixed_forms(gpu):
    xs = systems()
    hs = [gpu.System(x) for x in xs]
    srv = gpu.snp_server_create(1 << 30, 5)  # five at a time: requests join others half way
    try:
        for round_ in range(2):
            shapes = []
            for k, h in enumerate(hs):
                o = gpu.snp_explore_opts_init()
                o.depth, o.frontier_cap, o.candidate_budget = 2 + (k + round_) % 3, 33 + 100 * round_, 3000
                shapes.append((o.depth, o.frontier_cap, o.candidate_budget))
                gpu.snp_server_submit(srv, h.h, o)
            gpu.snp_server_wait(srv)
            assert (gpu.snp_server_poll(srv)[2] == 0).all()
            for h, x, s in zip(hs, xs, shapes):
                same(h, x, *s)
    finally:
        gpu.snp_server_destroy(srv)
