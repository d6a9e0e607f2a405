"""Marks, ranks and commit of a pass around the edges of its tiles (2048
candidates and more; up to and beyond 32 of them) against the oracle:
rows of any length, with and without a map to discovery order, parent records."""
import numpy as np
import pytest

import oracle
import snp_synth

PASSES = [31, 32, 33, 2047, 2048, 2049, 2048 * 33, 2048 * 40 + 17]


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", PASSES)
@pytest.mark.parametrize("m", [61, 64])
def test_ranks_and_parent_records(gpu, m, chunk):
    system = snp_synth.random_system(40 + m, m, (2, 3), (4, 4), (0, 6), "sparse")
    depth, cap, budget = 3, 5000, 120000
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    s = gpu.System(system)
    s.explore(depth, cap=cap, budget=budget, chunk=chunk, record_parents=True)
    got = s.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.truncated) for d in s.depth_stats()] == [(d.new, d.examined, d.truncated) for d in e.depths]
    par, idx = s.parents()
    o = oracle.Oracle(system)
    for k in np.linspace(1, len(got) - 1, 40).astype(int):
        assert (o.step(got[par[k]], cap=int(idx[k]) + 1)[int(idx[k])] == got[k]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", PASSES)
@pytest.mark.parametrize("m", [5, 61, 200])
def test_staged_rows(gpu, m, chunk):
    import torch
    system = snp_synth.random_system(50 + m, m, (2, 3), (min(4, m - 1), min(4, m - 1)), (0, 6), "sparse")
    depth, cap, budget = 3, 4000, 100000
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    s = gpu.System(system)
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget, o.chunk = depth, cap, budget, chunk
    out = torch.zeros((1 + depth * cap, m), dtype=torch.int32, device="cuda")
    n, reached = gpu.snp_explore_static(s.h, o, out, out.shape[0])
    assert n == len(e.configs) and reached == e.depth_reached
    assert (out[:n].cpu().numpy() == e.configs).all()
