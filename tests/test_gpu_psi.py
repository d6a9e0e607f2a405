"""Psi, its prefix sums and the parents' records around the edges of their
tiles (8 rows by a warp each, 256 rows by a lane each; batches of 8 and 256
neurons) against the oracle, through whole explorations: frontiers of a few to
many rows, rows of any length, packed and not, counts beyond the direct table,
rows held back by max_expand."""
import numpy as np
import pytest

import oracle
import snp_synth


def check(s, e):
    got = s.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.candidates, d.truncated) for d in s.depth_stats()] == \
        [(d.new, d.examined, d.candidates, d.truncated) for d in e.depths]


@pytest.mark.gpu
@pytest.mark.parametrize("m", [1, 7, 8, 9, 31, 33, 64, 72, 100, 255, 256, 257, 520])
@pytest.mark.parametrize("cap", [7, 9, 255, 257, 600])
def test_frontiers_and_row_lengths(gpu, m, cap):
    system = snp_synth.random_system(300 + m, m, (1, 3), (min(2, m - 1), min(5, m - 1)), (0, 5), "sparse")
    e = oracle.Oracle(system).explore(3, cap=cap, budget=20 * cap)
    for packed in (False, True):
        s = gpu.System(system)
        s.explore(3, cap=cap, budget=20 * cap, packed=packed)
        check(s, e)


@pytest.mark.gpu
@pytest.mark.parametrize("m", [40, 130])
def test_counts_beyond_the_direct_table(gpu, m):
    system = snp_synth.random_system(8 + m, m, (1, 3), (3, 5), (0, 200), "sparse")
    for cap, top in ((300, -1), (300, 120)):
        e = oracle.Oracle(system).explore(3, cap=cap, budget=6000, max_expand=top)
        s = gpu.System(system)
        s.explore(3, cap=cap, budget=6000, max_expand=top)
        check(s, e)


@pytest.mark.gpu
@pytest.mark.parametrize("m", [16, 24])
def test_large_frontier_of_short_rows(gpu, m):
    """Tiles of 256 rows, more than 32 of them (look-back over two windows)."""
    system = snp_synth.random_system(71 + m, m, (2, 3), (4, 4), (0, 6), "sparse")
    e = oracle.Oracle(system).explore(5, cap=12000, budget=100000)
    s = gpu.System(system)
    s.explore(5, cap=12000, budget=100000)
    check(s, e)
    assert max(d.parents for d in s.depth_stats()) > 256 * 33


@pytest.mark.gpu
def test_rows_past_the_last_candidate_of_a_wide_frontier(gpu):
    """A frontier whose first 8192 rows hold 2^64 - 1 candidates: the other
    rows go in tiles of 8, more of them than the whole frontier has tiles.
    Against the allocation-free path, which evaluates every row."""
    import torch
    system = snp_synth.random_system(5, 512, (4, 4), (32, 32), (0, 16), "dense")
    depth, cap, budget = 3, 90112, 1 << 20
    s = gpu.System(system)
    s.explore(depth, cap=cap, budget=budget)
    assert s.depth_stats()[2].candidates == gpu.SNP_PSI_SAT and s.depth_stats()[3].parents == cap
    n = s.count()
    got = torch.zeros((n, 512), dtype=torch.int32, device="cuda")
    gpu.snp_reachable(s.h, got, n)
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget = depth, cap, budget
    out = torch.zeros((1 + depth * cap, 512), dtype=torch.int32, device="cuda")
    assert gpu.snp_explore_static(s.h, o, out, out.shape[0])[0] == n
    assert bool((out[:n] == got).all())
