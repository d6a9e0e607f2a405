"""The int8 tensor-core form at the edges of its tiles (64 candidates x 64
columns per warp, pairs of 32-rule blocks) with entries up to +-127 that add up
in one column, against the oracle."""
import numpy as np
import pytest

import oracle
import snp_synth


def heavy(m, rules, seed):
    """Every neuron sends up to 127 spikes to neurons 0 and m // 2 (and its neighbour)."""
    rng = np.random.default_rng(seed)
    rn = np.repeat(np.arange(m), rules)
    c = rng.integers(1, 128, size=rn.size)
    p = rng.integers(100, 128, size=rn.size)
    targets = [sorted({t for t in (0, m // 2, (n + 1) % m) if t != n}) for n in range(m)]
    return snp_synth.make_system(m, rn, c, np.ones_like(c), c, p, targets, rng.integers(100, 300, size=m))


@pytest.mark.gpu
@pytest.mark.parametrize("m,rules", [(2, 1), (7, 3), (63, 2), (64, 1), (65, 4), (128, 2), (129, 3), (257, 2), (1000, 4)])
@pytest.mark.parametrize("cap,budget,chunk", [(100, 400, 0), (70, 200, 65), (40, 200, 1)])
def test_int8_tiles(gpu, m, rules, cap, budget, chunk):
    system = heavy(m, rules, 10 * m + rules)
    e = oracle.Oracle(system).explore(3, cap=cap, budget=budget)
    s = gpu.System(system)
    s.explore(3, cap=cap, budget=budget, chunk=chunk, transition=gpu.SNP_T_TC_I8)
    got = s.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.truncated) for d in s.depth_stats()] == [(d.new, d.examined, d.truncated) for d in e.depths]
