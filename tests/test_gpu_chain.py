"""Depths that run without the host (small passes enqueued ahead) against the
oracle: depths that take one pass and ones that take more, frontiers that
outgrow the buffers, explorations that end early, with parent records, packed
rows, resumed, cancelled and failing half way."""
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
@pytest.mark.parametrize("m", [5, 33, 64, 150])
@pytest.mark.parametrize("cap,budget", [(1, 0), (50, 0), (700, 4000), (700, 100000), (6000, 30000), (0, 3000)])
def test_capped_and_uncapped_depths(gpu, m, cap, budget):
    system = snp_synth.random_system(610 + m, m, (1, 3), (min(3, m - 1), min(5, m - 1)), (0, 5), "sparse")
    depth = 4 if cap == 0 or cap > 1000 else 7
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    for packed in (False, True):
        s = gpu.System(system)
        for _ in range(2):  # fresh buffers, then kept ones
            s.explore(depth, cap=cap, budget=budget, packed=packed, record_parents=not packed)
            check(s, e)
    o = oracle.Oracle(system)
    s = gpu.System(system)
    s.explore(depth, cap=cap, budget=budget, record_parents=True)
    rows, (par, idx) = s.reachable(), s.parents()
    for k in np.linspace(1, len(rows) - 1, min(30, max(len(rows) - 1, 0))).astype(int):
        assert (o.step(rows[par[k]], cap=int(idx[k]) + 1)[int(idx[k])] == rows[k]).all()
    s.explore(2, cap=cap, budget=budget)
    cp = s.checkpoint()
    later = gpu.System(system)
    later.resume(cp, depth, cap=cap, budget=budget)
    check(later, e)


@pytest.mark.gpu
def test_overflow_half_way(gpu):
    """A column that leaves the int32 range's safe part after some depths."""
    big = 2 ** 31 - 1 - 1000
    system = snp_synth.make_system(2, [0, 1], [1, 1], [1, 1], [1, 1], [300, 1], [[1], [0]], [50, big])
    s = gpu.System(system)
    with pytest.raises(gpu.SnpError) as ei:
        s.explore(20)
    assert ei.value.code == gpu.SNP_E_OVERFLOW
    s.explore(2)
    check(s, oracle.Oracle(system).explore(2))


@pytest.mark.gpu
def test_tree_that_ends(gpu):
    system = snp_synth.paper_example(exact=True)
    s = gpu.System(system)
    for _ in range(3):
        s.explore(100)
        check(s, oracle.Oracle(system).explore(100))
