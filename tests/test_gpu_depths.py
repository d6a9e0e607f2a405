"""Depths that run without the host, further cases: passes of the caller's
size, a frontier that outgrows the buffers it was given, a flag that cancels
while depths are enqueued ahead."""
import threading

import numpy as np
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu


def check(s, e):
    got = s.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.candidates, d.truncated) for d in s.depth_stats()] == \
        [(d.new, d.examined, d.candidates, d.truncated) for d in e.depths]


@pytest.mark.parametrize("m", [24, 150])
@pytest.mark.parametrize("cap,budget", [(0, 9000), (0, 30000), (300, 30000)])
@pytest.mark.parametrize("chunk", [500, 6000, 16384, 1 << 17])
def test_passes_of_the_callers_size(gpu, m, cap, budget, chunk):
    """chunk candidates per pass: a depth that examines x of them takes
    ceil(x / chunk) passes."""
    system = snp_synth.random_system(830 + m, m, (2, 3), (3, 5), (0, 6), "sparse")
    depth = 4
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    s = gpu.System(system)
    for _ in range(2):
        s.explore(depth, cap=cap, budget=budget, chunk=chunk)
        check(s, e)
        for d, x in enumerate(s.depth_stats()[1:], 1):
            assert x.chunks == -(-x.examined // chunk), (d, x.examined, x.chunks)


def widening(idle: int):
    """T = 1024, 1024, 8192, 8192, ... candidates at depths 1, 2, 3, 4, ...,
    all children distinct until a pair that passes one spike to and fro comes
    round again.  Ten neurons choose at the first step (2 spikes: consume both
    or one), three more at the third (their second spike comes down a chain of
    two neurons); `idle` neurons without rules make the rows longer."""
    two = lambda n: [(n, 2, 0, 2, 0), (n, 2, 0, 1, 0)]
    rules = [r for n in range(10) for r in two(n)]
    rules += [(10, 1, 0, 1, 1), (11, 1, 0, 1, 1)]
    rules += [r for n in (12, 13, 14) for r in two(n)]
    rules += [(15, 1, 0, 1, 1), (16, 1, 0, 1, 1)]
    targets = [[] for _ in range(10)] + [[11], [12, 13, 14]] + [[], [], []] + [[16], [15]] + [[] for _ in range(idle)]
    c0 = [2] * 10 + [1, 0] + [1] * 3 + [1, 0] + [0] * idle
    rn, i, j, c, p = zip(*rules)
    return snp_synth.make_system(17 + idle, rn, i, j, c, p, targets, c0)


@pytest.mark.parametrize("idle,packed", [(0, False), (7, False), (15, True), (120, False)])
def test_frontier_that_outgrows_its_buffers(gpu, idle, packed):
    """Uncapped: a depth enqueued ahead has buffers for 4096 frontier rows and
    the depth before it finds 8192; the host takes over with it in flight."""
    system = widening(idle)
    e = oracle.Oracle(system).explore(6)
    assert [d.new for d in e.depths[1:5]] == [1024, 1024, 8192, 8192]
    s = gpu.System(system)
    for _ in range(3):  # fresh buffers, then kept ones
        s.explore(6, packed=packed, record_parents=not packed)
        check(s, e)


def test_cancelled_between_depths(gpu):
    """A long chain of small depths (a system that counts up for ever) with a
    flag set while it runs: cancelled, the result discarded, the handle usable."""
    # two neurons that pass their spikes on and gain one each step
    system = snp_synth.make_system(3, [0, 1], [1, 1], [1, 1], [1, 1], [1, 1], [[1, 2], [0, 2], []], [1, 1, 0])
    s = gpu.System(system)
    flag = np.zeros(1, dtype=np.int32)
    timer = threading.Timer(0.1, lambda: flag.__setitem__(0, 1))
    timer.start()
    try:
        with pytest.raises(gpu.SnpError) as ei:
            s.explore(1_000_000, cancel=flag)
        assert ei.value.code == gpu.SNP_E_CANCELLED
    finally:
        timer.cancel()
    with pytest.raises(gpu.SnpError) as ei:
        s.reachable()
    assert ei.value.code == gpu.SNP_E_STATE
    for depth in (1, 2, 37):
        s.explore(depth)
        check(s, oracle.Oracle(system).explore(depth))
