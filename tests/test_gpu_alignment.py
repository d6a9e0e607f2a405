"""Device buffers of the caller that start off a 16-byte boundary, with rows
that are whole 16-byte units (so that the vector forms would be chosen by the
row length alone).  Results are whole numbers and compared exactly."""
import ctypes

import numpy as np
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu

MARK = -7


def shifted(rows: int, m: int, shift: int):
    """A marked buffer and its part of rows x m counts that starts `shift` counts in."""
    import torch
    buf = torch.full((rows * m + 8,), MARK, dtype=torch.int32, device="cuda")
    assert buf.data_ptr() % 16 == 0
    return buf, buf[shift:shift + rows * m].view(rows, m)


def check(buf, shift: int, want):
    got = buf.cpu().numpy()
    n = want.size
    assert (got[shift:shift + n] == want.reshape(-1)).all()
    assert (got[:shift] == MARK).all() and (got[shift + n:] == MARK).all()


def system_of(m: int, top: int = 6):
    return snp_synth.random_system(330 + m, m, (1, 3), (min(4, m - 1), min(4, m - 1)), (0, top), "sparse")


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("m,top,packed,width", [(4, 6, False, 4), (64, 6, False, 4), (61, 6, False, 4),
                                                (388, 6, False, 4), (64, 6, True, 1), (24, 6, True, 2),
                                                (400, 6, True, 1), (392, 300, True, 2)])
def test_reachable_into_a_shifted_buffer(gpu, m, top, packed, width, shift):
    system = system_of(m, top)
    s = gpu.System(system)
    s.explore(3, cap=300, budget=3000, packed=packed)
    assert s.row_width() == width
    want = oracle.Oracle(system).explore(3, cap=300, budget=3000).configs
    buf, out = shifted(len(want), m, shift)
    assert gpu.snp_reachable(s.h, out, len(want)) == len(want)
    check(buf, shift, want)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("m,depth,cap,budget", [(4, 4, 60, 0), (64, 3, 300, 3000), (61, 3, 300, 3000),
                                                (128, 3, 2000, 40000), (132, 3, 500, 9000), (1024, 2, 200, 3000)])
def test_static_into_a_shifted_buffer(gpu, m, depth, cap, budget, shift):
    system = system_of(m)
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    s = gpu.System(system)
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget = depth, cap, budget
    buf, out = shifted(1 + depth * cap, m, shift)
    n, reached = gpu.snp_explore_static(s.h, o, out, out.shape[0])
    assert n == len(e.configs) and reached == e.depth_reached
    check(buf, shift, e.configs)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("m,top,packed,width", [(64, 6, True, 1), (24, 6, True, 2), (392, 300, True, 2),
                                                (64, 6, False, 4)])
def test_resume_from_a_shifted_buffer(gpu, m, top, packed, width, shift):
    import torch
    system = system_of(m, top)
    s = gpu.System(system)
    s.explore(2, cap=300, budget=3000)
    rows, raw = s.checkpoint()
    buf, dev = shifted(len(rows), m, shift)
    dev.copy_(torch.from_numpy(rows))
    k = raw.nbytes // ctypes.sizeof(gpu.snp_depth_info)
    stats = (gpu.snp_depth_info * k).from_buffer_copy(raw.tobytes())
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget, o.packed = 4, 300, 3000, 1 if packed else 0
    later = gpu.System(system)
    later.depth_reached = gpu.snp_explore_resume(later.h, dev, stats, o)
    assert later.row_width() == width
    e = oracle.Oracle(system).explore(4, cap=300, budget=3000)
    got = later.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    check(buf, shift, rows)
