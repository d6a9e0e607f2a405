"""snp_step's kernels against the oracle, bit for bit: rows that are and are not
whole 16-byte units, output rows that start off a 16-byte boundary, runs of
one child and of many per warp, more children than the buffer takes."""
import numpy as np
import pytest

import oracle
import snp_synth


@pytest.mark.gpu
@pytest.mark.parametrize("m,rules,deg,mode", [(1, (1, 3), (0, 0), "sparse"), (3, (2, 3), (2, 2), "sparse"),
                                              (31, (2, 3), (4, 4), "sparse"), (64, (1, 4), (2, 8), "sparse"),
                                              (129, (4, 4), (16, 16), "dense"), (301, (2, 3), (4, 4), "sparse"),
                                              (1024, (4, 4), (64, 64), "dense")])
@pytest.mark.parametrize("capacity", [1, 33, 6001])
@pytest.mark.parametrize("shift", [0, 1])
def test_step_children_match_the_oracle(gpu, m, rules, deg, mode, capacity, shift):
    import paper_1104_1824_gb300 as snp
    import torch
    system = snp_synth.random_system(77 + m, m, rules, deg, (0, 6), mode)
    o = oracle.Oracle(system)
    s = snp.System(system)
    want = o.step(system.c0, cap=capacity)
    buf = torch.full((capacity * m + 2,), -7, dtype=torch.int32, device="cuda")
    psi = snp.snp_step(s.h, system.c0, capacity, buf[shift:])
    got = buf.cpu().numpy()
    n = min(psi, capacity)
    assert n == len(want)
    assert (got[shift:shift + n * m].reshape(n, m) == want).all()
    assert (got[:shift] == -7).all() and (got[shift + n * m:] == -7).all()
    host, psi_host = s.step(system.c0, capacity)
    assert psi_host == psi and (host == want).all()
    dev = torch.from_numpy(np.ascontiguousarray(system.c0)).cuda()
    assert snp.snp_step(s.h, dev, 0, None) == psi


@pytest.mark.gpu
@pytest.mark.parametrize("pin", [True, False])
def test_step_waits_for_copies_into_its_row(gpu, pin):
    """C in host memory, pinned or not, that a copy on the default stream is
    still writing when snp_step is called: the step is of the copied row."""
    import torch
    system = snp_synth.random_system(78, 64, (2, 3), (4, 4), (0, 6), "sparse")
    s = gpu.System(system)
    o = oracle.Oracle(system)
    later = (np.asarray(system.c0) + 1).astype(np.int32)
    want = o.step(later, cap=500)
    host = torch.from_numpy(np.array(system.c0, dtype=np.int32))
    if pin:
        host = host.pin_memory()
    dev = torch.from_numpy(later).cuda()
    out = np.zeros((500, 64), dtype=np.int32)
    gpu.snp_step(s.h, host, 500, out)  # loads the kernels
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)  # about 0.1 s
    host.copy_(dev, non_blocking=True)
    psi = gpu.snp_step(s.h, host, 500, out)
    assert min(psi, 500) == len(want)
    assert (out[:len(want)] == want).all()
