"""The batch engine's memory.  Where it runs short, whichever allocation
fails, the call either serves every system (in smaller groups and passes) and
leaves no message, or returns SNP_E_NOMEM and works the next time; and what
it keeps beside the results is bounded."""
import numpy as np
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", range(1, 10))
def test_failed_allocation(gpu, k):
    systems = snp_synth.batch_systems(6)
    hs = [gpu.System(x) for x in systems]
    gpu.snp_debug_fail_allocation(k)
    try:
        o = gpu.snp_explore_opts_init()
        o.depth, o.frontier_cap, o.candidate_budget = 3, 300, 5000
        status = np.full(len(hs), -1, dtype=np.int32)
        gpu.snp_explore_batch([h.h for h in hs], o, status)
        assert gpu.snp_last_error() == ""
        assert (status == 0).all()
    except gpu.SnpError as e:
        assert e.code == gpu.SNP_E_NOMEM
        gpu.snp_debug_fail_allocation(0)
        assert (gpu.explore_batch(hs, 3, cap=300, budget=5000) == 0).all()
    finally:
        gpu.snp_debug_fail_allocation(0)
    for h, x in zip(hs, systems):
        e = oracle.Oracle(x).explore(3, cap=300, budget=5000)
        got = h.reachable()
        assert got.shape == e.configs.shape and (got == e.configs).all()


def test_scratch_kept_with_the_results(gpu):
    """24 systems of 1024 neurons with cap 2^15 take 6.5 GB of scratch while
    they run; at most 4 GiB stay beside the pools (3.2 GB) and tables."""
    import torch
    systems = [snp_synth.random_system(8700 + k, 1024, (2, 3), (4, 4), (0, 6), "sparse") for k in range(24)]
    hs = [gpu.System(x) for x in systems]
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        assert (gpu.explore_batch(hs, 1, cap=1 << 15, budget=100) == 0).all()
        held = before - torch.cuda.mem_get_info()[0]
        pools = 24 * ((1 << 15) + 1) * 4096
        assert held <= pools + (4 << 30) + (64 << 20), held
        for k in (0, 23):
            e = oracle.Oracle(systems[k]).explore(1, cap=1 << 15, budget=100)
            got = hs[k].reachable()
            assert got.shape == e.configs.shape and (got == e.configs).all()
