"""snp_batch_autotune over the pass sizes of the engine."""
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [1 << 14, 5000])
def test_large_caps_take_the_engines_own_pass_size(gpu, cap):
    """With a cap several times 4096 a pass of 2 cap + 2048 candidates does
    what would be many smaller passes one after the other: the fastest setting
    by far, as fast as the automatic one."""
    systems = snp_synth.batch_systems(24)
    hs = [gpu.System(x) for x in systems]
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget = 6, cap, 16 * cap
    chunk, tile, warps = gpu.snp_batch_autotune([h.h for h in hs], o)
    assert chunk == min(2 * cap + 2048, 1 << 16) and tile in (8, 16, 32) and warps in (4, 8)
    assert (gpu.explore_batch(hs, 2, cap=cap, budget=16 * cap, chunk=chunk, tile=tile, warps=warps) == 0).all()
    for k in (0, 11):
        e = oracle.Oracle(systems[k]).explore(2, cap=cap, budget=16 * cap)
        got = hs[k].reachable()
        assert got.shape == e.configs.shape and (got == e.configs).all()


def test_tuning_a_batch_without_depths(gpu):
    systems = snp_synth.batch_systems(3)
    hs = [gpu.System(x) for x in systems]
    for t in (gpu.SNP_T_SPARSE_I32, gpu.SNP_T_TC_F8):
        o = gpu.snp_explore_opts_init()
        o.depth, o.frontier_cap, o.transition = 0, 100, t
        chunk, tile, warps = gpu.snp_batch_autotune([h.h for h in hs], o)
        assert chunk in (1024, 2048, 4096) and tile in (8, 16, 32) and warps in (4, 8)
