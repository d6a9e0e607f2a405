"""Buffers of a handle that has explored before, grown for a larger
exploration: whichever allocation fails, the call returns SNP_E_NOMEM or
succeeds, and the handle explores small and large afterwards as a fresh one."""
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu

SMALL, LARGE = (3, 100, 1000), (2, 1 << 17, 1 << 19)


@pytest.mark.parametrize("k", range(1, 19))
def test_failed_growth(gpu, k):
    system = snp_synth.random_system(881, 64, (2, 3), (4, 4), (0, 6), "sparse")
    o = oracle.Oracle(system)
    want = {x: o.explore(x[0], cap=x[1], budget=x[2]) for x in (SMALL, LARGE)}
    assert want[LARGE].depths[2].examined > 1 << 16  # a pass beyond the first buffers
    s = gpu.System(system)

    def explore(x, **more):
        s.explore(x[0], cap=x[1], budget=x[2], **more)
        got = s.reachable()
        assert got.shape == want[x].configs.shape and (got == want[x].configs).all()

    explore(SMALL)
    gpu.snp_debug_fail_allocation(k)
    try:
        s.explore(LARGE[0], cap=LARGE[1], budget=LARGE[2], record_parents=True)
    except gpu.SnpError as e:
        assert e.code == gpu.SNP_E_NOMEM
    finally:
        gpu.snp_debug_fail_allocation(0)
    explore(SMALL)
    explore(SMALL, chunk=64)
    explore(LARGE)
    explore(SMALL)
