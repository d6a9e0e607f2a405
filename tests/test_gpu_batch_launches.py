"""snp_depth_info.launches of a batch: depth 0 has the launches of the whole
call, the same for every system; the other depths have none."""
import pytest

import snp_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [0, 1, 4])
def test_launches_of_a_batch(gpu, depth):
    hs = [gpu.System(x) for x in snp_synth.batch_systems(8)]
    for t in (gpu.SNP_T_SPARSE_I32, gpu.SNP_T_TC_F8):
        for _ in range(2):
            assert (gpu.explore_batch(hs, depth, cap=200, budget=3000, transition=t) == 0).all()
            stats = [h.depth_stats() for h in hs]
            first = {s[0].launches for s in stats}
            assert len(first) == 1 and all(d.launches == 0 for s in stats for d in s[1:])
            n = first.pop()
            if t == gpu.SNP_T_TC_F8:  # table fill, C0 and a launch per depth
                assert n == depth + 2
            else:  # the same, and iterations of six launches: at least one pass per depth, two beyond the end
                passes = max(sum(d.chunks for d in s) for s in stats)
                assert (n - 2) % 6 == 0 and passes <= (n - 2) // 6 <= passes + 3
