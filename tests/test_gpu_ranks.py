"""Marks, ranks and commit at the edges of the kernels that do them: passes
around 256 candidates (a commit tile), around 4096 (up to there one CTA does
all of it) and around 2^19 (from there on tiles grow), and passes beyond 2^22
candidates, whose tiles take several rounds of 64 bitmap words."""
import numpy as np
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [255, 256, 257, 4095, 4096, 4097])
@pytest.mark.parametrize("m", [61, 64])
def test_small_passes(gpu, m, chunk):
    system = snp_synth.random_system(870 + m, m, (2, 3), (4, 4), (0, 6), "sparse")
    depth, cap, budget = 3, 5000, 30000
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    s = gpu.System(system)
    s.explore(depth, cap=cap, budget=budget, chunk=chunk, record_parents=True)
    got = s.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.truncated) for d in s.depth_stats()] == [(d.new, d.examined, d.truncated) for d in e.depths]
    par, idx = s.parents()
    o = oracle.Oracle(system)
    for k in np.linspace(1, len(got) - 1, 40).astype(int):
        assert (o.step(got[par[k]], cap=int(idx[k]) + 1)[int(idx[k])] == got[k]).all()


def choosers(bits: int):
    """bits + 1 neurons of 2 spikes that each keep none (consume 2) or one
    (consume 1); the last one has the second of these rules twice, so that
    candidate t = 3 h + d with d = 2 repeats the one before it.  Child of h, d:
    neuron n keeps bit n of h (neuron 0 the highest), the last one min(d, 1)."""
    m = bits + 1
    rn = [n for n in range(m) for _ in (0, 1)] + [m - 1]
    return snp_synth.make_system(m, rn, [2] * len(rn), [0] * len(rn), [2, 1] * m + [1], [0] * len(rn),
                                 [[] for _ in range(m)], [2] * m)


@pytest.mark.parametrize("bits,chunk,cap", [(19, (1 << 19) - 1, 0), (19, 1 << 19, 0), (19, (1 << 19) + 1, 0),
                                            (22, 1 << 22, 0), (22, (1 << 22) + 1, 0), (23, 1 << 25, 0),
                                            (23, 1 << 25, (1 << 23) + 12345)])
def test_large_passes(gpu, bits, chunk, cap):
    import torch
    system = choosers(bits)
    m = bits + 1
    s = gpu.System(system)
    s.explore(1, cap=cap, chunk=chunk, record_parents=True)
    n = min(2 << bits, cap) if cap else 2 << bits
    st = s.depth_stats()[1]
    examined = (n - 1) // 2 * 3 + (n - 1) % 2 + 1 if cap else 3 << bits
    assert (st.new, st.examined, st.candidates, st.truncated) == (n, examined, 3 << bits, 1 if cap else 0)
    out = torch.empty((n + 1, m), dtype=torch.int32, device="cuda")
    assert gpu.snp_reachable(s.h, out, n + 1) == n + 1
    assert (out[0] == 2).all()
    r = torch.arange(n, device="cuda")
    for k in range(bits):
        assert (out[1:, k] == ((r >> (bits - k)) & 1)).all(), k
    assert (out[1:, bits] == (r & 1)).all()
    par = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    idx = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    gpu.snp_parents(s.h, par, idx, n + 1)
    assert par[0] == -1 and (par[1:] == 0).all()
    assert idx[0] == 0 and (idx[1:] == (r >> 1) * 3 + (r & 1)).all()
