"""Handles used from several threads at once, a thread per handle: systems of
different sizes go through the same kernels with different shared memory."""
import threading

import numpy as np
import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu


def run_all(workers, rounds: int):
    """Runs every worker `rounds` times, each in a thread of its own, and re-raises what one raised."""
    errors = []
    start = threading.Barrier(len(workers))

    def body(fn):
        try:
            start.wait()
            for _ in range(rounds):
                if errors:
                    return
                fn()
        except BaseException as e:  # noqa: BLE001 -- reported below
            errors.append(e)

    ts = [threading.Thread(target=body, args=(w,)) for w in workers]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def explorer(gpu, m: int, transition, depth: int, cap: int, budget: int, rules=(2, 3), deg=(4, 4)):
    system = snp_synth.random_system(720 + m, m, rules, deg, (0, 6), "sparse")
    s = gpu.System(system)
    want = oracle.Oracle(system).explore(depth, cap=cap, budget=budget).configs

    def once():
        s.explore(depth, cap=cap, budget=budget, transition=transition)
        got = s.reachable()
        assert got.shape == want.shape and (got == want).all()
    return once


@pytest.mark.parametrize("form,sizes", [("sparse", (16, 128)), ("sparse", (152, 600)), ("sparse", (700, 1020)),
                                        ("i8", (880, 1020)), ("f8", (64, 1020))])
def test_explorations_of_different_sizes(gpu, form, sizes):
    t = {"sparse": gpu.SNP_T_SPARSE_I32, "i8": gpu.SNP_T_TC_I8, "f8": gpu.SNP_T_TC_F8}[form]
    run_all([explorer(gpu, m, t, 3, 40, 400) for m in sizes], 150)


def test_batches_of_different_sizes(gpu):
    def batch(ms):
        systems = [snp_synth.random_system(740 + m, m, (2, 3), (4, 4), (0, 6), "sparse") for m in ms]
        hs = [gpu.System(x) for x in systems]
        want = [oracle.Oracle(x).explore(3, cap=40, budget=400).configs for x in systems]

        def once():
            assert (gpu.explore_batch(hs, 3, cap=40, budget=400) == 0).all()
            for h, w in zip(hs, want):
                got = h.reachable()
                assert got.shape == w.shape and (got == w).all()
        return once
    run_all([batch((16, 20)), batch((900, 1000))], 100)
