"""What the serving loop holds and reports."""
import threading

import pytest

import snp_synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


def opts(gpu, depth, cap, budget):
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget = depth, cap, budget
    return o


def systems_of(n, m, seed=0):
    return [snp_synth.random_system(8100 + seed * 100 + k, m, (2, 3), (4, 4), (0, 6), "sparse") for k in range(n)]


def test_counters_account_for_every_request(gpu):
    """submitted = completed + active + pending whenever one looks, and a
    finished request can be polled once it is counted."""
    systems = systems_of(64, 200, seed=4)
    hs = [gpu.System(x) for x in systems]
    srv = gpu.snp_server_create(1024 * MB, 64)
    bad, stop = [], threading.Event()

    def watch():
        while not stop.is_set():
            i = gpu.snp_server_stats(srv)
            if i.submitted != i.completed + i.active + i.pending:
                bad.append((i.submitted, i.completed, i.active, i.pending))

    t = threading.Thread(target=watch)
    t.start()
    try:
        for _ in range(4):
            for h in hs:
                gpu.snp_server_submit(srv, h.h, opts(gpu, 3, 256, 4096))
            gpu.snp_server_wait(srv)
            assert len(gpu.snp_server_poll(srv)[2]) == 64
    finally:
        stop.set()
        t.join()
        gpu.snp_server_destroy(srv)
    assert not bad, bad[:5]
