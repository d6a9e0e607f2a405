"""What the serving loop holds and reports."""
import threading

import pytest

import oracle
import snp_synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


def opts(gpu, depth, cap, budget):
    o = gpu.snp_explore_opts_init()
    o.depth, o.frontier_cap, o.candidate_budget = depth, cap, budget
    return o


def systems_of(n, m, seed=0):
    return [snp_synth.random_system(8100 + seed * 100 + k, m, (2, 3), (4, 4), (0, 6), "sparse") for k in range(n)]


def same(h, system, depth, cap, budget):
    e = oracle.Oracle(system).explore(depth, cap=cap, budget=budget)
    got = h.reachable()
    assert got.shape == e.configs.shape and (got == e.configs).all()
    assert [(d.new, d.examined, d.candidates, d.truncated) for d in h.depth_stats()] == \
        [(d.new, d.examined, d.candidates, d.truncated) for d in e.depths]


def used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_memory_stays_within_the_budget(gpu):
    """24 requests of 512 neurons and cap 2^15: their pools and tables fill
    the budget 14 at a time, the scratch of a pass of 2^16 candidates is 135 MB
    each."""
    systems = systems_of(24, 512)
    hs = [gpu.System(x) for x in systems]
    budget = 1024 * MB
    before = used()
    srv = gpu.snp_server_create(budget, 64)
    try:
        for h in hs:
            gpu.snp_server_submit(srv, h.h, opts(gpu, 1, 1 << 15, 100))
        gpu.snp_server_wait(srv)
        held = used() - before
        assert (gpu.snp_server_poll(srv)[2] == 0).all()
        # beside the budget: the results (0.2 MB each), queues of at most some tens of MB
        assert held <= budget + 64 * MB, held / MB
        for k in (0, 11, 23):
            same(hs[k], systems[k], 1, 1 << 15, 100)
    finally:
        gpu.snp_server_destroy(srv)


def as_large_as_the_budget(gpu):
    """A server, a system, its depth, cap and budget: pool and table of the
    request fill the server's memory."""
    system = systems_of(1, 64)[0]
    depth, cap, budget = 3, 4096, 40000
    up = lambda b: (b + 255) // 256 * 256
    rows = 1 + depth * cap
    slots = 8
    while slots < (rows + depth * 2048) * 4 // 3 + 8:
        slots *= 2
    need = up(rows * 64 * 4) + up(slots * 8) + up(64 * (depth + 1))
    return gpu.snp_server_create(need + 4096, 8), system, depth, cap, budget


def test_request_as_large_as_the_budget(gpu):
    """Accepted, and served with scratch of its own, between requests that
    need little."""
    srv, system, depth, cap, budget = as_large_as_the_budget(gpu)
    small = systems_of(6, 40, seed=1)
    big = gpu.System(system)
    hs = [gpu.System(x) for x in small]
    try:
        for h in hs[:3]:
            gpu.snp_server_submit(srv, h.h, opts(gpu, 3, 50, 500))
        gpu.snp_server_submit(srv, big.h, opts(gpu, depth, cap, budget))
        for h in hs[3:]:
            gpu.snp_server_submit(srv, h.h, opts(gpu, 3, 50, 500))
        gpu.snp_server_wait(srv)
        st = gpu.snp_server_poll(srv)[2]
        assert len(st) == 7 and (st == 0).all()
        same(big, system, depth, cap, budget)
        for h, x in zip(hs, small):
            same(h, x, 3, 50, 500)
    finally:
        gpu.snp_server_destroy(srv)


def test_scratch_of_its_own_cannot_be_had(gpu):
    """That allocation fails: the request is reported and counted, the server
    serves it when it is submitted again."""
    srv, system, depth, cap, budget = as_large_as_the_budget(gpu)
    big = gpu.System(system)
    try:
        gpu.snp_debug_fail_allocation(1)
        gpu.snp_server_submit(srv, big.h, opts(gpu, depth, cap, budget))
        gpu.snp_server_wait(srv)
        assert list(gpu.snp_server_poll(srv)[2]) == [gpu.SNP_E_NOMEM]
        with pytest.raises(gpu.SnpError):
            big.reachable()
        gpu.snp_server_submit(srv, big.h, opts(gpu, depth, cap, budget))
        gpu.snp_server_wait(srv)
        assert list(gpu.snp_server_poll(srv)[2]) == [0]
        same(big, system, depth, cap, budget)
        info = gpu.snp_server_stats(srv)
        assert info.submitted == info.completed == 2 and info.active == 0 and info.pending == 0
    finally:
        gpu.snp_debug_fail_allocation(0)
        gpu.snp_server_destroy(srv)


@pytest.mark.parametrize("k", range(1, 12))
def test_failed_allocation_fails_its_request_alone(gpu, k):
    """The k-th allocation of a burst fails: that request is reported, every
    other one is served, the counters account for all of them."""
    systems = systems_of(4, 64, seed=2)
    hs = [gpu.System(x) for x in systems]
    srv = gpu.snp_server_create(256 * MB, 8)
    try:
        gpu.snp_debug_fail_allocation(k)
        ids = []
        for h in hs:  # one at a time: what is allocated is the request's
            ids.append(gpu.snp_server_submit(srv, h.h, opts(gpu, 2, 64, 1000)))
            gpu.snp_server_wait(srv)
        got_ids, _, st = gpu.snp_server_poll(srv)
        status = dict(zip([int(i) for i in got_ids], [int(s) for s in st]))
        assert sorted(status) == sorted(ids)
        assert [status[i] for i in ids].count(gpu.SNP_E_NOMEM) == 1
        for i, h, x in zip(ids, hs, systems):
            if status[i] == gpu.SNP_E_NOMEM:
                with pytest.raises(gpu.SnpError):
                    h.reachable()
            else:
                assert status[i] == 0
                same(h, x, 2, 64, 1000)
        info = gpu.snp_server_stats(srv)
        assert info.submitted == info.completed == 4 and info.active == 0 and info.pending == 0
    finally:
        gpu.snp_debug_fail_allocation(0)
        gpu.snp_server_destroy(srv)


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
