"""Timed cases of the simulator, each through its public entry points.

A case is one thing a program asks of the library once its system is loaded:
explore it and take the configurations into a device buffer, list the
successors of one configuration, explore many systems together, or serve a
burst of requests.  Kinds:

  tree    the paper's 3-neuron system to a small depth: latency and launches
  step    every successor of one configuration (snp_step)
  static  an exploration into the caller's buffer, without allocation
  explore snp_explore and snp_reachable of one system, in its transitions
          (plain int32, fp8 and int8 tensor core) and options (packed store,
          parent records)
  batch   independent systems explored together (snp_explore_batch)
  serve   a burst of requests through the serving loop (snp_server_*)

Systems are drawn from the seed by snp_synth's recipes.  All outputs are whole
numbers.
"""
from __future__ import annotations

import dataclasses

import numpy as np
import torch

import paper_1104_1824_gb300 as snp
import snp_synth

TREE_ROWS = 4096  # configurations of the paper's system to depth 12 from at most 3 spikes per neuron: far fewer
TRANSITIONS = {"sparse": snp.SNP_T_SPARSE_I32, "i8": snp.SNP_T_TC_I8, "f8": snp.SNP_T_TC_F8}


def _explore(name, m, rules, deg, c0, mode, depth, cap, budget, transition="sparse", packed=False, parents=False):
    return {"name": name, "kind": "explore", "m": m, "rules_lo": rules[0], "rules_hi": rules[1], "deg_lo": deg[0],
            "deg_hi": deg[1], "c0_hi": c0, "mode": mode, "depth": depth, "cap": cap, "budget": budget,
            "transition": transition, "packed": packed, "parents": parents}


def listed():
    return [
        # the paper's own example: ten depths of a few configurations, all latency
        {"name": "tree_3", "kind": "tree", "depth": 10},
        # one configuration expanded for a user who walks the computation tree by hand
        {"name": "step_1024", "kind": "step", "m": 1024, "rules_lo": 4, "rules_hi": 4, "deg_lo": 64, "deg_hi": 64,
         "c0_hi": 16, "mode": "dense", "capacity": 1 << 15},
        # a latency-critical loop that may not allocate
        {"name": "static_64", "kind": "static", "m": 64, "rules_lo": 2, "rules_hi": 3, "deg_lo": 4, "deg_hi": 4,
         "c0_hi": 6, "mode": "sparse", "depth": 6, "cap": 1 << 14, "budget": 1 << 18},
        # the 64-neuron workload of the benchmark, with int32 and packed configurations
        _explore("explore_64", 64, (2, 3), (4, 4), 6, "sparse", 8, 1 << 20, 1 << 24),
        _explore("explore_64_packed", 64, (2, 3), (4, 4), 6, "sparse", 8, 1 << 20, 1 << 24, packed=True),
        # an ordinary exploration with the computation graph's edges; rows of no whole 16-byte units
        _explore("explore_61_parents", 61, (2, 3), (4, 4), 6, "sparse", 8, 1 << 16, 1 << 20, parents=True),
        # rows longer than a lane holds, of an odd length
        _explore("explore_301", 301, (2, 3), (4, 4), 6, "sparse", 6, 1 << 18, 1 << 22),
        # the 1024-neuron system of the benchmark in its three transitions; a frontier small enough that three
        # explorations fit the card (the int8 product at a size it finishes in some ms)
        _explore("explore_1024", 1024, (4, 4), (64, 64), 16, "dense", 3, 1 << 19, 1 << 23),
        _explore("explore_1024_f8", 1024, (4, 4), (64, 64), 16, "dense", 3, 1 << 18, 1 << 22, transition="f8"),
        _explore("explore_1024_i8", 1024, (4, 4), (64, 64), 16, "dense", 2, 1 << 15, 1 << 19, transition="i8"),
        # an eighth of the benchmark's batch of independent systems
        {"name": "batch_512", "kind": "batch", "n": 512, "m_lo": 16, "m_hi": 256, "depth": 6, "cap": 1 << 12,
         "budget": 1 << 16},
        # what the serving loop holds at a time under the benchmark's arrival rate
        {"name": "serve_48", "kind": "serve", "n": 48, "m_lo": 8, "m_hi": 512, "depth_lo": 4, "depth_hi": 32,
         "cap": 1 << 12, "budget": 1 << 16},
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["tree", "step", "static", "narrow", "narrow", "wide", "wide", "tensor", "batch", "serve"])
    if kind == "tree":
        return {"kind": "tree", "depth": rng.randint(5, 12), "bump": rng.randint(0, 1)}
    if kind in ("narrow", "static"):
        m = _log(rng, 16, 128)
        if rng.random() < 0.5:
            m = max(16, m // 16 * 16)  # rows of whole 16-byte units
        sys = {"m": m, "rules_lo": 2, "rules_hi": 3, "deg_lo": 4, "deg_hi": rng.randint(4, 8), "c0_hi": 6,
               "mode": "sparse"}
        if kind == "static":
            cap = _log(rng, 1 << 8, 1 << 14)
            return {"kind": "static", **sys, "depth": rng.randint(3, 6), "cap": cap, "budget": 16 * cap}
        cap = _log(rng, 1 << 10, 1 << 20)
        return {"kind": "explore", **sys, "depth": rng.randint(4, 8), "cap": cap, "budget": 16 * cap,
                "transition": "sparse", "packed": rng.random() < 0.3, "parents": rng.random() < 0.3}
    if kind in ("wide", "step", "tensor"):
        m = _log(rng, 16 if kind == "step" else 129, 1024)
        dense = kind == "tensor" or rng.random() < 0.5
        deg = min(m - 1, rng.randint(16, 64)) if dense else 4
        sys = {"m": m, "rules_lo": 4 if dense else 2, "rules_hi": 4 if dense else 3, "deg_lo": deg, "deg_hi": deg,
               "c0_hi": 16 if dense else 6, "mode": "dense" if dense else "sparse"}
        if kind == "step":
            return {"kind": "step", **sys, "capacity": _log(rng, 1 << 6, 1 << 15)}
        if kind == "tensor":
            i8 = rng.random() < 0.5
            cap = _log(rng, 1 << 10, 1 << (15 if i8 else 18))
            return {"kind": "explore", **sys, "depth": 2, "cap": cap, "budget": 16 * cap,
                    "transition": "i8" if i8 else "f8", "packed": False, "parents": False}
        cap = _log(rng, 1 << 10, 1 << 19)
        return {"kind": "explore", **sys, "depth": rng.randint(2, 3), "cap": cap, "budget": 16 * cap,
                "transition": "sparse", "packed": rng.random() < 0.3, "parents": rng.random() < 0.3}
    cap = _log(rng, 1 << 8, 1 << 12)
    if kind == "batch":
        return {"kind": "batch", "n": _log(rng, 16, 512), "m_lo": 16, "m_hi": rng.randint(32, 256),
                "depth": rng.randint(3, 6), "cap": cap, "budget": 16 * cap}
    return {"kind": "serve", "n": _log(rng, 4, 48), "m_lo": 8, "m_hi": rng.randint(64, 512), "depth_lo": 4,
            "depth_hi": rng.randint(8, 32), "cap": cap, "budget": 16 * cap}


def _system(case, seed):
    if case["kind"] == "tree":
        base = snp_synth.paper_example()
        rng = snp_synth.Rng(seed)
        c0 = rng.randint(1, 3, 3) + np.array([1, 0, case.get("bump", 0)])  # neuron 1 can fire: the tree does not end
        return dataclasses.replace(base, c0=c0.astype(np.int32))
    return snp_synth.random_system(seed, case["m"], (case["rules_lo"], case["rules_hi"]),
                                   (case["deg_lo"], case["deg_hi"]), (0, case["c0_hi"]), case["mode"])


def _many_depths(case):
    """Depths by size: evenly spread over their range, large and small ones in turn."""
    n = case["n"]
    lo, hi = (case["depth"], case["depth"]) if case["kind"] == "batch" else (case["depth_lo"], case["depth_hi"])
    return [lo + (hi + 1 - lo) * ((7 * j + 3) % n) // n for j in range(n)]


def _many(case, seed):
    """The batch's or burst's systems and depths."""
    rng = snp_synth.Rng(seed)
    rules, deg = ((1, 4), (2, 8)) if case["kind"] == "batch" else ((2, 3), (4, 4))
    # neuron counts spread evenly over their range, so that two seeds ask for about the same work
    n = case["n"]
    ms = case["m_lo"] + ((case["m_hi"] - case["m_lo"]) * (np.arange(n) + rng.uniform(n)) / n).astype(np.int64)
    depths = _many_depths(case)
    base = int(rng.randint(1, 1 << 30, 1)[0])
    order = np.argsort(rng.uniform(n))
    return [(snp_synth.random_system(base + k, int(ms[j]), rules, deg, (0, 6), "sparse"), depths[j])
            for k, j in enumerate(order)]


def _capacity(case):
    """Rows of the result buffer (rows past the result stay zero)."""
    return TREE_ROWS if case["kind"] == "tree" else 1 + case["depth"] * case["cap"]


class _State:
    """What a program holds: loaded systems, result buffers, a server."""

    server = None

    def __del__(self):
        if self.server is not None:
            snp.snp_server_destroy(self.server)


def prepare(case, seed):
    st = _State()
    st.kind, st.case = case["kind"], case
    dev = torch.device("cuda")
    if st.kind in ("batch", "serve"):
        many = _many(case, seed)
        st.systems = [snp.System(s) for s, _ in many]
        st.capacity = [1 + d * case["cap"] for _, d in many]
        st.depths = [d for _, d in many]
        at = np.concatenate([[0], np.cumsum([c * s.m for c, s in zip(st.capacity, st.systems)])])
        # one buffer for all results, as large as any seed's neuron counts ask for
        spread = case["m_lo"] + (case["m_hi"] - case["m_lo"]) * np.arange(1, case["n"] + 1) / case["n"]
        size = sum((1 + d * case["cap"]) * int(m) for d, m in zip(_many_depths(case), spread))
        st.flat = torch.zeros(size, dtype=torch.int32, device=dev)
        st.rows = [st.flat[int(a):int(b)] for a, b in zip(at[:-1], at[1:])]
        if st.kind == "serve":
            # memory for the whole burst: each request's rows and its hash table
            need = sum(c * (4 * s.m + 64) + (1 << 20) for c, s in zip(st.capacity, st.systems))
            st.server = snp.snp_server_create(2 * int(need), 256)
        return st
    system = _system(case, seed)
    st.s = snp.System(system)
    if st.kind == "step":
        st.C = system.c0
        st.out = torch.zeros((case["capacity"], case["m"]), dtype=torch.int32, device=dev)
        return st
    st.capacity = _capacity(case)
    st.out = torch.zeros((st.capacity, st.s.m), dtype=torch.int32, device=dev)
    if case.get("parents"):
        st.parent = torch.zeros(st.capacity, dtype=torch.int64, device=dev)
        st.index = torch.zeros(st.capacity, dtype=torch.int64, device=dev)
    return st


def _padded(a, n):
    """a with zero rows up to n of them."""
    return np.concatenate([a, np.zeros((n - len(a), *a.shape[1:]), dtype=a.dtype)])


def _depths(s, depth):
    d = np.array([(d.new, d.parents, d.examined, d.truncated) for d in s.depth_stats()], dtype=np.int64)
    return _padded(d, depth + 1)


def run(st):
    case = st.case
    if st.kind == "step":
        psi = snp.snp_step(st.s.h, st.C, case["capacity"], st.out)
        return {"children": st.out, "count": min(psi, case["capacity"])}
    if st.kind == "static":
        o = snp.snp_explore_opts_init()
        o.depth, o.frontier_cap, o.candidate_budget = case["depth"], case["cap"], case["budget"]
        new = np.zeros(case["depth"] + 1, dtype=np.int64)
        n, reached = snp.snp_explore_static(st.s.h, o, st.out, st.capacity, new)
        return {"configs": st.out, "count": n, "new": new, "reached": reached}
    if st.kind == "batch":
        o = snp.snp_explore_opts_init()
        o.depth, o.frontier_cap, o.candidate_budget = case["depth"], case["cap"], case["budget"]
        status = np.zeros(len(st.systems), dtype=np.int32)
        snp.snp_explore_batch([s.h for s in st.systems], o, status)
        counts = [snp.snp_reachable(s.h, r, c) for s, r, c in zip(st.systems, st.rows, st.capacity)]
        return {"configs": st.flat, "counts": np.array(counts, dtype=np.int64), "status": status}
    if st.kind == "serve":
        for s, depth in zip(st.systems, st.depths):
            o = snp.snp_explore_opts_init()
            o.depth, o.frontier_cap, o.candidate_budget = depth, case["cap"], case["budget"]
            snp.snp_server_submit(st.server, s.h, o)
        snp.snp_server_wait(st.server)
        _, _, status = snp.snp_server_poll(st.server)
        counts = [snp.snp_reachable(s.h, r, c) for s, r, c in zip(st.systems, st.rows, st.capacity)]
        return {"configs": st.flat, "counts": np.array(counts, dtype=np.int64), "status": np.sort(status)}
    if st.kind == "tree":
        st.s.explore(case["depth"])
        n = snp.snp_reachable(st.s.h, st.out, st.capacity)
        return {"configs": st.out, "count": n, "depths": _depths(st.s, case["depth"])}
    st.s.explore(case["depth"], cap=case["cap"], budget=case["budget"], transition=TRANSITIONS[case["transition"]],
                 packed=case["packed"], record_parents=case["parents"])
    n = snp.snp_reachable(st.s.h, st.out, st.capacity)
    got = {"configs": st.out, "count": n, "depths": _depths(st.s, case["depth"])}
    if case["parents"]:
        snp.snp_parents(st.s.h, st.parent, st.index, st.capacity)
        got["parent"], got["index"] = st.parent, st.index
    return got


def work(case):
    """Bytes: every configuration written once, as the caller gets it, and every expanded one read once (a
    capped depth finds `cap` configurations; the last depth's are not expanded).  The arithmetic is a few
    integer additions per count written."""
    kind = case["kind"]
    if kind == "tree":
        n = 5 * case["depth"]
        return {"bytes": 2 * n * 3 * 4, "flops": 0}
    if kind == "step":
        return {"bytes": (1 + case["capacity"]) * case["m"] * 4, "flops": 0}
    if kind in ("batch", "serve"):
        m = (case["m_lo"] + case["m_hi"]) / 2
        d = case["depth"] if kind == "batch" else (case["depth_lo"] + case["depth_hi"]) / 2
        return {"bytes": case["n"] * case["cap"] * (2 * d - 1) * m * 4, "flops": 0}
    parents = 16 * case["depth"] * case["cap"] if case.get("parents") else 0
    return {"bytes": case["cap"] * (2 * case["depth"] - 1) * case["m"] * 4 + parents, "flops": 0}


# --- the same results from the definitions, in 64 bits ------------------------------------

def _applies(x, i, j, c):
    if x < c or x < i:
        return False
    return x == i if j == 0 else (x - i) % j == 0


def _choices(system, C):
    """Per neuron: its applicable rules in rule order, or None if it cannot fire."""
    by = [[] for _ in range(system.m)]
    for r in range(system.R):
        n = int(system.rule_neuron[r])
        if _applies(int(C[n]), int(system.rule_i[r]), int(system.rule_j[r]), int(system.rule_c[r])):
            by[n].append(r)
    return by


def _children(system, M, C, limit):
    """The first `limit` children of C (last neuron's choice varies fastest), and how many there are."""
    by = [b for b in _choices(system, C) if b]
    psi = 1
    for b in by:
        psi *= len(b)
    n = min(psi, limit)
    out = np.repeat((C + sum((M[b[0]] for b in by), np.zeros(system.m, np.int64)))[None, :], n, axis=0)
    q = np.arange(n, dtype=np.int64)
    for b in reversed(by):
        if len(b) == 1:
            continue
        if not q.any():
            break
        out += (M[b] - M[b[0]])[q % len(b)]
        q //= len(b)
    return out, psi


def _bfs(system, depth, cap, budget):
    M = system.M.astype(np.int64)
    rows = [system.c0.astype(np.int64)]
    seen = {rows[0].tobytes()}
    level, depths = [rows[0]], [(1, 0, 0, 0)]
    for _ in range(depth):
        total = 0
        for C in level:
            psi = 1
            for b in _choices(system, C):
                psi *= max(1, len(b))
            total += psi
        examined, new, left = 0, [], budget if budget > 0 else 1 << 62
        for C in level:
            full = left <= 0 or (cap > 0 and len(new) >= cap)
            if full:
                break
            kids, _ = _children(system, M, C, min(left, 1 << 20))
            for k in kids:
                examined += 1
                left -= 1
                key = k.tobytes()
                if key not in seen:
                    seen.add(key)
                    new.append(k.copy())
                    if cap > 0 and len(new) >= cap:
                        break
        depths.append((len(new), len(level), examined, int(examined < total)))
        if not new:
            break
        rows += new
        level = new
    return np.array(rows), np.array(depths, dtype=np.int64)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        system = _system(case, seed)
        kids, psi = _children(system, system.M.astype(np.int64), system.c0.astype(np.int64), case["capacity"])
        return {"children": _padded(kids, case["capacity"]), "count": min(psi, case["capacity"])}
    small = kind in ("static", "explore") and case["budget"] * case["depth"] * case["m"] <= 1 << 27
    if kind != "tree" and not small:
        return None
    rows, depths = _bfs(_system(case, seed), case["depth"], case.get("cap", 0), case.get("budget", 0))
    got = {"configs": _padded(rows, _capacity(case)), "count": len(rows)}
    depths = _padded(depths, case["depth"] + 1)
    if kind == "static":
        return {**got, "new": depths[:, 0], "reached": int(np.nonzero(depths[:, 0])[0][-1])}
    got["depths"] = depths
    return {**got, "parent": None, "index": None} if case.get("parents") else got
