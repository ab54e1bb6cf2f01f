"""The annealing work whose speed is measured: listed cases and a draw of more of the same ranges.

A case is one call of the library as a program makes it: the instance, the schedule and the seed are in hand
(``prepare``), and a pass (``run``) starts the anneal, waits for it and reads its results back.  Sizes, schedules and
laws are those of the benchmark's workloads and of the tests:

* EA cubes (3D Edwards-Anderson, +-1 or N(0,1) bonds, with or without fields), L = 2 .. 32, 1 .. 1024 replicas;
* bicliques K_{n,n} with +-1, N(0,1) or U(-1,1) couplings, n = 20 .. 4096, 32 .. 4096 replicas;
* general sparse graphs with three or more colours, annealed or under parallel tempering;
* a mixed batch of cubes and bicliques of uneven sizes, replica counts and sweep budgets.

Couplings of +-1 give whole-number energies and trajectories that are the same on every machine.  Real couplings
give +-1 states and FP64 energies of those states.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2510_23419_gb300 import native as pb

KINDS = ("ea", "biclique", "graph", "tempering", "batch")
LAWS = {"pm1": pb.PB_DIST_PM1, "gauss": pb.PB_DIST_GAUSS, "unif": pb.PB_DIST_UNIF}
SCHEDS = {"linear": pb.PB_SCHED_LINEAR, "geometric": pb.PB_SCHED_GEOMETRIC}


# --------------------------------------------------------------------- cases
def listed():
    def ea(name, L, law, R, S, sched, b0, b1, h=0, stream="own", target=0.0):
        return dict(name=name, kind="ea", L=L, law=law, replicas=R, sweeps=S, sched=sched, beta0=b0, beta1=b1, h=h,
                    stream=stream, target=target)

    def bq(name, n, law, R, S, stream="own"):
        return dict(name=name, kind="biclique", n=n, law=law, replicas=R, sweeps=S, sched="linear", beta0=0.35,
                    beta1=3.5, h=0, stream=stream, target=0.0)

    return [
        # one small cube and few replicas, waited for: latency of a single solve (the smallest workload of the benchmark)
        ea("ea_L6_pm1_R64", 6, "pm1", 64, 1000, "linear", 0.1, 3.0, stream="default"),
        # a ragged request: a side that no compile-time shape covers, whole-number fields, odd replica count, a target
        # energy to record (a target run of a user who looks for the first sweep at a given quality)
        ea("ea_L10_pm1_fields_R101", 10, "pm1", 101, 700, "linear", 0.35, 3.5, h=2, stream="default", target=-1.5),
        # the ordinary single solves: medium cubes, a full replica set, both coupling types
        ea("ea_L16_pm1_R1024", 16, "pm1", 1024, 1000, "geometric", 0.1, 5.0),
        ea("ea_L16_gauss_R256", 16, "gauss", 256, 1000, "geometric", 0.1, 5.0),
        # the large cubes of the batched benchmark, each alone
        ea("ea_L32_pm1_R1024", 32, "pm1", 1024, 500, "geometric", 0.1, 5.0),
        ea("ea_L32_gauss_R1024", 32, "gauss", 1024, 250, "geometric", 0.1, 5.0),
        # bicliques: the paper's own size range (couplings from [-1, 1], resident form), a latency-bound one, and the
        # largest of the benchmark's sweep on both tensor-core couplings
        bq("bq_n100_unif_R100", 100, "unif", 100, 500, stream="default"),
        bq("bq_n512_pm1_R256", 512, "pm1", 256, 400),
        bq("bq_n2048_gauss_R1024", 2048, "gauss", 1024, 150),
        bq("bq_n4096_pm1_R4096", 4096, "pm1", 4096, 100),
        # an odd periodic cube (not bipartite: four greedy colours), the general-graph benchmark
        dict(name="graph_cube25_pm1_R1024", kind="graph", graph="cube", size=25, law="pm1", replicas=1024, sweeps=150,
             sched="linear", beta0=0.1, beta1=3.0, h=0, stream="own", target=0.0),
        # uneven jobs of one batch call, as a server's admission round or a study of many instances sends them
        dict(name="batch_mixed_12", kind="batch", jobs=12, mix=12, sweeps_lo=50, sweeps_hi=1000, stream="own"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(KINDS, weights=(5, 4, 2, 1, 1))[0]
    stream = rng.choice(("own", "default"))
    if kind == "batch":
        return dict(kind=kind, jobs=rng.randint(2, 12), mix=rng.randrange(1 << 20), sweeps_lo=50, sweeps_hi=1000,
                    stream=stream)
    if kind == "ea":
        law = rng.choice(("pm1", "gauss"))
        L = 2 * rng.randint(1, 16)
        R = _log_int(rng, 1, 1024)
        # sweeps log-uniform, within the cost of the largest listed cube of the law
        cap = (32 ** 3) * 1024 * (500 if law == "pm1" else 250) // 2
        S = max(1, min(_log_int(rng, 50, 1000), cap // (max(L, 6) ** 3 * max(R, 152))))
        sched, b0, b1 = rng.choice((("linear", 0.1, 3.0), ("geometric", 0.1, 5.0), ("linear", 0.35, 3.5)))
        return dict(kind=kind, L=L, law=law, replicas=R, sweeps=S, sched=sched, beta0=b0, beta1=b1,
                    h=rng.choice((0, 0, 0, 1, 3)), stream=stream, target=rng.choice((0.0, 0.0, -1.4)))
    if kind == "biclique":
        law = rng.choice(("pm1", "gauss", "unif"))
        n = _log_int(rng, 20, 4096)
        R = _log_int(rng, 32, 4096)
        cap = 4096 * 4096 * 4096 * (80 if law == "pm1" else 20)
        S = max(2, min(_log_int(rng, 50, 500), cap // (max(n, 512) ** 2 * max(R, 512))))
        return dict(kind=kind, n=n, law=law, replicas=R, sweeps=S, sched="linear", beta0=0.35, beta1=3.5,
                    h=rng.choice((0, 0, 0, 2)), stream=stream, target=0.0)
    graph = rng.choice(("cube", "random"))
    size = 2 * rng.randint(2, 12) + 1 if graph == "cube" else _log_int(rng, 200, 4000)
    law = rng.choice(("pm1", "pm1", "gauss"))
    if kind == "graph":
        return dict(kind=kind, graph=graph, size=size, law=law, replicas=_log_int(rng, 5, 1024),
                    sweeps=_log_int(rng, 20, 150), sched="linear", beta0=0.1, beta1=3.0, h=rng.choice((0, 0, 2)),
                    stream=stream, target=0.0)
    return dict(kind=kind, graph=graph, size=size, law=law, temps=rng.randint(2, 16), chains=_log_int(rng, 4, 64),
                sweeps=_log_int(rng, 20, 100), beta0=0.1, beta1=3.0, h=0, stream=stream, target=0.0)


# -------------------------------------------------------------------- inputs
def _graph_edges(case):
    """(N, eu, ev): the periodic cube of an odd side, or a random graph of mean degree about eight whose
    structure belongs to the size (its couplings come from the seed)."""
    size = case["size"]
    if case["graph"] == "cube":
        idx = np.arange(size ** 3).reshape(size, size, size)
        eu = np.concatenate([idx.reshape(-1)] * 3)
        ev = np.concatenate([np.roll(idx, -1, axis=ax).reshape(-1) for ax in (2, 1, 0)])
        return size ** 3, eu.astype(np.int32), ev.astype(np.int32)
    rng = np.random.default_rng(size)
    pairs = rng.integers(0, size, size=(4 * size, 2))
    pairs = np.sort(pairs[pairs[:, 0] != pairs[:, 1]], axis=1)
    pairs = np.unique(pairs, axis=0)
    return size, pairs[:, 0].astype(np.int32), pairs[:, 1].astype(np.int32)


def _mix_jobs(case):
    """Jobs of the batch: cubes and bicliques, +-1 and N(0,1), 32 .. 1024 replicas, log-uniform sweep budgets."""
    rng = random.Random(case["mix"])
    jobs = []
    for _ in range(case["jobs"]):
        law = rng.choice(("pm1", "gauss"))
        S = _log_int(rng, case["sweeps_lo"], case["sweeps_hi"])
        R = 2 ** rng.randint(5, 10)
        if rng.random() < 0.5:
            jobs.append(dict(kind="ea", L=rng.choice((8, 12, 16, 24)), law=law, replicas=R, sweeps=S))
        else:
            jobs.append(dict(kind="biclique", n=rng.choice((128, 256, 512, 1024, 2048)), law=law, replicas=R, sweeps=S))
    for j in jobs:
        j.update(sched="geometric", beta0=0.1, beta1=5.0, h=0)
    return jobs


def _couplings(case, seed):
    """Couplings and fields of one instance from the seed (fields None without any)."""
    kind = case["kind"]
    rng = np.random.default_rng((seed, 1))
    if kind == "ea":
        J, N = pb.pb_generate_ea(case["L"], LAWS[case["law"]], seed), case["L"] ** 3
    elif kind == "biclique":
        J, N = pb.pb_generate_biclique(case["n"], LAWS[case["law"]], seed), 2 * case["n"]
    else:
        N, eu, _ = _graph_edges(case)
        J = (rng.choice(np.array([-1, 1], np.int8), size=eu.size) if case["law"] == "pm1"
             else rng.standard_normal(eu.size).astype(np.float32))
    h = None
    if case["h"]:
        h = (rng.integers(-case["h"], case["h"] + 1, size=N).astype(np.int8) if case["law"] == "pm1"
             else (0.5 * case["h"] * rng.standard_normal(N)).astype(np.float32))
    return J, h, N


class _State:
    """What the program holds between calls: instance handles, schedules, seeds, its stream."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.insts = []
        self.stream = torch.cuda.Stream() if case["stream"] == "own" else None
        jobs = _mix_jobs(case) if case["kind"] == "batch" else [case]
        self.jobs, self.scheds, self.sizes = jobs, [], []
        for q, j in enumerate(jobs):
            J, h, N = _couplings(j, seed + 1000 * q)
            if j["kind"] == "ea":
                inst = pb.pb_create_instance(pb.PB_TOPO_EA3D, J, h, L=j["L"], stream=self.stream)
            elif j["kind"] == "biclique":
                inst = pb.pb_create_instance(pb.PB_TOPO_BICLIQUE, J, h, n=j["n"], stream=self.stream)
            else:
                _, eu, ev = _graph_edges(j)
                inst = pb.pb_create_graph_instance(N, eu, ev, J, h, stream=self.stream)
            self.insts.append(inst)
            self.sizes.append(N)
            if j["kind"] != "tempering":
                self.scheds.append(pb.make_schedule(SCHEDS[j["sched"]], j["sweeps"], j["beta0"], j["beta1"]))
        if case["kind"] == "tempering":
            self.ladder = np.linspace(case["beta0"], case["beta1"], case["temps"])
        target = case.get("target", 0.0)
        self.opts = pb.make_opts(target_energy=target * self.sizes[0]) if target else None

    def __del__(self):
        for inst in self.insts:
            pb.pb_instance_destroy(inst)


def prepare(case, seed):
    return _State(case, seed)


# ---------------------------------------------------------------------- pass
def _read(run, R, N):
    fe, be, bs = pb.pb_energy(run, R)
    return dict(final_E=fe, best_E=be, best_sweep=bs, best_states=pb.pb_best_states(run, R, N),
                final_states=pb.pb_final_states(run, R, N))


def run(state):
    case = state.case
    if case["kind"] == "batch":
        R = [j["replicas"] for j in state.jobs]
        seeds = [state.seed + 17 * q for q in range(len(R))]
        runs = pb.pb_anneal_batch(state.insts, state.scheds, R, seeds, stream=state.stream)
        try:
            return [_read(r, Rq, N) for r, Rq, N in zip(runs, R, state.sizes)]
        finally:
            for r in runs:
                pb.pb_run_destroy(r)
    if case["kind"] == "tempering":
        M, C = case["temps"], case["chains"]
        r = pb.pb_anneal_pt(state.insts[0], state.ladder, case["sweeps"], C, state.seed, stream=state.stream)
        try:
            out = _read(r, M * C, state.sizes[0])
            out["slot_temp"], out["accepted"] = pb.pb_pt_state(r, M, C)
            return out
        finally:
            pb.pb_run_destroy(r)
    R = case["replicas"]
    r = pb.pb_anneal(state.insts[0], state.scheds[0], R, state.seed, state.opts, stream=state.stream)
    try:
        out = _read(r, R, state.sizes[0])
        if state.opts is not None:
            out["target_sweep"] = pb.pb_target_sweeps(r, R)
        return out
    finally:
        pb.pb_run_destroy(r)


# ---------------------------------------------------------------------- work
def _job_work(j):
    size = 1 if j["law"] == "pm1" else 4
    if j["kind"] == "ea":
        N, deg, edges = j["L"] ** 3, 6, 3 * j["L"] ** 3
    elif j["kind"] == "biclique":
        N, deg, edges = 2 * j["n"], j["n"], j["n"] ** 2
    else:
        N, eu, _ = _graph_edges(j)
        deg, edges = 2.0 * eu.size / N, eu.size * (1 + 8 // size)  # a coupling and its two ends
    R = j["temps"] * j["chains"] if j["kind"] == "tempering" else j["replicas"]
    # couplings in; best and final states and three numbers per replica out; a multiply and an add per neighbour of
    # every update
    return edges * size + 2 * R * N + 20 * R, 2.0 * deg * N * R * j["sweeps"]


def work(case):
    parts = [_job_work(j) for j in (_mix_jobs(case) if case["kind"] == "batch" else [case])]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# --------------------------------------------------------------------- exact
# The anneal itself in plain numpy with 64-bit arithmetic, for +-1 couplings (real couplings decide in FP32, and one
# decision that falls the other way gives another trajectory).
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on arrays of counter words (uint64 holding 32-bit values): [..., 4] words."""
    m32 = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)
    x = [np.asarray(v, np.uint64) for v in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(b >> s32) ^ x[1] ^ np.uint64(k0), b & m32, (a >> s32) ^ x[3] ^ np.uint64(k1), a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack(x, axis=-1)


def _greedy(N, eu, ev):
    """Greedy colouring: vertices by decreasing degree, ties by index, smallest free colour."""
    adj = [[] for _ in range(N)]
    for u, v in zip(eu.tolist(), ev.tolist()):
        adj[u].append(v)
        adj[v].append(u)
    colour = [-1] * N
    for i in sorted(range(N), key=lambda i: (-len(adj[i]), i)):
        used = {colour[j] for j in adj[i]}
        c = 0
        while c in used:
            c += 1
        colour[i] = c
    return np.array(colour)


def exact(case, seed):
    if case["kind"] not in ("ea", "biclique", "graph") or case["law"] != "pm1":
        return None
    if _job_work(case)[1] > 1.0e9 or (case["kind"] == "biclique" and case["n"] > 256):
        return None  # more than some ten seconds
    J, h, N = _couplings(case, seed)
    R, S = case["replicas"], case["sweeps"]
    if case["kind"] == "ea":
        L = case["L"]
        idx = np.arange(N).reshape(L, L, L)
        eu = np.concatenate([idx.reshape(-1)] * 3)
        ev = np.concatenate([np.roll(idx, -1, axis=ax).reshape(-1) for ax in (2, 1, 0)])
        Je = J.reshape(-1)
        colour = np.indices((L, L, L)).sum(0).reshape(-1) & 1
    elif case["kind"] == "biclique":
        n = case["n"]
        eu, ev = (a.reshape(-1) for a in np.mgrid[0:n, n:2 * n])
        Je = J.reshape(-1)
        colour = (np.arange(N) >= n).astype(int)
    else:
        _, eu, ev = _graph_edges(case)
        Je = J
        colour = _greedy(N, eu, ev)
    hv = np.zeros(N) if h is None else h.astype(np.float64)
    # neighbour lists padded to the largest degree (slot N: a spin that is always zero)
    ends, other, Jd = np.concatenate([eu, ev]), np.concatenate([ev, eu]), np.concatenate([Je, Je]).astype(np.float64)
    order = np.argsort(ends, kind="stable")
    ends, other, Jd = ends[order], other[order], Jd[order]
    first = np.searchsorted(ends, np.arange(N))
    slot = np.arange(ends.size) - first[ends]
    width = int(slot.max()) + 1
    nb, Jn = np.full((N, width), N), np.zeros((N, width))
    nb[ends, slot], Jn[ends, slot] = other, Jd
    classes = [np.flatnonzero(colour == c) for c in range(int(colour.max()) + 1)]
    quads = np.arange((R + 3) // 4)

    def words(c, s, tag):
        k = np.arange(classes[c].size)
        return _philox(k[:, None], s, quads[None, :], (tag << 24) | c, seed).reshape(k.size, -1)[:, :R]

    def field(sites, m):
        F = np.repeat(hv[sites][:, None], R, axis=1)
        for a in range(width):
            F += Jn[sites, a][:, None] * m[nb[sites, a]]
        return F

    def energy(m):
        return -0.5 * ((field(np.arange(N), m) + hv[:, None]) * m[:N]).sum(0)

    m = np.zeros((N + 1, R))
    for c, sites in enumerate(classes):
        m[sites] = np.where(words(c, 0, 1) < 2 ** 31, 1.0, -1.0)
    E = energy(m)
    best_E, best, best_sweep = E.copy(), m[:N].copy(), np.full(R, -1, np.int32)
    target = case.get("target", 0.0) * N
    hit = np.full(R, -1, np.int32)
    for s in range(S):
        x = s / (S - 1) if S > 1 else 0.0
        b0, b1 = case["beta0"], case["beta1"]
        beta = b0 + (b1 - b0) * x if case["sched"] == "linear" else b0 * (b1 / b0) ** x
        for c, sites in enumerate(classes):
            F = field(sites, m)
            T = np.minimum(np.floor((0.5 + 0.5 * np.tanh(beta * F)) * 2.0 ** 32), 2.0 ** 32 - 1)
            m[sites] = np.where(words(c, s, 0) < T, 1.0, -1.0)
        E = energy(m)
        better = E < best_E
        best_E[better], best_sweep[better] = E[better], s
        best[:, better] = m[:N, better]
        if target:
            hit[(hit < 0) & (E <= target)] = s
    out = dict(final_E=E, best_E=best_E, best_sweep=best_sweep, best_states=best.T.astype(np.int8),
               final_states=m[:N].T.astype(np.int8))
    if target:
        out["target_sweep"] = hit
    return out
