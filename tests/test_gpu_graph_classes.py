"""General +-1 graphs with caller-given colourings of many, of empty and of large classes, against the CPU oracle.

A spin's class index is part of the result (it orders the updates and feeds the random words), so any proper
colouring with values 0 .. 254 is legal input, up to one spin per class.  Whole-number couplings: everything is exact,
the recorded target sweeps too (first sweep whose energy in the oracle's trace is at or below the target).
"""
import numpy as np
import pytest

import synth_inputs as syn

pytestmark = pytest.mark.gpu

KEYS = ("final_state", "best_state", "final_E", "best_E", "best_sweep")


@pytest.fixture(scope="module")
def pb():
    from paper_2510_23419_gb300 import _build, native
    _build.build()
    native.load()
    return native


def _circulant(N, degree):
    """Every spin joined to the degree / 2 next ones on a ring."""
    v = np.arange(N, dtype=np.int32)
    steps = range(1, degree // 2 + 1)
    return np.concatenate([v for _ in steps]), np.concatenate([(v + d) % N for d in steps]).astype(np.int32)


def _two_sided(n, degree):
    """Sides of n spins, spin i of one joined to the spins i + 37 d of the other."""
    v = np.arange(n, dtype=np.int32)
    return (np.concatenate([v for _ in range(degree)]),
            np.concatenate([n + (v + 37 * d) % n for d in range(degree)]).astype(np.int32))


def _case(name):
    if name.startswith("own"):  # one spin per class: the sequential update
        N, deg = 255, int(name[3:])
        return (N,) + _circulant(N, deg) + (np.arange(N, dtype=np.int32),)
    if name == "pairs15":  # 120 classes of 5 spins, two words each; a ring of degree 14 and one matching: 15
        N = 600
        eu, ev = _circulant(N, 14)
        v = np.arange(N // 2, dtype=np.int32)
        return N, np.concatenate([eu, v]), np.concatenate([ev, v + N // 2]), (np.arange(N) % 120).astype(np.int32)
    if name == "gaps":  # class numbers with empty classes between, before and after
        N = 9 ** 3
        eu, ev = syn.graph_periodic_cube(9)
        return N, eu, ev, None
    n = 2304 if name == "wide15" else 2100  # several words of a class per thread, the last round part-filled
    deg = 15 if name == "wide15" else 7
    return (2 * n,) + _two_sided(n, deg) + ((np.arange(2 * n) >= n).astype(np.int32),)


@pytest.mark.parametrize("name,R,S", [("own14", 9, 120), ("own12", 9, 120), ("own8", 5, 80), ("pairs15", 700, 24),
                                      ("gaps", 13, 30), ("wide15", 9, 20), ("wide7", 6, 20)])
def test_given_classes_exact(pb, orc, name, R, S):
    N, eu, ev, col = _case(name)
    if col is None:
        col = 3 + 17 * pb.pb_greedy_colouring(N, eu, ev)[0].astype(np.int32)
    J = syn.edge_couplings(eu.size, "pm1", N + eu.size)
    betas = orc.schedule(0, 0.1, 3.0, S)
    o = orc.anneal(eu, ev, J.astype(float), None, col, betas, R, 11, trace=True)
    target = float(np.median(o["best_E"]))
    tr = o["trace_E"]
    hit = np.where((tr <= target).any(axis=1), (tr <= target).argmax(axis=1), -1)
    inst = pb.pb_create_graph_instance(N, eu, ev, J, None, col)
    try:
        run = pb.pb_anneal(inst, pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.1, 3.0), R, 11,
                           pb.make_opts(target_energy=target))
        try:
            fe, be, bs = pb.pb_energy(run, R)
            g = dict(final_E=fe, best_E=be, best_sweep=bs, final_state=pb.pb_final_states(run, R, N),
                     best_state=pb.pb_best_states(run, R, N))
            got = pb.pb_target_sweeps(run, R)
        finally:
            pb.pb_run_destroy(run)
    finally:
        pb.pb_instance_destroy(inst)
    for k in KEYS:
        assert np.array_equal(g[k], o[k]), k
    assert np.array_equal(got, hit)
