"""Resident forms at the edges of their tile shapes, against the CPU oracle.

+-1 instances are whole-number exact.  Real couplings: a spin's field is the same
sum in the same order in the resident and in the plain (CUDA-core) form, so the
trajectories are equal; returned energies are those of the states, within 1e-9
of sum |J| (FP64 against FP64, N terms).
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


# sides with 2, 4, 6 and 8 sites per word; one word, part of a warp, several tiles per SM; ragged replicas
@pytest.mark.parametrize("L,R,hmax", [(2, 1, 0), (2, 9, 1), (4, 40, 0), (6, 64, 0), (6, 1301, 1), (8, 2500, 0),
                                      (10, 101, 2), (12, 1217, 0), (14, 9, 0), (16, 700, 1), (18, 5, 0), (24, 6, 2)])
def test_ea_pm1_words(pb, orc, L, R, hmax):
    S = 5
    J = syn.ea_couplings(L, "pm1", L + R)
    h = syn.int_fields(L ** 3, hmax, L) if hmax else None
    g = pb.anneal(pb.PB_TOPO_EA3D, J, pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.2, 2.0), R, 5, h=h, L=L,
                  form=pb.PB_FORM_RESIDENT)
    o = orc.anneal_ea(L, J.astype(float), None if h is None else h.astype(float), orc.schedule(0, 0.2, 2.0, S), R, 5)
    for k in KEYS:
        assert np.array_equal(g[k], o[k]), k


# three, five and two threads per summation lane, one lane per thread (L = 12: 576 lanes), two lanes per thread
@pytest.mark.parametrize("L,R,fields", [(2, 3, False), (6, 64, True), (6, 700, False), (10, 7, True), (12, 1300, True),
                                        (14, 30, False), (16, 9, True), (16, 700, False), (8, 2500, True),
                                        (20, 620, False), (24, 6, True)])
def test_ea_f32_lanes(pb, orc, L, R, fields):
    S = 6
    J = syn.ea_couplings(L, "gauss", L + R)
    h = 0.5 * np.random.default_rng(L).standard_normal(L ** 3).astype(np.float32) if fields else None
    sc = pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.2, 2.0)
    run = lambda form: pb.anneal(pb.PB_TOPO_EA3D, J, sc, R, 5, h=h, L=L, form=form)
    g, p = run(pb.PB_FORM_RESIDENT), run(pb.PB_FORM_PLAIN)
    assert np.array_equal(g["final_state"], p["final_state"])
    eu, ev, _ = orc.ea_graph(L)
    Jd = J.astype(float).reshape(-1)
    hd = None if h is None else h.astype(float)
    tol = 1e-9 * (np.abs(Jd).sum() + (0 if hd is None else np.abs(hd).sum()))
    for r in {0, R // 2, R - 1}:
        for s, e in (("final_state", "final_E"), ("best_state", "best_E")):
            assert abs(g[e][r] - orc.energy(eu, ev, Jd, hd, g[s][r])) <= tol


# words per row of a side, rows of a partial word, quads of replicas per CTA (from R); n > 256: the rule that
# takes the resident form without being asked
@pytest.mark.parametrize("n,R,hmax", [(1, 3, 0), (31, 20, 1), (32, 1, 0), (33, 700, 0), (64, 1300, 0), (65, 2500, 2),
                                      (128, 20, 0), (129, 9, 1), (255, 620, 0), (256, 4, 0), (257, 37, 1),
                                      (300, 700, 0), (512, 40, 0)])
def test_biclique_pm1_words(pb, orc, n, R, hmax):
    S = 4
    J = syn.biclique_couplings(n, "pm1", n + R)
    h = syn.int_fields(2 * n, hmax, n) if hmax else None
    g = pb.anneal(pb.PB_TOPO_BICLIQUE, J, pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.05, 0.5), R, 7, h=h, n=n,
                  form=pb.PB_FORM_RESIDENT if n <= 256 else pb.PB_FORM_AUTO)
    o = orc.anneal_biclique(n, J.astype(float), None if h is None else h.astype(float),
                            orc.schedule(0, 0.05, 0.5, S), R, 7)
    for k in KEYS:
        assert np.array_equal(g[k], o[k]), k


@pytest.mark.parametrize("n,R", [(1, 2), (3, 33), (100, 100), (127, 620), (128, 1300)])
def test_biclique_f32_quads(pb, n, R):
    J = syn.biclique_couplings(n, "gauss", n)
    sc = pb.make_schedule(pb.PB_SCHED_LINEAR, 6, 0.05, 0.5)
    run = lambda form: pb.anneal(pb.PB_TOPO_BICLIQUE, J, sc, R, 3, n=n, form=form)
    g, c = run(pb.PB_FORM_RESIDENT), run(pb.PB_FORM_CUDACORE)
    assert np.array_equal(g["final_state"], c["final_state"])
    E = -np.einsum("ri,ij,rj->r", g["final_state"][:, :n].astype(float), J.reshape(n, n).astype(float),
                   g["final_state"][:, n:].astype(float), optimize=True)
    assert np.all(np.abs(g["final_E"] - E) <= 1e-9 * np.abs(J.astype(float)).sum())


def _ring_with_chords(N, isolated, step):
    v = np.arange(N - isolated)
    n = v.size
    e = np.concatenate([np.stack([v, (v + 1) % n], 1), np.stack([v[::step], (v[::step] + n // 3) % n], 1)])
    e = np.unique(np.sort(e, axis=1), axis=0)
    return e[:, 0].astype(np.int32), e[:, 1].astype(np.int32)


# regular rows of six; rows of uneven degree with isolated spins and a partial last word; degrees above seven
@pytest.mark.parametrize("graph,R", [("cube5", 3), ("cube5", 700), ("cube7", 1301), ("ring77", 5), ("ring77", 650),
                                     ("random300", 9), ("random300", 1217)])
def test_graph_pm1_words(pb, orc, graph, R):
    S = 6
    if graph == "ring77":
        N, (eu, ev) = 77, _ring_with_chords(77, 8, 3)
    elif graph == "random300":
        N, (eu, ev) = 300, syn.graph_random(300, 750, 3)
    else:
        N, (eu, ev) = int(graph[4:]) ** 3, syn.graph_periodic_cube(int(graph[4:]))
    J = syn.edge_couplings(eu.size, "pm1", N)
    col, _ = pb.pb_greedy_colouring(N, eu, ev)
    inst = pb.pb_create_graph_instance(N, eu, ev, J, None, col)
    try:
        run = pb.pb_anneal(inst, pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.1, 2.0), R, 11)
        try:
            fe, be, bs = pb.pb_energy(run, R)
            g = dict(final_E=fe, best_E=be, best_sweep=bs, final_state=pb.pb_final_states(run, R, N),
                     best_state=pb.pb_best_states(run, R, N))
        finally:
            pb.pb_run_destroy(run)
    finally:
        pb.pb_instance_destroy(inst)
    o = orc.anneal(eu, ev, J.astype(float), None, col, orc.schedule(0, 0.1, 2.0, S), R, 11)
    for k in KEYS:
        assert np.array_equal(g[k], o[k]), k
