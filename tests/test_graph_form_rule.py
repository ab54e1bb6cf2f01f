"""Which form a general +-1 graph takes under PB_FORM_AUTO: the rule, compiled from the library's own header, against
both forms' measured times (GB300, us per sweep), and both forms' results against each other."""
import os
import subprocess

import numpy as np
import pytest

import synth_inputs as syn

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# spins, classes, mean degree, rounds, slot rounds and slot words of the resident rows; replicas: (class launches, resident)
MEASURED = [
    (1331, 4, 6.0, 4, 34, 2930, {1: (26.8, 5.3), 64: (28.1, 5.3), 1024: (29.6, 7.6)}),
    (4000, 6, 14.0, 6, 114, 19862, {1: (41.0, 15.7), 1024: (59.5, 19.6)}),
    (15625, 4, 6.0, 10, 88, 34732, {4: (33.7, 19.6), 64: (34.7, 19.7), 256: (42.9, 21.1), 1024: (70.3, 28.4)}),
    (29791, 4, 6.0, 16, 142, 66374, {4: (44.6, 32.5), 16: (37.6, 32.5), 64: (39.8, 32.8), 1024: (107.3, 47.8)}),
    (50653, 4, 6.0, 26, 232, 113014, {8: (45.9, 51.9), 64: (45.2, 52.2), 256: (66.5, 56.0), 1024: (175.6, 77.2)}),
    (59319, 4, 6.0, 32, 284, 132404, {8: (49.4, 61.5), 64: (48.9, 62.0), 128: (58.1, 66.5), 256: (74.7, 66.4), 512: (112.3, 66.6)}),
    (60000, 7, 8.0, 35, 412, 178800, {4: (74.2, 85.2), 16: (65.0, 85.4), 64: (68.8, 85.8), 512: (131.8, 91.4)}),
    (60000, 8, 12.0, 33, 566, 258416, {4: (84.7, 101.4), 64: (86.4, 102.1), 256: (127.1, 107.5), 1024: (338.8, 134.3)}),
    (60000, 3, 2.0, 31, 92, 44674, {4: (54.5, 45.5), 256: (67.0, 50.7)}),
]

PROG = r'''
#include <stdio.h>
#include "csr_launch.h"
int main() {
  int N, k, ro, sr, sw, R; double d;
  while (scanf("%d %d %lf %d %d %d %d", &N, &k, &d, &ro, &sr, &sw, &R) == 7)
{
    pb::CsrResDevice g{};
    g.rounds = ro;
    g.slot_rounds = sr;
    g.slot_words = sw;
    double cl, cr;
    const double l = pb::csr_seconds(g, k, N, d, (R + 3) / 4, 1000, 152, false, &cl);
    const double r = pb::csr_seconds(g, k, N, d, (R + 3) / 4, 1000, 152, true, &cr);
    printf("%d %.17g %.17g %.17g %.17g\n", pb::csr_res_us(g, (R + 3) / 4, 152) < pb::csr_launches_us(k, N, d, (R + 3) / 4),
           l, cl, r, cr);
  }
  return 0; }'''


def _rule(tmp_path):
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.isdir(d)), None)
    if cuda is None:
        pytest.skip("CUDA headers not available")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2510_23419_gb300", "csrc"), "-I", os.path.join(cuda, "include"),
                           str(src), "-o", str(exe)])
    points = [(m[:6], R, t) for m in MEASURED for R, t in m[6].items()]
    text = "\n".join(" ".join(map(str, m + (R,))) for m, R, _ in points)
    rows = [l.split() for l in subprocess.check_output([str(exe)], input=text.encode()).decode().splitlines()]
    assert len(rows) == len(points)
    return [(p, r[0] == "1", [float(x) for x in r[1:]]) for p, r in zip(points, rows)]


def test_rule_takes_the_faster_form(tmp_path):
    for (m, R, (launches, resident)), pick, _ in _rule(tmp_path):
        assert (resident < launches) == pick, (m, R)


def test_job_cost_follows_the_form(tmp_path):
    """Seconds of 1000 sweeps within a third of the measured times (the fit's own spread is 25%), the share that needs
    SMs between none and all of them."""
    for (m, R, (launches, resident)), _, (l, cl, r, cr) in _rule(tmp_path):
        for sec, c, us in ((l, cl, launches), (r, cr, resident)):
            assert 0.75 <= sec / (1e-3 * us) <= 4 / 3 and 0.0 <= c <= sec, (m, R, sec, us)
        assert cr <= r * max(1, (R + 3) // 4) / 152 + 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("graph,R", [("cube9", 5), ("cube9", 700), ("ring60000", 6), ("ring60000", 700)])
def test_forms_agree(graph, R):
    from paper_2510_23419_gb300 import _build, native as pb
    _build.build()
    pb.load()
    if graph == "cube9":
        N, (eu, ev) = 729, syn.graph_periodic_cube(9)
    else:  # the launches with 6 replicas, the resident form with 700
        N = 60000
        v = np.arange(N, dtype=np.int32)
        steps = (1, 2, 5, 1001)
        eu, ev = np.concatenate([v] * len(steps)), np.concatenate([(v + d) % N for d in steps]).astype(np.int32)
    J = syn.edge_couplings(eu.size, "pm1", N)
    inst = pb.pb_create_graph_instance(N, eu, ev, J)
    out = []
    try:
        for form in (pb.PB_FORM_AUTO, pb.PB_FORM_PLAIN):
            run = pb.pb_anneal(inst, pb.make_schedule(pb.PB_SCHED_LINEAR, 5, 0.1, 2.0), R, 9, pb.make_opts(form))
            try:
                out.append((*pb.pb_energy(run, R), pb.pb_final_states(run, R, N), pb.pb_best_states(run, R, N)))
            finally:
                pb.pb_run_destroy(run)
    finally:
        pb.pb_instance_destroy(inst)
    for a, b in zip(*out):
        assert np.array_equal(a, b)
