"""The autotuner on small +-1 bicliques: every form that PB_FORM_AUTO would take untuned is among its candidates, and a
tuned AUTO run gives the same results, in about the same time or less, as an untuned one."""
import numpy as np
import pytest

import synth_inputs as syn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pb():
    from paper_2510_23419_gb300 import _build, native
    _build.build()
    native.load()
    return native


def _run(pb, inst, n, sc, R, opts=None):
    run = pb.pb_anneal(inst, sc, R, 7, opts)
    try:
        out = (*pb.pb_energy(run, R), pb.pb_best_states(run, R, 2 * n))
        return pb.pb_run_kernel_ms(run), out
    finally:
        pb.pb_run_destroy(run)


# n = 256 and 512 keep most SMs busy for a 25th and a 10th of the tensor form's time
@pytest.mark.parametrize("n,R", [(100, 33), (256, 512), (257, 128), (300, 256), (512, 256)])
def test_tuned_auto_not_slower(pb, n, R):
    S = 100
    J = syn.biclique_couplings(n, "pm1", n)
    sc = pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.1, 1.0)
    inst = pb.pb_create_instance(pb.PB_TOPO_BICLIQUE, J, None, n=n)
    stop = pb.make_opts(target_energy=-1e9, flags=pb.PB_FLAG_STOP_AT_TARGET)  # never reached: all sweeps run
    pb.pb_autotune_clear()
    try:
        t0, a = min((_run(pb, inst, n, sc, R) for _ in range(3)), key=lambda r: r[0])
        t = pb.pb_autotune(inst, R, 32)
        forms = [t.candidate_form[c] for c in range(t.n_candidates)]
        assert t.form in forms and (pb.PB_FORM_RESIDENT if n <= 256 else pb.PB_FORM_AUTO) in forms
        t1, b = min((_run(pb, inst, n, sc, R) for _ in range(3)), key=lambda r: r[0])
        assert t1 <= 2.0 * t0, (t0, t1, t.form)
        _, c = _run(pb, inst, n, sc, R, stop)  # flags exclude the form that only the library names
    finally:
        pb.pb_autotune_clear()
        pb.pb_instance_destroy(inst)
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
