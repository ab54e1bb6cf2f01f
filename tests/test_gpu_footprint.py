"""pb_run_footprint of +-1 bicliques counts the readout's sign words: by replica, the footprint is at least the
encoded spins and best states of both sides, the returned states and energies, the readout's row-tile partials and
one bit per spin of the state set being read."""
import pytest

import synth_inputs as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 256])
@pytest.mark.parametrize("form", ["resident", "cudacore"])
def test_sign_words_are_counted(n, form):
    from paper_2510_23419_gb300 import _build, native as pb
    _build.build()
    pb.load()
    f = {"resident": pb.PB_FORM_RESIDENT, "cudacore": pb.PB_FORM_CUDACORE}[form]
    inst = pb.pb_create_instance(pb.PB_TOPO_BICLIQUE, syn.biclique_couplings(n, "pm1", 1), None, n=n)
    try:
        sc = pb.make_schedule(pb.PB_SCHED_LINEAR, 10, 0.1, 1.0)
        fp = [pb.pb_run_footprint(inst, sc, R, pb.make_opts(f)) for R in (256, 512)]
    finally:
        pb.pb_instance_destroy(inst)
    ld, words, tiles = (n + 15) // 16 * 16, (n + 31) // 32, (n + 63) // 64
    sbits = 2 * words * 4
    known = 4 * ld + 2 * 2 * n + 2 * 8 + 8 * tiles + 3 * 4 + 2 * tiles * 4  # with the running bests and the sweeps' partials
    assert fp[1] - fp[0] >= 256 * (known + sbits)
