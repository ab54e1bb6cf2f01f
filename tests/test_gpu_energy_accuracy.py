"""Energies of returned states for real couplings of mixed magnitude, against correctly rounded sums (math.fsum).

One coupling of 1 and all the others just below 2^-36: any rounding of the small terms beside the large one, or of
their own partial sums in FP32, shows.  Bounds:
* cubes: the large and the small terms are summed apart, the large ones exactly and the small ones in FP64 (error at
  most 2^17 2^-53 times their sum 2^-20: 2^-56), so one rounding of a result near 1 is left: 2^-53 + 2^-55;
* bicliques: a row's sum is held as a pair of floats (exact here: the row of the large coupling has no other); rows are
  added in FP64 (4 of a thread, 16 threads, 32 lanes in a tree, a lane's tiles), and at most 3 + 15 + 5 + 1 of those
  additions have a partial sum near 1: 24 2^-53.
"""
import math

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


def _small(rng, shape):
    return (2.0 ** -36.5 * rng.uniform(0.75, 1.0, shape)).astype(np.float32)


def _check(E, exact, tol):
    err = np.abs(np.array([float(e - x) for e, x in zip(E, exact)]))
    assert np.all(err <= tol), (err.max(), tol)


@pytest.mark.parametrize("L,fields", [(32, False), (32, True), (10, True)])
def test_cube(pb, orc, L, fields):
    R, N = 8, L ** 3
    rng = np.random.default_rng(L)
    J = _small(rng, (3, N))
    J[1, N // 3] = 1.0
    h = _small(rng, N) if fields else None
    g = pb.anneal(pb.PB_TOPO_EA3D, J, pb.make_schedule(pb.PB_SCHED_LINEAR, 2, 0.5, 1.0), R, 3, h=h, L=L)
    eu, ev, _ = orc.ea_graph(L)
    Jd = J.astype(float).reshape(-1)
    for st, key in (("final_state", "final_E"), ("best_state", "best_E")):
        m = g[st].astype(float)
        exact = [math.fsum(np.concatenate([-Jd * m[r][eu] * m[r][ev], [] if h is None else -h.astype(float) * m[r]]))
                 for r in range(R)]
        _check(g[key], exact, 2.0 ** -53 + 2.0 ** -55)


@pytest.mark.parametrize("n,form", [(512, "tensor"), (100, "resident"), (333, "cudacore")])
def test_biclique(pb, n, form):
    R = 16
    J = _small(np.random.default_rng(n), (n, n))
    J[0] = 0.0
    J[0, 7] = 1.0
    # fields of the small couplings decide: the sides align, and their terms add up
    sc = pb.make_schedule(pb.PB_SCHED_LINEAR, 6, 2.0 ** 36, 2.0 ** 38)
    f = {"tensor": pb.PB_FORM_TENSOR, "resident": pb.PB_FORM_RESIDENT, "cudacore": pb.PB_FORM_CUDACORE}[form]
    g = pb.anneal(pb.PB_TOPO_BICLIQUE, J, sc, R, 3, n=n, form=f)
    Jd = J.astype(float)
    for st, key in (("final_state", "final_E"), ("best_state", "best_E")):
        m = g[st].astype(float)
        exact = [math.fsum((-Jd * np.outer(m[r][:n], m[r][n:])).reshape(-1)) for r in range(R)]
        _check(g[key], exact, 24 * 2.0 ** -53)
