"""State outputs of the cube readout at any address: pb_anneal_ea_noalloc writes into its caller's own buffers, which
may be slices of an arena with no alignment beyond a byte's.

On the CPU: the rule that picks the width of the stores, compiled from the library's own header, keeps every store
on a multiple of its size.  On the GPU: the same results at every offset from an aligned address.
"""
import os
import subprocess

import numpy as np
import pytest

import synth_inputs as syn

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROG = r'''
#include <stdio.h>
#include "ea_launch.h"
int main() {
  for (int L = 2; L <= 32; L += 2)
    for (unsigned long long off = 0; off < 16; ++off) printf("%d %llu %d\n", L, off, pb::ea_readout_sites(L, 4096 + off));
  return 0; }'''


def test_store_width_fits_the_address(tmp_path):
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.isdir(d)), None)
    if cuda is None:
        pytest.skip("CUDA headers not available")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2510_23419_gb300", "csrc"), "-I", os.path.join(cuda, "include"),
                           str(src), "-o", str(exe)])
    rows = [tuple(map(int, l.split())) for l in subprocess.check_output([str(exe)]).decode().splitlines()]
    assert len(rows) == 16 * 16
    for L, off, v in rows:
        size = max(1, 2 * v)  # bytes per store
        starts = off + np.arange(0, 4 * L, size)  # stores of four rows; replicas and planes are whole rows
        assert np.all(starts % size == 0) and (v == 0 or L // 2 % v == 0), (L, off, v)
        if off == 0:  # an aligned output keeps the widest stores that the rows allow
            assert v == (4 if L % 8 == 0 else 2 if L % 4 == 0 else 1)


@pytest.mark.gpu
@pytest.mark.parametrize("L,R", [(2, 5), (4, 9), (6, 33), (8, 13), (12, 6), (16, 20), (32, 3)])
def test_outputs_at_any_offset(L, R):
    import torch
    from paper_2510_23419_gb300 import _build, native as pb
    _build.build()
    pb.load()
    N, S, seed, pad = L ** 3, 12, 4, 64
    J = syn.ea_couplings(L, "pm1", L)
    sc = pb.make_schedule(pb.PB_SCHED_LINEAR, S, 0.2, 2.0)
    want = pb.anneal(pb.PB_TOPO_EA3D, J, sc, R, seed, L=L, form=pb.PB_FORM_RESIDENT)
    Jd = torch.from_numpy(np.ascontiguousarray(J)).cuda()
    E = torch.empty((2, R), dtype=torch.float64, device="cuda")
    sweep = torch.empty(R, dtype=torch.int32, device="cuda")
    arena = torch.empty(2 * (R * N + 2 * pad), dtype=torch.int8, device="cuda")
    for best_off, final_off in ((0, 1), (1, 0), (2, 4), (3, 6), (4, 2), (5, 7), (8, 8)):
        arena.fill_(77)
        at = (pad + best_off, 3 * pad + R * N + final_off)
        pb.pb_anneal_ea_noalloc(L, Jd.data_ptr(), sc, R, seed, E[0].data_ptr(), sweep.data_ptr(),
                                arena.data_ptr() + at[0], E[1].data_ptr(), arena.data_ptr() + at[1],
                                stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        got = arena.cpu().numpy()
        for k, key in enumerate(("best_state", "final_state")):
            assert np.array_equal(got[at[k]:at[k] + R * N].reshape(R, N), want[key]), (best_off, final_off, key)
            got[at[k]:at[k] + R * N] = 77
        assert np.all(got == 77)  # nothing outside the outputs
        assert np.array_equal(E[0].cpu().numpy(), want["best_E"]) and np.array_equal(E[1].cpu().numpy(), want["final_E"])
        assert np.array_equal(sweep.cpu().numpy(), want["best_sweep"])
