"""Line-form passes of the FFT step (N = 192, 512) against the four-pass kernels, and at N = 192
against the FP64 oracle.

Tolerances as for the other FFT forms: a step stays within 2e-6 (1 + log2 N) of FP64 in the
2-norm, so two forms within twice that; energies within 1e-5.
"""
import math

import numpy as np
import pytest

from oracle import qfdtd_oracle as O
from paper_2211_10185_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2211_10185_gb300 import build

    build.build()


def _rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


@pytest.mark.parametrize("n,kind,complex_v", [(192, O.FFT_REL, False), (192, O.FFT_NAIVE, True),
                                              (512, O.FFT_SYMANZIK, False), (512, O.FFT_REL, True)])
def test_line_passes_match_four_pass_kernels(n, kind, complex_v):
    from paper_2211_10185_gb300.lattice import Lattice

    a, steps = 6.0 / n, 3
    v = I.cornell(n, a, 0.45, 0.2)
    if complex_v:
        v = v - 0.07j * np.abs(v)
    psi0 = I.gaussian_field(n, n)
    got, e = {}, {}
    for line in (True, False):
        lat = Lattice(n, a, precision="c64", n_snap=1)
        lat.set_potential(v)
        lat.set_kinetic(kind, 0.9)
        lat.set_wavefunction(psi0)
        lat.use_two_pass_fft(line)
        lat.step_n(steps, tol=0.0, check_every=2, snap_every=0)
        got[line], e[line] = lat.get_wavefunction(), lat.energies()["e"]
        lat.close()
    tol = 2e-6 * (1 + math.log2(n)) * steps
    assert _rel(got[True], got[False]) < 2 * tol
    assert abs(e[True] - e[False]) < 1e-5 * abs(e[False])
    if n == 192:
        ref = O.Lattice(n, a)
        ref.set_potential(v.real, v.imag if complex_v else None)
        ref.set_kinetic(kind, 0.9)
        ref.set_wavefunction(psi0)
        ref.step_n(steps, check_every=2, snap_every=0)
        assert _rel(got[True], ref.psi) < tol
        assert abs(e[True] - ref.energies()["e"]) < 1e-5 * abs(e[True])


def test_autotuner_times_the_passes_that_the_line_form_leaves():
    """One warm pass, then four rounds of two tile variants of the y passes (1 and 3) at N = 192, whose x
    and z passes run in the line form: 17 launches before the first step's five."""
    import ctypes as C

    from paper_2211_10185_gb300 import qfdtd as Q
    from paper_2211_10185_gb300.lattice import Lattice

    n, lib, old = 192, Q.load(), C.c_int()
    assert lib.qf_get_fft_tiles(n, C.byref(old)) == Q.QF_OK
    try:
        assert lib.qf_set_fft_tiles(n, -1) == Q.QF_OK
        lat = Lattice(n, 0.1, precision="c64")
        lat.set_potential(I.cornell(n, 0.1, 0.4, 0.2))
        lat.set_kinetic(O.FFT_REL, 1.0)
        lat.set_wavefunction(I.gaussian_field(n, 1))
        before = lat.info()["launches"]
        lat.step_n(1, tol=0.0, check_every=0, snap_every=0)
        assert lat.info()["launches"] - before == 1 + 4 * 2 * 2 + 5
    finally:
        lib.qf_set_fft_tiles(n, old.value)


def test_two_members_and_a_change_of_form_between_batch_steps():
    """N = 192 with Eq. HK2, two members a launch, the form switched off and on again between intervals
    that the batch replays from graphs: bit for bit what the lattices do alone."""
    from paper_2211_10185_gb300.lattice import Lattice
    from paper_2211_10185_gb300.serve import Batch

    n, a = 192, 1.0 / 12

    def pair():
        out = []
        for seed in (1, 2):
            lat = Lattice(n, a, precision="c64", n_snap=1)
            lat.set_potential(I.cornell(n, a, 0.3 + 0.1 * seed, 0.2))
            lat.set_kinetic(O.FFT_SYMANZIK, 0.8 + 0.1 * seed)
            lat.set_wavefunction(I.gaussian_field(n, seed))
            out.append(lat)
        return out

    alone, members = pair(), pair()
    b = Batch()
    for lat in members:
        b.add(lat, 1000, 0.0)
    for line in (True, False, True):
        for lat in alone + members:
            lat.use_two_pass_fft(line)
        b.step(16, check_every=8)
        for lat, mem in zip(alone, members):
            lat.step_n(16, tol=0.0, check_every=8, snap_every=8)
            assert np.array_equal(mem.get_wavefunction(), lat.get_wavefunction()), line
            assert mem.energies() == lat.energies()
    assert b.graph_info()[1] >= 5
