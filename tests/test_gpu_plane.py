"""Plane form of the FFT step (N = 48, 64, 96): against the four-pass form and the FP64 oracle, the
k-space energies of excited states, and a batch against the lattices alone.

Tolerances as for the other FFT forms: a step stays within 2e-6 (1 + log2 N) of FP64 in the
2-norm; energies within 1e-5.  A batch member runs the launches it runs alone: bitwise.
"""
import math

import numpy as np
import pytest

from oracle import qfdtd_oracle as O
from paper_2211_10185_gb300 import inputs as I

pytestmark = pytest.mark.gpu
SIZES = [48, 64, 96]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2211_10185_gb300 import build

    build.build()


def _lattice(n, kind, complex_v, plane=True, seed=None):
    from paper_2211_10185_gb300.lattice import Lattice

    a = 6.0 / n
    v = I.cornell(n, a, 0.45, 0.2)
    if complex_v:
        v = v - 0.07j * np.abs(v)
    psi0 = I.gaussian_field(n, n if seed is None else seed)
    lat = Lattice(n, a, precision="c64")
    lat.set_potential(v)
    lat.set_kinetic(kind, 0.9)
    lat.set_wavefunction(psi0)
    lat.use_two_pass_fft(plane)
    return lat, (a, v, psi0)


def _rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("kind", [O.FFT_NAIVE, O.FFT_SYMANZIK, O.FFT_REL])
@pytest.mark.parametrize("n", SIZES)
def test_plane_steps_match_four_pass_and_oracle(n, kind, complex_v):
    steps, tol = 5, 2e-6 * (1 + math.log2(n)) * 5
    plane, (a, v, psi0) = _lattice(n, kind, complex_v)
    four, _ = _lattice(n, kind, complex_v, plane=False)
    assert plane.info()["fft_passes"] == 2 and four.info()["fft_passes"] == 4
    ref = O.Lattice(n, a)
    ref.set_potential(v.real, v.imag if complex_v else None)
    ref.set_kinetic(kind, 0.9)
    ref.set_wavefunction(psi0)
    for x in (plane, four):
        x.step_n(steps, tol=0.0, check_every=2, snap_every=2)
    ref.step_n(steps, check_every=2, snap_every=2)
    assert _rel(plane.get_wavefunction(), ref.psi) < tol
    assert _rel(four.get_wavefunction(), ref.psi) < tol
    er = ref.energies()["e"]
    assert abs(plane.energies()["e"] - er) < 1e-5 * abs(er)
    # energies of states: position space in the four-pass form, k-space here
    for p, q in zip(plane.project_excited(2), four.project_excited(2)):
        assert abs(p["e"] - q["e"]) < 1e-5 * abs(q["e"])


def test_plane_members_of_a_batch_match_alone_bitwise():
    from paper_2211_10185_gb300.serve import Batch

    specs = [(48, O.FFT_REL, False), (64, O.FFT_NAIVE, True), (96, O.FFT_SYMANZIK, False), (48, O.FFT_NAIVE, False),
             (64, O.FFT_REL, True)]
    alone = [_lattice(*s, seed=i)[0] for i, s in enumerate(specs)]
    mixed = [_lattice(*s, seed=i)[0] for i, s in enumerate(specs)]
    for lat in alone:
        lat.step_n(70, tol=0.0, check_every=32, snap_every=32)
    b = Batch()
    for lat in mixed:
        b.add(lat, 70, 0.0)
    while b.step(35, check_every=32) > 0:
        pass
    for la, lm in zip(alone, mixed):
        assert np.array_equal(la.get_wavefunction(), lm.get_wavefunction())
        assert la.energies()["e"] == lm.energies()["e"]
