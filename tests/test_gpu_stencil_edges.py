"""FDTD kernels at the sizes where their tiles can go wrong: lattices narrower than, equal to
and just past a warp's 28 output columns and a block's 128 positions, row counts that the
rows of a warp do not divide, and the smallest lattice.

Tolerances: a site's update takes about 20 roundings, each within 2^-24 (2^-53) of terms no
larger than a few |psi|, so s steps stay within 2e-6 (1 + s) (1e-14 (1 + s)) of the FP64
oracle in the 2-norm.  Two steps in one pass are the same rounded operations as two single
steps: bitwise.
"""
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


def _inputs(n, complex_v):
    a = 6.0 / n
    v = I.cornell(n, a, 0.45, 0.2)
    if complex_v:
        v = v - 0.07j * np.abs(v)
    return a, v, I.zero_dirichlet_planes(I.gaussian_field(n, n))


def _run(n, a, v, psi0, prec, tblock, steps):
    from paper_2211_10185_gb300.lattice import Lattice

    lat = Lattice(n, a, precision=prec)
    lat.set_potential(v)
    lat.set_kinetic(O.FDTD, 1.1)
    lat.set_wavefunction(psi0)
    lat.set_temporal_blocking(tblock)
    lat.step_n(steps, tol=0.0, check_every=6, snap_every=0)
    return lat.get_wavefunction(), lat.energies()["e"]


def _oracle(n, a, v, psi0, steps):
    ref = O.Lattice(n, a)
    ref.set_potential(v.real, v.imag if np.iscomplexobj(v) else None)
    ref.set_kinetic(O.FDTD, 1.1)
    ref.set_wavefunction(psi0)
    ref.step_n(steps, check_every=6, snap_every=0)
    return ref.psi, ref.energies()["e"]


@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("n", [8, 10, 22, 28, 30, 34, 58, 126])
def test_complex_fp32_single_and_paired_steps(n, complex_v):
    a, v, psi0 = _inputs(n, complex_v)
    one, e1 = _run(n, a, v, psi0, "c64", 1, 11)
    two, e2 = _run(n, a, v, psi0, "c64", 2, 11)
    assert np.array_equal(one, two) and e1 == e2
    ref, er = _oracle(n, a, v, psi0, 11)
    assert np.linalg.norm((two - ref).ravel()) < 2e-6 * 12 * np.linalg.norm(ref.ravel())
    assert abs(e2 - er) < 1e-5 * abs(er)
    assert not two[0].any() and not two[:, 0].any() and not two[:, :, 0].any()


@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("n", [8, 10, 22, 34, 126])
def test_complex_fp64_steps(n, complex_v):
    a, v, psi0 = _inputs(n, complex_v)
    got, e = _run(n, a, v, psi0, "c128", 1, 11)
    ref, er = _oracle(n, a, v, psi0, 11)
    assert np.linalg.norm((got - ref).ravel()) < 1e-14 * 12 * np.linalg.norm(ref.ravel())
    assert abs(e - er) < 1e-12 * abs(er)
    assert not got[0].any() and not got[:, 0].any() and not got[:, :, 0].any()


@pytest.mark.parametrize("wall", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("n", [8, 30, 58, 200])
def test_potential_on_the_dirichlet_planes_is_not_used(n, complex_v, wall):
    """V there multiplies a psi that is zero: an infinite wall or no number changes no bit, in single
    steps and in pairs.  (200: with the prefetch of the larger sizes.)"""
    a, v, psi0 = _inputs(n, complex_v)
    walled = v.copy()
    w = complex(wall, wall) if complex_v else wall
    walled[0], walled[:, 0], walled[:, :, 0] = w, w, w
    want, e = _run(n, a, v, psi0, "c64", 1, 11)
    assert np.isfinite(want).all()
    for tblock in (1, 2):
        got, eg = _run(n, a, walled, psi0, "c64", tblock, 11)
        assert np.array_equal(got, want) and eg == e
