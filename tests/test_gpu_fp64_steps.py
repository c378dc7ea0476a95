"""Complex-FP64 steps with a real potential against extended precision (numpy's long double, 64 bits
of mantissa at least), over enough steps that a rounding which is the same in every step adds up.

Tolerance: the roundings of a step that differ from step to step are within 2 x 2^-53 of the
field for the stencil and, with the transforms, within 4 x 2^-53 for Eq. HK3; 256 of them add up to
16 times that: 3.6e-15 and 7.2e-15.
"""
import numpy as np
import pytest

from oracle import qfdtd_oracle as O
from paper_2211_10185_gb300 import inputs as I

pytestmark = pytest.mark.gpu
STEPS = 256


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2211_10185_gb300 import build

    build.build()


def _extended(kind, n, a, mass, dt, v, psi):
    L = np.longdouble
    a, mass, w = L(a), L(mass), L(dt) / 2 * v.astype(L)
    p = psi.astype(np.clongdouble)
    j = np.arange(n)
    s = 4 * np.sin(np.arctan2(L(0), L(-1)) * np.where(j <= n // 2, j, j - n) / L(n)) ** 2
    t = np.sqrt(s[:, None, None] + s[None, :, None] + s[None, None, :] + (a * mass) ** 2) / a
    for _ in range(STEPS):
        if kind == O.FDTD:
            h = 6 * p
            for d in range(3):
                h = h - np.roll(p, 1, d) - np.roll(p, -1, d)
            h = h / (2 * mass * a * a)
        else:
            h = np.fft.ifftn(t * np.fft.fftn(p))
        p = ((1 - w) * p - L(dt) * h) / (1 + w)
        if kind == O.FDTD:
            p[0] = p[:, 0] = p[:, :, 0] = 0
    return p


@pytest.mark.parametrize("kind,n,a,seed,tol", [(O.FDTD, 20, 0.6, 1, 3.6e-15), (O.FDTD, 20, 0.6, 2, 3.6e-15),
                                               (O.FDTD, 18, 0.3, 3, 3.6e-15), (O.FFT_REL, 16, 0.25, 4, 7.2e-15)])
def test_many_fp64_steps_against_extended_precision(kind, n, a, seed, tol):
    from paper_2211_10185_gb300.lattice import Lattice

    v = I.cornell(n, a, 0.3 + 0.1 * seed, 0.2)
    psi = I.gaussian_field(n, seed)
    if kind == O.FDTD:
        psi = I.zero_dirichlet_planes(psi)
    lat = Lattice(n, a, precision="c128")
    lat.set_potential(v)
    lat.set_kinetic(kind, 0.9)
    lat.set_wavefunction(psi)
    lat.step_n(STEPS, tol=0.0, check_every=0, snap_every=0)
    ref = _extended(kind, n, a, 0.9, lat.info()["dtau"], v, psi)
    off = (lat.get_wavefunction().astype(np.clongdouble) - ref).ravel()
    assert float(np.sqrt((np.abs(off) ** 2).sum() / (np.abs(ref) ** 2).sum())) < tol


def test_setting_potential_or_time_step_returns_with_its_work_done():
    """A batch may step the lattice on another stream right after: nothing is left on the lattice's."""
    import ctypes as C

    from paper_2211_10185_gb300 import qfdtd as Q
    from paper_2211_10185_gb300.lattice import Lattice

    n = 160
    lat = Lattice(n, 0.1, precision="c128")
    v = np.ascontiguousarray(I.cornell(n, 0.1, 0.4, 0.2)).reshape(-1)
    lat.set_kinetic(O.FDTD, 1.0)
    lat.set_potential(v)
    for _ in range(20):
        assert lat.lib.qf_set_kinetic(lat.h, C.c_int(O.FDTD), C.c_double(1.0), C.c_double(0.001)) == Q.QF_OK
        assert lat.stream.query()
    for _ in range(3):
        assert lat.lib.qf_set_potential(lat.h, Q.dptr(v), None) == Q.QF_OK
        assert lat.stream.query()
