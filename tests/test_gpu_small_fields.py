"""Fields that sit on few sites: start fields of served requests (a Gaussian narrower than two sites of a
heavy particle) after a check interval of 64 steps, against the FP64 oracle.

With few sites that matter, and those of one distance from the origin rounding alike, the roundings
of the field do not average out.  Tolerance: two of 2^-24 a step, adding up over 64 steps as
independent ones: 2 x 2^-24 x 8 = 9.5e-7.
"""
import math

import numpy as np
import pytest

from oracle import qfdtd_oracle as O
from paper_2211_10185_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 2 * 2.0 ** -24 * 8


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2211_10185_gb300 import build

    build.build()


def _request(n, seed):
    """Mass, potential and start field of a request in a box of 16, from the seed."""
    mass = float(np.random.default_rng(1000 * n + seed).uniform(0.3, 5.0))
    rng, a = np.random.default_rng(seed * 100 + n), 16.0 / n
    v = I.cornell(n, a, float(rng.uniform(0.3, 0.6)), float(rng.uniform(0.1, 0.25)))
    w = float(np.random.default_rng(seed * 100 + n).uniform(0.5, 2.0)) / math.sqrt(mass)
    x = ((np.arange(n) - n // 2) * a) ** 2
    return a, mass, v, np.exp(-0.5 * (x[:, None, None] + x[:, None] + x) / w ** 2).astype(np.complex128)


def _check(n, kind, seed):
    from paper_2211_10185_gb300.lattice import Lattice

    a, mass, v, psi = _request(n, seed)
    lat, ref = Lattice(n, a, precision="c64"), O.Lattice(n, a)
    for x in (lat, ref):
        x.set_potential(v)
        x.set_kinetic(kind, mass)
        x.set_wavefunction(psi)
        x.step_n(64, check_every=64, snap_every=0)
    got, want = lat.get_wavefunction(), ref.psi
    assert np.linalg.norm((got - want).ravel()) < TOL * np.linalg.norm(want.ravel())


@pytest.mark.parametrize("n,kind,seed", [(32, O.FFT_NAIVE, 3), (32, O.FFT_NAIVE, 1), (32, O.FFT_SYMANZIK, 3),
                                         (48, O.FFT_SYMANZIK, 4), (64, O.FFT_NAIVE, 2)])
def test_narrow_fields_of_heavy_particles(n, kind, seed):
    _check(n, kind, seed)


@pytest.mark.parametrize("n,seed", [(32, 18), (32, 1), (48, 4), (64, 1)])
def test_heavy_relativistic_particles(n, seed):
    """Eq. HK3 with T(k) close to the mass for all k that matter."""
    _check(n, O.FFT_REL, seed)
