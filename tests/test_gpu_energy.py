"""Check energies of FFT lattices whose kinetic and potential energies nearly cancel.

An energy E = <T> + <V> with |E| << <T> shows every relative error of <T> enlarged by <T>/|E|.
N = 96 takes the four-pass form unless another is asked for: bit for bit.
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


def _lattice(n, a, kind, mass, v, psi, form=None):
    from paper_2211_10185_gb300.lattice import Lattice

    lat = Lattice(n, a, precision="c64")
    lat.set_potential(v)
    lat.set_kinetic(kind, mass)
    lat.set_wavefunction(psi)
    if form is not None:
        lat.use_two_pass_fft(form)
    return lat


@pytest.mark.parametrize("kind", [O.FFT_NAIVE, O.FFT_REL])
def test_n96_takes_the_four_pass_form_alone_and_in_a_batch(kind):
    from paper_2211_10185_gb300.serve import Batch

    n, a = 96, 1.0 / 6
    v, psi = I.cornell(n, a, 0.45, 0.2), I.gaussian_field(n, 3)
    plain, four, member = (_lattice(n, a, kind, 0.9, v, psi, form) for form in (None, False, None))
    assert plain.info()["fft_passes"] == 4
    for lat in (plain, four):
        lat.step_n(66, tol=0.0, check_every=32, snap_every=0)
    b = Batch()
    b.add(member, 66, 0.0)
    while b.step(33, check_every=32) > 0:
        pass
    for lat in (plain, member):
        assert np.array_equal(lat.get_wavefunction(), four.get_wavefunction())
        assert lat.energies() == four.energies()
