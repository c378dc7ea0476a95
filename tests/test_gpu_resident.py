"""Resident FFT steps (small complex-FP32 lattices, many steps per launch): every size, kinetic
term and kind of potential against the four-pass form and the FP64 oracle, launches of
different lengths against one, and the allocation-free step.

Tolerances: a step's transforms carry about log2(N) roundings each way on top of the update's,
so a step stays within 2e-6 (1 + log2 N) of FP64 in the 2-norm and s steps within s times
that (the tolerance of the other FFT tests).  How the steps are cut into launches changes no
operation: bitwise.
"""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import qfdtd_oracle as O
from paper_2211_10185_gb300 import inputs as I
from paper_2211_10185_gb300 import qfdtd as Q

pytestmark = pytest.mark.gpu
SIZES = [8, 12, 16, 24, 32]


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
    return a, v, I.gaussian_field(n, n)


def _gpu(n, a, v, psi0, kind, resident=True):
    from paper_2211_10185_gb300.lattice import Lattice

    lat = Lattice(n, a, precision="c64")
    lat.set_potential(v)
    lat.set_kinetic(kind, 0.9)
    lat.set_wavefunction(psi0)
    lat.use_two_pass_fft(resident)  # (off: the four-pass form)
    return lat


def _rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("kind", [O.FFT_NAIVE, O.FFT_SYMANZIK, O.FFT_REL])
@pytest.mark.parametrize("n", SIZES)
def test_resident_steps_match_four_pass_and_oracle(n, kind, complex_v):
    a, v, psi0 = _inputs(n, complex_v)
    steps, tol = 7, 2e-6 * (1 + math.log2(n)) * 7
    ref = O.Lattice(n, a)
    ref.set_potential(v.real, v.imag if complex_v else None)
    ref.set_kinetic(kind, 0.9)
    ref.set_wavefunction(psi0)
    ref.step_n(steps, check_every=4, snap_every=0)
    got = {}
    for resident in (True, False):
        lat = _gpu(n, a, v, psi0, kind, resident)
        lat.step_n(steps, tol=0.0, check_every=4, snap_every=0)
        got[resident] = lat.get_wavefunction()
        assert _rel(got[resident], ref.psi) < tol
        assert abs(lat.energies()["e"] - ref.energies()["e"]) < 1e-5 * abs(ref.energies()["e"])
    assert _rel(got[True], got[False]) < 2 * tol


@pytest.mark.parametrize("n", SIZES)
def test_cutting_steps_into_launches_changes_no_bit(n):
    a, v, psi0 = _inputs(n, False)
    one, many = _gpu(n, a, v, psi0, O.FFT_SYMANZIK), _gpu(n, a, v, psi0, O.FFT_SYMANZIK)
    one.step_n(40, tol=0.0, check_every=16, snap_every=0)
    for k in (1, 2, 13, 1, 23):
        many.step_n(k, tol=0.0, check_every=16, snap_every=0)
    assert np.array_equal(one.get_wavefunction(), many.get_wavefunction())
    assert one.energies() == many.energies()


@pytest.mark.parametrize("complex_v", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_allocation_free_step_matches_resident_step(n, complex_v):
    import torch

    a, v, psi0 = _inputs(n, complex_v)
    lat = _gpu(n, a, v, psi0, O.FFT_REL)
    dt = lat.info()["dtau"]
    lat.step_n(1, tol=0.0, check_every=0, snap_every=0)
    psi = torch.from_numpy(psi0).to(torch.complex64).cuda()
    vd = torch.from_numpy(v).to(torch.complex64 if complex_v else torch.float32).cuda()
    sums = torch.empty(5, dtype=torch.float64, device="cuda")
    st = Q.load().qf_fft_step_static(n, a, O.FFT_REL, 0.9, dt, C.c_void_p(psi.data_ptr()), C.c_void_p(vd.data_ptr()),
                                     int(complex_v), 1.0, C.c_void_p(sums.data_ptr()), None)
    assert st == Q.QF_OK
    torch.cuda.synchronize()
    # (one step of the same arithmetic in another instantiation, and the sums of its input)
    assert _rel(psi.cpu().numpy().astype(np.complex128), lat.get_wavefunction()) < 2e-6 * (1 + math.log2(n))
    assert abs(sums[0].item() - np.linalg.norm(psi0) ** 2) < 1e-6 * np.linalg.norm(psi0) ** 2


def test_resident_steps_whose_waits_run_out_end_and_say_so():
    """The self-test runs resident steps that give up at their first wait; the lattice steps on as if
    it had not been called, and so does one that shares the GPU."""
    a, v, psi0 = _inputs(32, False)
    plain, probed = _gpu(32, a, v, psi0, O.FFT_REL), _gpu(32, a, v, psi0, O.FFT_REL)
    for lat in (plain, probed):
        lat.step_n(5, tol=0.0, check_every=4, snap_every=0)
    assert probed.lib.qf_selftest_bounded_wait(probed.h) == Q.QF_ETIMEOUT
    for lat in (plain, probed):
        lat.step_n(6, tol=0.0, check_every=4, snap_every=0)
    assert np.array_equal(plain.get_wavefunction(), probed.get_wavefunction())


def _set_error_flag(lat):
    """Sets the flag that a run-out wait sets: the last int pair but one double of the scalars, which
    lie before the staging area at the workspace's end (256-byte multiples)."""
    import torch

    up = lambda x: (x + 255) // 256 * 256
    total, scalars = lat.info()["workspace_bytes"], 32 * 8
    at = total - up(min(16 * lat.n ** 3, 32 << 20)) - up(scalars) + scalars - 16
    flag = lat.workspace[at:at + 8].view(torch.int32)
    assert flag.tolist() == [0, 0]
    torch.cuda.synchronize()
    flag[0] = 1
    torch.cuda.synchronize()
    return flag


def test_a_run_out_wait_is_reported_once_by_steps_and_batches():
    from paper_2211_10185_gb300.serve import Batch

    a, v, psi0 = _inputs(16, False)
    lat = _gpu(16, a, v, psi0, O.FFT_REL)
    flag = _set_error_flag(lat)
    with pytest.raises(Q.QFError) as e:
        lat.step_n(3, tol=0.0, check_every=0, snap_every=0)
    assert e.value.status == Q.QF_ETIMEOUT and flag.tolist() == [0, 0]
    lat.step_n(3, tol=0.0, check_every=0, snap_every=0)
    b = Batch()
    b.add(lat, 100, 0.0)
    _set_error_flag(lat)
    with pytest.raises(Q.QFError) as e:
        b.step(3, check_every=0)
    assert e.value.status == Q.QF_ETIMEOUT and flag.tolist() == [0, 0]
    b.step(3, check_every=0)


def test_a_batch_cuts_long_intervals_like_a_lattice_alone():
    """Intervals of 2100 steps: a launch takes 2048 at most, replayed from a graph too (per interval the
    check step, its finishing sums and two launches)."""
    from paper_2211_10185_gb300.serve import Batch

    a, v, psi0 = _inputs(8, False)
    alone, member = _gpu(8, a, v, psi0, O.FFT_SYMANZIK), _gpu(8, a, v, psi0, O.FFT_SYMANZIK)
    for lat in (alone, member):
        lat.set_kinetic(O.FFT_SYMANZIK, 0.9, 1e-3)  # (an interval decays by less than exp(-30))
    alone.step_n(4200, tol=0.0, check_every=2100, snap_every=0)
    b = Batch()
    b.add(member, 10000, 0.0)
    b.step(4200, check_every=2100, snap_every=0)
    assert np.isfinite(alone.get_wavefunction()).all()
    assert np.array_equal(alone.get_wavefunction(), member.get_wavefunction())
    n = C.c_int64()
    assert b.lib.qf_batch_info(b.h, C.byref(n)) == Q.QF_OK
    assert b.graph_info()[1] == 2 and n.value == 2 * 4
