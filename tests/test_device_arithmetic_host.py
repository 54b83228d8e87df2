"""The kernels' own cell and face arithmetic, compiled for the host
(tests/hostdevice.py), at the edges of its range, against the textbook HLLC flux
of the oracle and against plain FP64 formulas.  CPU only."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests.hostdevice import HostDevice


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return HostDevice(tmp_path_factory.mktemp("hostdevice"), small_rho=1e-150, small_p=1e-300)


def test_root_plus_a_far_smaller_number(dev):
    """s / (s + b): a root lies up to three units of 2^-62 below an exact power of
    two, and so does the sum where b is too small to lift it.  The result is
    rounded once from a chain within 2^-57: one ulp."""
    k = np.arange(0, 200)
    a, b = np.meshgrid(np.exp2(np.array([-300.0, -2.0, 0.0, 4.0, 200.0])), np.exp2(-k.astype(float)), indexing="ij")
    s = np.sqrt(a)
    r = dev.weight(a.ravel(), (b * s).ravel()).reshape(a.shape)
    ref = 1.0 / (1.0 + b)
    assert np.max(np.abs(r - ref)) <= np.spacing(1.0)


@pytest.mark.parametrize("ul,ur", [(0.0, 0.0), (0.5, 0.25), (-3.0, 2.0), (40.0, 39.0)])
def test_hllc_between_densities_far_apart(dev, ul, ur):
    """Density and pressure 1 beside 2^-k, at rest and moving: every flux within
    1e-13 of the largest one of the textbook form (that of the face checks)."""
    for k in range(0, 300, 5):
        q = 2.0 ** -k
        a, b = np.array([1.0, ul, 0.1, 0.0, 1.0]), np.array([q, ur, 0.2, 0.0, q])
        for L, R in ((a, b), (b, a)):
            ref = orc.hllc(L, R)
            got = dev.hllc(L, R)[0]
            assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref)), (k, got, ref)


# magnitudes whose squares, products or E + p leave the range of a double
OVERFLOWS = [
    ([1.0, 0.1, 2e154, 0.0, 1.0], [1.0, 0.1, 2e154, 0.0, 1.0], [4]),              # |v|^2
    ([1e10, 0.1, 1e151, 0.0, 1.0], [1e10, 0.1, 1e151, 0.0, 1.0], [4]),            # rho |v|^2
    ([1.0, 0.5, 0.0, 0.0, 1e306], [1.0, 0.5, 0.0, 1.8e154, 1e306], range(5)),      # |u_L - u_R|^2
    ([1e200, 3e119, 0.0, 0.0, 1e300], [1e200, -3e119, 0.0, 0.0, 1e300], [4]),      # rho u^2, m u
    ([1.0, 2e154, 0.0, 0.0, 1.0], [1.0, -2e154, 0.0, 0.0, 1.0], range(5)),
]


@pytest.mark.parametrize("L,R,where", OVERFLOWS)
def test_an_overflow_in_a_flux_stays_visible(dev, L, R, where):
    """Finite states whose flux overflows: the components of it that the textbook
    form gives as an infinity or NaN are not finite numbers."""
    L, R = np.array(L), np.array(R)
    for a, b in ((L, R), (R, L)):
        ref, got = orc.hllc(a, b), dev.hllc(a, b)[0]
        for v in where:
            assert not np.isfinite(ref[v]) and not np.isfinite(got[v]), (v, got, ref)


def test_a_quotient_that_rounds_up_to_the_end_of_the_range(dev):
    """m / rho next to 2^1024: a number there or an infinity, never a zero."""
    for sign in (1.0, -1.0):
        for k in range(-8, 9):
            W, _, _ = dev.prim([2.0 ** -24 * (1.0 + k * 2.0 ** -52), sign * np.nextafter(2.0 ** 1000, 0.0), 0.0, 0.0, 1.0])
            u = sign * W[0, 1]
            assert u >= 2.0 ** 1023 * 1.999999, (k, u)
            if k > 1:
                assert np.isfinite(u)
            if k < -1:
                assert np.isinf(u)


def test_the_kinetic_energy_overflow_of_a_cell(dev):
    """m^2 / rho past the range is an infinite kinetic energy: the pressure is the
    floor, the velocity and the CFL speed are those of the momentum."""
    for m in (1e155, 3.3e170, 1.7e200, -4.4e300):
        for y in (0.0, 1e154):
            W, hit, s = dev.prim([1.0, m, y, 0.0, 2.5])
            assert W[0, 1] == m and W[0, 4] == 1e-300 and hit[0] == 1
            assert s[0] >= abs(m) and np.isfinite(s[0])
    W, hit, s = dev.prim([1e-100, 1e300, 0.0, 0.0, 1.0])
    assert W[0, 1] == np.inf and W[0, 4] == 1e-300 and s[0] == np.inf
