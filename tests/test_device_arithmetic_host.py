"""The kernels' own cell and face arithmetic, compiled for the host
(tests/hostdevice.py), at the edges of its range, against the textbook HLLC flux
of the oracle and against plain FP64 formulas.  CPU only."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests.hostdevice import HostDevice
from tests.test_hllc_arrangement import states


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


# beyond 2^1017, where the FP32 watch on the high words takes a number for an infinity
BEYOND = [[1.0, 0.0, 0.0, 0.0, 1e307], [1e306, 1e290, -1e290, 1e280, 1.7e308], [1e307, 1.0, 0.0, 0.0, 1.0],
          [1e307, 1e307, 0.0, 0.0, 1e307], [1.0, 1e300, 0.0, 0.0, 1e307], [1e306, 1e300, -1.7e308, 1e290, 1.7e308],
          [1e-100, 0.0, 2e306, 0.0, 1.0]]


@pytest.mark.parametrize("U", BEYOND)
def test_finite_states_beyond_2_to_the_1017(dev, U):
    """The CFL speed of finite states of any magnitude is that of the plain FP64
    formulas; a stage takes them for non-finite ones."""
    W, hit, s = dev.prim(U, inv_dx=(0.5, 0.25, 0.125), beyond=True)
    with np.errstate(over="ignore"):
        u = np.array(U[1:4]) / U[0]
        p = 0.4 * (U[4] - 0.5 * np.dot(U[1:4], u))
        c = np.sqrt(1.4 * max(p, 1e-300) / U[0])
        ref = c * 0.875 + np.abs(u) @ [0.5, 0.25, 0.125]
    assert W[0, 0] == U[0] and np.allclose(W[0, 1:4], u, rtol=4e-16, atol=0)
    assert W[0, 4] == 1e-300 if not p >= 1e-300 else abs(W[0, 4] / p - 1) < 1e-15
    assert s[0] == ref or abs(s[0] / ref - 1) < 1e-14
    assert np.all(np.isnan(dev.prim(U)[0][0, 1:4]))


@pytest.mark.parametrize("u", [0.0, 0.5, -0.25])
def test_a_flux_at_pressures_beyond_2_to_the_1017(dev, u):
    W = np.array([1.0, u, 0.1, 0.0, 1e307])
    ref, got = orc.hllc(W, W), dev.hllc(W, W)[0]
    assert np.all(np.isfinite(got)) and np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("k,x", [(k, x) for k in range(5) for x in (np.inf, -np.inf, np.nan)])
def test_a_non_finite_variable_of_a_cell(dev, k, x):
    """In a stage it makes the velocities NaN.  For the CFL speed an infinite momentum is an infinite velocity (dt = 0) at the
    pressure floor, and a NaN stays a NaN."""
    for E in (2.5, -2.5, 1e-3):
        U = np.array([1.0, 0.3, -0.2, 0.1, E])
        U[k] = x
        V, _, s = dev.prim(U)
        assert np.all(np.isnan(V[0, 1:4])) and (np.isnan(V[0, 4]) or V[0, 4] == 1e-300)
        W, _, _ = dev.prim(U, beyond=True)
        if 1 <= k <= 3 and np.isinf(x):
            assert W[0, k] == x and W[0, 4] == 1e-300 and s[0] == np.inf
            assert np.allclose(np.delete(W[0, 1:4], k - 1), np.delete(U[1:4], k - 1), rtol=1e-15)
        elif np.isnan(x):
            assert np.isnan(W[0, 4]) and np.isnan(s[0]) and (np.isnan(W[0, k]) or k == 0)
        elif k == 4:
            assert np.array_equal(W[0, :4], U[:4]) and W[0, 4] == (np.inf if x > 0 else 1e-300)
        elif x > 0:
            assert np.isnan(W[0, 4]) and np.isnan(s[0])


@pytest.mark.parametrize("v", range(5))
@pytest.mark.parametrize("x", [np.inf, -np.inf, np.nan])
def test_a_non_finite_face_state_has_no_flux(dev, v, x):
    a, b = np.array([1.0, 0.3, 0.1, 0.0, 1.0]), np.array([0.5, 0.2, 0.0, 0.1, 0.7])
    a[v] = x
    assert np.all(np.isnan(dev.hllc(a, b))) and np.all(np.isnan(dev.hllc(b, a)))


@pytest.mark.parametrize("u", [1e10, -1e10, 3e120, -7e16])
def test_both_sound_speeds_lost_in_the_velocities(dev, u):
    """u + c = u - c = u on both sides, where the contact speed is 0 / 0: no flux (NaN),
    not one of another speed."""
    for p, q in ((1e-14, 1e-14), (1e-30, 1e-14), (1e-300, 1e-20)):
        L, R = np.array([1.0, u, 0.1, 0.0, p]), np.array([0.7, u, 0.1, 0.0, q])
        for a, b in ((L, R), (R, L), (L, L)):
            assert np.all(np.isnan(dev.hllc(a, b)))
    # one side's is lost: the flux of the textbook form
    a, b = np.array([1.0, 1e10, 0.0, 0.0, 1e-14]), np.array([1.0, 1e10, 0.0, 0.0, 1e16])
    for L, R in ((a, b), (b, a)):
        ref = orc.hllc(L, R)
        assert np.max(np.abs(dev.hllc(L, R)[0] - ref)) <= 1e-13 * np.max(np.abs(ref))


def test_receding_states_with_both_sound_speeds_lost(dev):
    L, R = np.array([1.0, -1e10, 0.0, 0.0, 1e-14]), np.array([1.0, 1e10, 0.0, 0.0, 1e-14])
    assert np.all(np.isnan(orc.hllc(L, R))) and np.all(np.isnan(dev.hllc(L, R)))


def gas(n, seed, mach, jump):
    rng = np.random.default_rng(seed)
    rho, p = (10.0 ** rng.uniform(-jump, jump, n) for _ in range(2))
    c = np.sqrt(1.4 * p / rho)
    return np.stack([rho, *(mach * c * rng.uniform(-1, 1, n) for _ in range(3)), p], axis=1)


@pytest.mark.parametrize("seeds,mach,tol", [((1, 2), 0.8, 1e-13), ((3, 4), 10.0, 1e-12)])
def test_the_arrangement_of_the_kernels_against_the_textbook_flux(dev, seeds, mach, tol):
    """Weights s / (s + rho_R) and rho_R / (s + rho_R) with s = sqrt(rho_L rho_R), the
    Roe sound speed as a sum of non-negative terms, the star state through
    t = S* (S_K - u_K) / (S_K - S*): the states and bounds of
    test_hllc_arrangement.py (the textbook form's own rounding sets them)."""
    L, R = (np.array(states(2000, k, mach)) for k in seeds)
    got = dev.hllc(L, R)
    for a, b, f in zip(L, R, got):
        ref = orc.hllc(a, b)
        assert np.max(np.abs(f - ref)) <= tol * np.max(np.abs(ref))


def test_the_conversion_against_the_plain_formulas(dev):
    W0 = gas(3000, 3, 10.0, 2.0)
    rho, u, v, w, p = W0.T
    U = np.stack([rho, rho * u, rho * v, rho * w, 2.5 * p + 0.5 * rho * (u * u + v * v + w * w)], axis=1)
    W, hit, s = dev.prim(U)
    assert not hit.any() and np.array_equal(W[:, 0], rho)
    assert np.allclose(W[:, 1:4], U[:, 1:4] / rho[:, None], rtol=4e-16, atol=0)
    assert np.all(np.abs(W[:, 4] - p) <= 1e-15 * U[:, 4])
    ref = np.sqrt(1.4 * W[:, 4] / rho) * 6.0 + np.abs(W[:, 1]) + 2.0 * np.abs(W[:, 2]) + 3.0 * np.abs(W[:, 3])
    assert np.allclose(s, ref, rtol=4e-15, atol=0)
