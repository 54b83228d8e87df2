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
