"""The reciprocal and square root of the integer pipes, on the GPU, at the edges
of their argument ranges: mantissas next to powers of two over the exponent
range, both exponent parities, and the arguments that give NaN.

Tolerance: the functions are within 0.52 and 0.56 ulp of the exact value
(gbh_intmath.cuh), so they differ from the IEEE results by at most one ulp.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2401_03378_gb300 as gb
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gb


def selftest(gb, x):
    xd = torch.from_numpy(x).cuda()
    out = torch.empty(6 * len(x), dtype=torch.float64, device="cuda")
    assert gb.load().gbh_fastmath_selftest(xd.data_ptr(), out.data_ptr(), len(x),
                                           torch.cuda.current_stream().cuda_stream) == 0
    return out.cpu().numpy().reshape(6, -1)


def edge_arguments():
    k = np.arange(-1000, 1001, dtype=np.float64)
    base = np.exp2(k)
    steps = [0, 1, 2, 3, 2 ** 20, 2 ** 28, 2 ** 29, 2 ** 32, 2 ** 51, -1, -2, -(2 ** 20), -(2 ** 29)]
    bits = base.view(np.int64)
    return np.concatenate([(bits + s).view(np.float64) for s in steps])


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_reciprocal_and_root_edges(gb, sign):
    x = sign * edge_arguments()
    o = selftest(gb, x)
    for r in ((0, 4) if sign > 0 else (0,)):
        fast, ieee = o[r], o[r + 1]
        assert np.max(np.abs(fast - ieee) / np.spacing(np.abs(ieee))) <= 1.0, r
    if sign > 0:
        # powers of two are exact, and powers of four have exact roots
        p = np.exp2(np.arange(-1000, 1001, 2, dtype=np.float64))
        q = selftest(gb, p)
        assert np.array_equal(q[0], 1.0 / p) and np.array_equal(q[4], np.sqrt(p))
    else:
        assert np.all(np.isnan(o[4]))


def test_arguments_without_a_result(gb):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310])
    o = selftest(gb, x)
    assert np.all(np.isnan(o[0])) and np.all(np.isnan(o[4]))


@pytest.mark.parametrize("span,mach", [(0.0, 0.0), (2.0, 0.0), (8.0, 0.5), (8.0, 50.0)])
def test_wave_speeds_over_wide_ranges(gb, span, mach):
    """One stage on states whose densities and pressures differ by up to
    10^(2 span) between neighbouring cells, at rest and up to high Mach numbers,
    against the oracle.  Bound: the 1e-13 of a single step (relative to each
    variable's largest value, exact zero where the oracle's variable is zero)."""
    import workloads as wl
    from oracle.oracle import Oracle
    lat = wl.lattice_2d(4, 4, 8, 8, 4, bc="periodic")
    rng = np.random.default_rng(5)
    sh = (lat.nblocks,) + lat.padded
    rho = 10.0 ** rng.uniform(-span, span, sh)
    p = 10.0 ** rng.uniform(-span, span, sh)
    c = np.sqrt(1.4 * p / rho)
    u, v = (mach * c * rng.uniform(-1, 1, sh) for _ in range(2))
    U = np.ascontiguousarray(np.moveaxis(wl.conserved(rho, u, v, np.zeros(sh), p, 1.4), 0, 1))
    h = gb.Hydro.from_lattice(lat)
    o = Oracle(lat)
    Ud = torch.from_numpy(U).cuda()
    dt = float(np.ravel(o.compute_dt(U))[0])
    assert abs(float(h.compute_dt(Ud)[0]) / dt - 1.0) < 1e-15 * 4
    got = torch.zeros_like(Ud)
    h.stage(Ud, None, got, dt, 0.0, 1.0)
    Uf = U.copy()
    o.fill_guardcells(Uf)
    ref = np.zeros_like(U)
    o.stage(Uf, U, ref, dt, 0.0, 1.0)
    zs, ys, xs = lat.interior_slices()
    for k in range(5):
        a, b = got.cpu().numpy()[:, k, zs, ys, xs], ref[:, k, zs, ys, xs]
        m = np.max(np.abs(b))
        assert (np.max(np.abs(a - b)) <= 1e-13 * m) if m > 0 else np.all(a == 0), k


@pytest.mark.parametrize("var", range(5))
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_cell_stays_visible(gb, var, bad):
    """A NaN or infinity in any conserved variable of a cell is not swallowed: the
    cell is not finite after a stage, nor is a neighbour it exchanges flux with."""
    import workloads as wl
    lat = wl.lattice_2d(2, 2, 8, 8, 4, bc="periodic")
    U = wl.random_state(lat, seed=3, rough=False)
    U[1, var, 0, 4 + 3, 4 + 4] = bad
    h = gb.Hydro.from_lattice(lat)
    Ud = torch.from_numpy(U).cuda()
    out = torch.zeros_like(Ud)
    h.stage(Ud, None, out, 1e-4, 0.0, 1.0)
    r = torch.isfinite(out[1, :, 0, 4:-4, 4:-4]).all(0).cpu().numpy()
    assert not r[3, 4]
    assert not (r[2, 4] and r[4, 4] and r[3, 3] and r[3, 5])
