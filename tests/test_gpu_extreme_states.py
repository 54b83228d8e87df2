"""Stages and time steps on states at the edges of the accepted range, against
the oracle or against the plain definition."""
import numpy as np
import pytest
import torch

import workloads as wl
from oracle.oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2401_03378_gb300 as gb
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gb


def state(lat, rho, u, v, w, p):
    return np.ascontiguousarray(np.moveaxis(wl.conserved(rho, u, v, w, p, 1.4), 0, 1))


@pytest.mark.parametrize("k", [40, 120, 130, 140])
@pytest.mark.parametrize("u1,u2", [(0.0, 0.0), (0.5, 0.25)])
def test_a_power_of_two_floor_beside_unit_density(gb, k, u1, u2):
    """Half the domain at density and pressure 1, the other half at the floors
    2^-k: one stage, within 1e-13 of each variable's largest value."""
    lat = wl.lattice_2d(4, 4, 8, 8, 4, bc="periodic")
    X, Y, _ = wl.cell_centers(lat)
    q = np.where(X < 0.5, 1.0, 2.0 ** -k)
    z = np.zeros_like(q)
    U = state(lat, q, np.where(X < 0.5, u1, u2), z, z, q)
    kw = dict(small_rho=2.0 ** -k, small_p=2.0 ** -(k + 60))
    h, o = gb.Hydro.from_lattice(lat, **kw), Oracle(lat, **kw)
    dt = 0.2 * lat.dx[0]
    Ud = torch.from_numpy(U.copy()).cuda()
    out = torch.zeros_like(Ud)
    h.stage(Ud, None, out, dt, 0.0, 1.0)
    Uf, ref = U.copy(), np.zeros_like(U)
    o.fill_guardcells(Uf)
    o.stage(Uf, U, ref, dt, 0.0, 1.0)
    zs, ys, xs = lat.interior_slices()
    got = out.cpu().numpy()
    for v in range(5):
        a, b = got[:, v, zs, ys, xs], ref[:, v, zs, ys, xs]
        assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(b)), v


@pytest.mark.parametrize("k", [-400, 300, 500, 511, 530, 600, 900])
def test_scaled_states(gb, k):
    """The update is homogeneous in (rho, momentum, E): a state times 2^k gives
    2^k times the result, and the same vector-Jacobian product."""
    lat = wl.lattice_2d(3, 3, 8, 8, 4, bc="periodic")
    U0 = wl.random_state(lat, seed=11, rough=False)
    rng = np.random.default_rng(12)
    M = torch.from_numpy(rng.normal(size=U0.shape)).cuda()
    h = gb.Hydro.from_lattice(lat, small_rho=1e-150, small_p=1e-200)
    zs, ys, xs = lat.interior_slices()
    res = []
    for s in (1.0, 2.0 ** k):
        U = torch.from_numpy(U0 * s).cuda()
        out, lam = torch.zeros_like(U), torch.zeros_like(U)
        h.stage(U, None, out, 1e-3, 0.0, 1.0)
        h.stage_vjp(U, M, 1e-3, out=lam)
        res.append((out[:, :, zs, ys, xs].cpu().numpy() / s, lam[:, :, zs, ys, xs].cpu().numpy()))
    (a, la), (b, lb) = res
    assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(a))
    assert np.max(np.abs(la - lb)) <= 1e-12 * np.max(np.abs(la))


@pytest.mark.parametrize("ndim,var", [(2, 1), (2, 2), (3, 1), (3, 2), (3, 3)])
@pytest.mark.parametrize("x", [np.inf, -np.inf])
@pytest.mark.parametrize("n", [4, 16])
def test_an_infinite_momentum_leaves_no_time_step(gb, ndim, var, x, n):
    lat = wl.lattice_2d(3, 2, n, n, 4) if ndim == 2 else wl.lattice_3d(2, 2, 2, n, n, 6, 4)
    U = wl.random_state(lat, seed=3, rough=False)
    U[4, var, lat.gz, 4 + 1, 4 + 2] = x
    assert float(gb.Hydro.from_lattice(lat).compute_dt(torch.from_numpy(U).cuda())[0]) == 0.0


def test_the_time_step_of_a_gas_beyond_2_to_the_1017(gb):
    lat = wl.lattice_2d(2, 2, 8, 8, 4, bc="periodic")
    one = np.ones((lat.nblocks,) + lat.padded)
    U = state(lat, one, 0 * one, 0 * one, 0 * one, 4e306 * one)
    dt = float(gb.Hydro.from_lattice(lat).compute_dt(torch.from_numpy(U).cuda())[0])
    assert abs(dt / (0.8 / (2 * np.sqrt(1.4 * 4e306) / lat.dx[0])) - 1.0) <= 1e-14


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_a_flow_whose_sound_speed_is_lost(gb, sign):
    """u + c = u: the contact speed has no value.  The cells are not finite afterwards;
    they are not ones whose mass has stopped moving."""
    lat = wl.lattice_2d(2, 2, 8, 8, 4, bc="periodic")
    rng = np.random.default_rng(8)
    rho = 2.0 ** rng.integers(0, 2, (lat.nblocks,) + lat.padded)      # so that m / rho is u
    U = state(lat, rho, sign * 1e10 + 0 * rho, 0 * rho, 0 * rho, 1e-14 + 0 * rho)
    h = gb.Hydro.from_lattice(lat)
    out = torch.zeros(lat.shape, dtype=torch.float64, device="cuda")
    h.stage(torch.from_numpy(U).cuda(), None, out, 1e-13, 0.0, 1.0)
    zs, ys, xs = lat.interior_slices()
    assert not torch.isfinite(out[:, 0, zs, ys, xs]).any()
