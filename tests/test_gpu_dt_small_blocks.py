"""compute_dt on blocks of fewer cells than a CTA has threads: the value, and its
time against the same cells in blocks of 16^2."""
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


@pytest.mark.parametrize("lat", [wl.lattice_2d(1, 1, 4, 4, 2), wl.lattice_2d(5, 7, 4, 4, 4), wl.lattice_2d(16, 17, 4, 4, 3),
                                 wl.lattice_2d(3, 5, 8, 8, 4), wl.lattice_3d(3, 3, 2, 4, 4, 4, 2),
                                 wl.lattice_3d(2, 5, 3, 4, 4, 10, 4), wl.lattice_3d(3, 2, 2, 8, 8, 3, 2),
                                 wl.lattice_3d(2, 2, 3, 4, 4, 16, 4), wl.lattice_3d(2, 2, 3, 4, 4, 15, 4)],
                         ids=lambda l: f"{l.n}x{l.nblocks}")
def test_every_cell_counts(gb, lat):
    """The fastest cell moved over the lattice: each block, each corner of it."""
    U0 = wl.random_state(lat, seed=3, rough=True)
    h, o = gb.Hydro.from_lattice(lat), Oracle(lat)
    gz = lat.ng if lat.ndim == 3 else 0
    nz, ny, nx = (lat.n[2] if lat.ndim == 3 else 1), lat.n[1], lat.n[0]
    spots = [(0, 0, 0), (nz - 1, ny - 1, nx - 1), (nz // 2, ny // 2, 1)]
    for b in sorted({0, lat.nblocks - 1, lat.nblocks // 2, min(15, lat.nblocks - 1), min(16, lat.nblocks - 1)}):
        for k, j, i in spots:
            U = U0.copy()
            U[b, 4, gz + k, lat.ng + j, lat.ng + i] *= 1e6
            got = float(h.compute_dt(torch.from_numpy(U).cuda())[0])
            ref = float(o.compute_dt(U))
            assert abs(got / ref - 1.0) <= 1e-15 * 4, (b, k, j, i)


@pytest.mark.parametrize("n", [4, 8])
def test_small_blocks_take_no_longer_per_cell(gb, n):
    """2^20 cells in blocks of n^2 against blocks of 16^2: 219 us against 33 for n = 4
    with a CTA to each block.  The bound covers the smaller rows of a block."""
    us = []
    for m in (16, n):
        lat = wl.lattice_2d(1024 // m, 1024 // m, m, m, 4, bc="periodic")
        h = gb.Hydro.from_lattice(lat)
        U = torch.ones((lat.nblocks, 5) + tuple(lat.padded), dtype=torch.float64, device="cuda")
        dt = h.compute_dt(U)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(8):
            e0.record()
            for _ in range(5):
                h.compute_dt(U, dt)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1) / 5 * 1e3)
        us.append(best)
        h.close()
        del U
    assert us[1] <= (2.5 if n == 4 else 1.6) * us[0], us
