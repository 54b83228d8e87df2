"""The guard fill and the CFL reduction at the edges of their work splits: odd
guard widths, guards as wide as the block, more planes than the multiply-high
quotients cover, one block and many, blocks of every width; fill bitwise and dt
within one rounding of the oracle's, per problem on batched contexts."""
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


LATTICES = [
    wl.lattice_3d(1, 1, 1, 4, 4, 4, 2),
    wl.lattice_3d(3, 2, 2, 8, 8, 5, 3, bc=("periodic", "outflow", "outflow")),
    wl.lattice_3d(2, 2, 3, 16, 16, 17, 16, bc=("outflow", "periodic", "periodic")),
    wl.lattice_3d(1, 1, 1, 16, 16, 920, 16, bc=("outflow", "periodic", "outflow")),
    wl.lattice_3d(11, 12, 10, 4, 4, 4, 4, bc="periodic"),
    wl.lattice_2d(1, 1, 4, 4, 3),
    wl.lattice_2d(7, 5, 16, 16, 7, bc=("periodic", "outflow")),
    wl.lattice_2d(60, 50, 8, 8, 2, bc="periodic"),
]


@pytest.mark.parametrize("lat", LATTICES)
def test_fill_and_dt(gb, lat):
    rng = np.random.default_rng(7)
    sh = (lat.nblocks,) + lat.padded
    U0 = np.ascontiguousarray(np.moveaxis(
        wl.conserved(rng.uniform(0.5, 2, sh), *rng.uniform(-1, 1, (3,) + sh), rng.uniform(0.5, 2, sh), 1.4), 0, 1))
    U0 = wl.poison_guards(U0, lat)
    h, o = gb.Hydro.from_lattice(lat), Oracle(lat)
    U = torch.from_numpy(U0.copy()).cuda()
    dt = float(h.compute_dt(U)[0])
    h.fill_guardcells(U)
    ref = U0.copy()
    o.fill_guardcells(ref)
    assert np.array_equal(U.cpu().numpy(), ref)
    want = float(np.ravel(o.compute_dt(ref))[0])
    assert abs(dt / want - 1.0) <= 4 * np.finfo(float).eps


def test_dt_per_problem(gb):
    lats = [wl.lattice_2d(2, 3, 8, 8, 4, bc="periodic"), wl.lattice_2d(1, 1, 8, 8, 4), wl.lattice_2d(4, 4, 8, 8, 4)]
    states = [wl.random_state(l, seed=50 + i, rough=True) for i, l in enumerate(lats)]
    h = gb.Hydro.from_batch(lats)
    dt = h.compute_dt(torch.from_numpy(np.concatenate(states)).cuda()).cpu().numpy()
    for i, (l, U) in enumerate(zip(lats, states)):
        want = float(np.ravel(Oracle(l).compute_dt(U))[0])
        assert abs(dt[i] / want - 1.0) <= 4 * np.finfo(float).eps
