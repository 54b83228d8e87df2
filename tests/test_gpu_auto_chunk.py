"""The z-chunks a stage takes when the caller sets no decomposition: the state,
dt and floor counts are bit for bit those of whole blocks, from one block (one
plane per work item) to lattices that fill the chip, for every block width,
uneven nz, both stage counts, telescoping and two-level grids."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2401_03378_gb300 as gb
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return gb


def run(h, U0, steps=2):
    U = torch.from_numpy(U0.copy()).cuda()
    dt = h.compute_dt(U)
    hist = torch.zeros(steps * h.nproblems, dtype=torch.float64, device="cuda")
    h.floor_hits()
    h.advance(U, steps, dt, hist)
    return U, dt, hist, h.floor_hits()


def compare(make, U0):
    a, b = make(), make()
    b.set_decomposition(0, 1)
    ra, rb = run(a, U0), run(b, U0)
    assert all(torch.equal(x, y) for x, y in zip(ra[:3], rb[:3])) and ra[3] == rb[3]


@pytest.mark.parametrize("stages,telescoping", [(2, False), (3, False), (2, True), (3, True)])
@pytest.mark.parametrize("nb,n,nz", [((1, 1, 1), 16, 16), ((3, 2, 2), 16, 7), ((5, 5, 6), 16, 16), ((5, 3, 7), 8, 12),
                                     ((9, 8, 8), 8, 9), ((3, 3, 3), 4, 5)])
def test_uniform(gb, nb, n, nz, stages, telescoping):
    ng = 2 * stages if telescoping else 4
    if ng > min(n, nz):
        pytest.skip("more guard cells than cells")
    lat = wl.lattice_3d(*nb, n, n, nz, ng, bc=("periodic", "outflow", "periodic"))
    U0 = wl.random_state(lat, seed=17, rough=True)

    def make():
        h = gb.Hydro.from_lattice(lat)
        h.set_rk_stages(stages)
        h.set_telescoping(telescoping)
        return h
    compare(make, U0)


@pytest.mark.parametrize("telescoping", [False, True])
def test_two_level(gb, telescoping):
    tl = wl.two_level(wl.lattice_3d(4, 3, 4, 8, 8, 8, 4), (1, 1, 1), (3, 2, 3))
    U0 = wl.sedov_two_level(tl)[tl.gpu_blocks]

    def make():
        h = gb.Hydro.from_two_level(tl)
        h.set_telescoping(telescoping)
        return h
    compare(make, U0)


def test_batched(gb):
    lats = [wl.lattice_3d(2, 1, 3, 8, 8, 8, 4, bc="periodic"), wl.lattice_3d(1, 1, 1, 8, 8, 8, 4, bc="periodic")]
    U0 = np.concatenate([wl.random_state(l, seed=40 + i, rough=True) for i, l in enumerate(lats)])
    compare(lambda: gb.Hydro.from_batch(lats), U0)


@pytest.mark.parametrize("stages,telescoping", [(2, False), (3, True)])
@pytest.mark.parametrize("nb,n", [((1, 1), 16), ((9, 8), 16), ((3, 26), 16), ((1, 1), 8), ((13, 7), 8), ((24, 19), 8),
                                  ((24, 20), 8), ((1, 1), 4), ((40, 30), 4)])
def test_wide_ctas_2d(gb, nb, n, stages, telescoping):
    """A thread per face on small 2-D lattices, at both sides of the rule's lines."""
    ng = 2 * stages if telescoping else 4
    if ng > n:
        pytest.skip("more guard cells than cells")
    lat = wl.lattice_2d(*nb, n, n, ng, bc=("periodic", "outflow"))
    U0 = wl.random_state(lat, seed=23, rough=True)

    def make():
        h = gb.Hydro.from_lattice(lat)
        h.set_rk_stages(stages)
        h.set_telescoping(telescoping)
        return h
    compare(make, U0)


@pytest.mark.parametrize("nb,n,nz", [((2, 1, 2), 16, 16), ((1, 1, 1), 16, 4), ((2, 2, 2), 8, 8), ((3, 3, 2), 8, 7),
                                     ((4, 4, 4), 4, 4), ((5, 3, 5), 4, 6)])
def test_wide_ctas_3d(gb, nb, n, nz):
    lat = wl.lattice_3d(*nb, n, n, nz, 4, bc=("outflow", "periodic", "periodic"))
    compare(lambda: gb.Hydro.from_lattice(lat), wl.random_state(lat, seed=29, rough=True))


def test_wide_ctas_two_level(gb):
    tl = wl.two_level(wl.lattice_2d(5, 4, 8, 8, 4), (1, 1), (4, 3))
    U0 = wl.sedov_two_level(tl)[tl.gpu_blocks]
    compare(lambda: gb.Hydro.from_two_level(tl), U0)
