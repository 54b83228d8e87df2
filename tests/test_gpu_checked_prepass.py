"""The bounds-checked build with the face pre-pass asked for: the stage of 16-wide
blocks that reads its boundary fluxes from the pre-pass and lays the plane's
fluxes over its primitives, z-chunks and whole blocks, two and three stages."""
import pytest
import torch

import workloads as wl
from tests.test_gpu_checked import both, dev, gb  # noqa: F401

pytestmark = pytest.mark.gpu

LATS = {"16": wl.lattice_3d(3, 2, 2, 16, 16, 16, 4, bc=("periodic", "outflow", "periodic")),
        "16-nz5": wl.lattice_3d(2, 3, 2, 16, 16, 5, 4, bc="outflow"),
        "8": wl.lattice_3d(2, 2, 3, 8, 8, 8, 4, bc="periodic"),
        "2d-16": wl.lattice_2d(3, 3, 16, 16, 4, bc=("periodic", "outflow"))}


@pytest.mark.parametrize("stages", [2, 3])
@pytest.mark.parametrize("name", list(LATS))
def test_asked_prepass(gb, name, stages):  # noqa: F811
    lat = LATS[name]
    U0 = wl.random_state(lat, seed=71, rough=True)

    def make(checked):
        h = gb.Hydro.from_lattice(lat, checked=checked)
        h.set_rk_stages(stages)
        h.set_face_prepass(True)
        return h

    def run(h):
        U = dev(U0)
        dt = h.compute_dt(U)
        h.advance(U, 2, dt)
        h.set_decomposition(0, 3)
        h.advance(U, 1, dt)
        out = torch.zeros_like(U)
        h.stage(U, U, out, 1e-3, 0.5, 0.5)
        return [U, dt, out]
    both(gb, make, run)


def test_asked_prepass_two_level(gb):  # noqa: F811
    tl = wl.two_level(wl.lattice_3d(3, 4, 3, 16, 16, 16, 4), (1, 1, 1), (2, 3, 2))
    U0 = wl.sedov_two_level(tl)[tl.gpu_blocks]

    def make(checked):
        h = gb.Hydro.from_two_level(tl, checked=checked)
        h.set_face_prepass(True)
        return h

    def run(h):
        U = dev(U0)
        h.fill_guardcells(U)
        dt = h.compute_dt(U)
        h.advance(U, 2, dt)
        return [U, dt]
    both(gb, make, run)
