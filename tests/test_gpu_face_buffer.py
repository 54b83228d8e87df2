"""The face pre-pass is on, and its buffer held, where a stage can take it."""
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


@pytest.mark.parametrize("lat,default", [(wl.lattice_3d(4, 4, 4, 16, 16, 16, 4), False),
                                         (wl.lattice_3d(12, 12, 12, 8, 8, 8, 4), True),
                                         (wl.lattice_2d(9, 9, 8, 8, 4), False)])
def test_getter_and_plan(gb, lat, default):
    h = gb.Hydro.from_lattice(lat)
    assert h.face_prepass() == default and h.stage_plan()["face_prepass"] == default
    h.set_face_prepass(True)
    assert h.face_prepass() and h.stage_plan()["face_prepass"]
    h.set_tile_split(0, 2)
    assert h.face_prepass() and not h.stage_plan()["face_prepass"]
    h.set_tile_split(0, 1)
    h.set_face_prepass(False)
    assert not h.face_prepass() and not h.stage_plan()["face_prepass"]


def test_no_buffer_that_no_stage_reads(gb):
    """A context of 16^3 blocks holds three states of device memory (the intermediate
    stage and the two primitive arrays) and its tables; the buffer is 126 MB here."""
    lat = wl.lattice_3d(16, 16, 8, 16, 16, 16, 2)
    torch.cuda.synchronize()
    gb.Hydro.from_lattice(wl.lattice_3d(1, 1, 1, 16, 16, 16, 2)).close()   # kernels loaded
    free0, _ = torch.cuda.mem_get_info()
    h = gb.Hydro.from_lattice(lat)
    free1, _ = torch.cuda.mem_get_info()
    state = lat.nblocks * 5 * 20 ** 3 * 8
    assert free0 - free1 <= 3 * state + (32 << 20)
    h.set_face_prepass(True)
    free2, _ = torch.cuda.mem_get_info()
    assert free1 - free2 >= lat.nblocks * 6 * 5 * 256 * 8
