"""The chunks the pipelined host step forms by default (gbh_abi.cu, pipe_setup),
restated: a power of two by the square root of the copies' time, of equal
numbers of blocks; and the schedule check of test_host_pipeline_schedule.py on
them, for lattices of every chunk count it comes to."""
import pytest

from tests.test_host_pipeline_schedule import check_schedule, face_table


def default_chunks(cells, nblocks):
    """Chunks of nblocks blocks of `cells` cells: the largest power of two K with
    4 (K/2)^2 13 us <= the time of both copies at 200 GB/s, at most 64."""
    copies = 2.0 * 8.0 * 5.0 * cells * nblocks / 200e9
    K = 1
    while K < 64 and 4.0 * K * K * 13e-6 <= copies:
        K *= 2
    return min(K, nblocks)


@pytest.mark.parametrize("cells,nblocks,chunks", [(16 ** 3, 64, 2), (16 ** 3, 216, 4), (16 ** 3, 512, 8),
                                                  (16 ** 3, 990, 8), (16 ** 3, 4096, 16), (8 ** 3, 1728, 4),
                                                  (16 ** 2, 64, 1), (16 ** 3, 1, 1), (256 ** 3, 1, 1),
                                                  (256 ** 3, 100, 64)])
def test_number_of_chunks(cells, nblocks, chunks):
    assert default_chunks(cells, nblocks) == chunks


@pytest.mark.parametrize("nb,periodic", [((4, 4, 4), (True, True, True)), ((6, 6, 6), (False, True, False)),
                                         ((8, 8, 8), (False, False, True)), ((9, 10, 11), (True, True, True)),
                                         ((16, 16, 16), (False, False, False))])
def test_default_chunks_schedule(nb, periodic):
    face = face_table(3, nb, periodic)
    check_schedule(face, 3, default_chunks(16 ** 3, face.shape[0]))
