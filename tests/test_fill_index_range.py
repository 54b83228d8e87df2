"""The guard fill's index arithmetic on blocks of very many planes, restated: the
launcher's rule for divisions by multiplication (gbh_aux.cu, launch_fill) leaves
only blocks whose padded index fits 32 bits to the kernel that forms it there;
the other kernel forms it in 64 bits, as blocks of more than 2^31 padded cells
(86 GB a state) need."""
import pytest


def launch(n, g, nz):
    """(multiplication allowed, padded cells) of a 3-D block of n x n x nz and g guards."""
    nxp = n + 2 * g
    ring = 2 * g * nxp + n * 2 * g
    cells = 2 * g * nxp * nxp + nz * ring
    return cells * nxp * nxp < 2 ** 32, (nz + 2 * g) * nxp * nxp


@pytest.mark.parametrize("n", [4, 8, 16])
def test_32_bit_indices_only_where_they_fit(n):
    for g in range(2, n + 1):
        lo, hi = 2, 2 ** 32
        while hi - lo > 1:                      # the largest nz that takes the multiplications
            mid = (lo + hi) // 2
            lo, hi = (mid, hi) if launch(n, g, mid)[0] else (lo, mid)
        fast, padded = launch(n, g, lo)
        assert fast and padded < 2 ** 31
        # quotients q / d of q < cells by multiply-high: exact for q d < 2^32, d <= the plane
        for d in (n + 2 * g, 2 * g, (n + 2 * g) ** 2, 2 * g * (n + 2 * g) + n * 2 * g):
            m = 2 ** 32 // d + 1
            top = 2 ** 32 // (n + 2 * g) ** 2
            for q in [0, 1, d - 1, d, top - 1, top // d * d - 1, top // d * d]:
                if 0 <= q <= top:
                    assert (q * m) >> 32 == q // d


def test_a_block_of_more_than_2_to_the_31_cells_takes_the_wide_index():
    nz = 2 ** 31 // 24 ** 2 + 1
    fast, padded = launch(16, 4, nz)
    assert not fast and padded > 2 ** 31
    k, j, i = nz + 7, 23, 23                    # the last padded cell
    assert (k * 24 + j) * 24 + i == padded - 1
    wrapped = ((k * 24 + j) * 24 + i + 2 ** 31) % 2 ** 32 - 2 ** 31
    assert wrapped < 0                          # what 32 bits would make of it
