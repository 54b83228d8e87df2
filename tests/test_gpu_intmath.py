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
