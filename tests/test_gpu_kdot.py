"""GPU parity of the long-K kernel (small side of at most 32 rows, K >= 2^6)
beyond the one-launch kernel's sizes: one K tile and many, one split and many,
single rows, the largest tile, batch entries, every block shape, operands
scattered or in the order the kernels ask for.  Every entry against the FP64
oracle; FP32 sums below 1e-5 in relative L2.  The tensor-core modes keep the
bounds of their own kernels (some of these shapes run there).
"""
import pytest

from test_gpu_batched import TOL, contract, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
@pytest.mark.parametrize("order", ["scattered", "stored"])
@pytest.mark.parametrize("shape", [(0, 0, 20, 0), (0, 2, 18, 0), (2, 3, 15, 0), (3, 3, 14, 2), (1, 1, 12, 7),
                                   (5, 5, 10, 0), (4, 6, 9, 2), (2, 7, 10, 4), (5, 10, 6, 0), (0, 13, 7, 0),
                                   (3, 5, 11, 0), (1, 4, 16, 0), (4, 4, 13, 0)])
def test_long_k(prec, order, shape):
    got, ref = contract(prec, *shape, seed=sum(shape), order=order)
    assert rel(got, ref) <= TOL[prec], rel(got, ref)
