"""GPU parity of the one-launch kernel for small contractions (at most 2^18
complex multiply-adds, K <= 2^10): operands read and output written through bit
deposits in any order, up to 32 lanes per output element.  Edges: a scalar, no
contracted index, no free index, the longest K, the largest size and the first
one beyond it, every kind of output order.  Every entry against the FP64 oracle;
FP32 sums of K <= 2^10 terms stay below 1e-5 in relative L2 (K random-sign
roundings of 2^-24), TF32 operand rounding below 5e-3.
"""
import numpy as np
import pytest

from test_gpu_batched import TOL, contract, rel

pytestmark = pytest.mark.gpu

SHAPES = [(0, 0, 0, 0), (0, 0, 1, 0), (0, 0, 10, 0), (1, 0, 4, 0), (0, 3, 0, 2), (3, 3, 0, 0), (2, 5, 3, 4),
          (6, 6, 6, 0), (6, 6, 7, 0), (1, 1, 10, 6), (2, 2, 11, 3), (0, 1, 0, 17), (3, 12, 3, 0), (5, 7, 2, 4)]


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", ["scattered", "stored"])
def test_small_contraction(prec, shape, order):
    got, ref = contract(prec, *shape, seed=sum(shape) + 3, order=order)
    assert np.all(np.isfinite(got))
    assert rel(got, ref) <= TOL[prec], rel(got, ref)
