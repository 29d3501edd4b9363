"""A pairwise contraction whose output shares memory with an operand (a gate
applied in place) gives what it gives into a buffer of its own: the one-launch,
long-K, gather, tall-skinny and general kernels, the output at the start of an
operand or inside it, in the order the kernels write and in others.  Every entry
against the FP64 oracle, at the bounds of each precision's kernels.
"""
import numpy as np
import pytest

from oracle import contraction
from test_gpu_batched import TOL, rel

pytestmark = pytest.mark.gpu

SHAPES = [  # (log2 M, N, K, H)
    (2, 5, 2, 2), (4, 5, 5, 0), (1, 6, 9, 0), (2, 10, 8, 0), (3, 8, 10, 1), (2, 2, 16, 0), (3, 16, 3, 0), (5, 12, 5, 0),
    (6, 6, 7, 0), (8, 8, 8, 0)]


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", ["scattered", "written"])
def test_output_overlaps_operand(prec, shape, order):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    m, n, k, h = shape
    rng = np.random.default_rng(sum(shape))
    ml, nl, kl, hl = (list(range(100 * i, 100 * i + d)) for i, d in enumerate(shape))
    al, bl = ([int(x) for x in rng.permutation(x)] for x in (ml + kl + hl, nl + kl + hl))
    ol = [x for x in bl if x in nl] + [x for x in al if x in ml] + [x for x in bl if x in hl]
    if order == "scattered":
        ol = [int(x) for x in rng.permutation(ol)]
    A, B = (((rng.standard_normal(2 ** len(x)) + 1j * rng.standard_normal(2 ** len(x))) / 2 ** (k / 4)).astype(
        np.complex64) for x in (al, bl))
    ref = contraction.contract_labeled(A, al, B, bl, ol)
    ctx = T.Context(0, prec)
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    # one buffer for both operands: A, then B; the output starts at B, inside B, or spans the two
    na, nB, no = A.size, B.size, ref.size
    starts = {na, na + nB // 2, max(0, na - no // 2)}
    for at in starts:
        buf = torch.zeros(max(na + nB, at + no), dtype=torch.complex64, device="cuda")
        buf[:na], buf[na:na + nB] = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
        C = buf[at:at + no]
        T.tnq_contract_pair(ctx.h, buf[:na], al, buf[na:na + nB], bl, C, ol, ws, nb)
        got = C.cpu().numpy()
        assert rel(got, ref) <= TOL[prec], (at, rel(got, ref))
