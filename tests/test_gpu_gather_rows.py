"""GPU parity of the gather kernel with two rows a thread (rows of one batch entry
of at least 2^9 and enough rows to fill the chip), at K = 1 to 32, in 256- and
128-thread CTAs, one row block a CTA and several.  The output is too large for a
full oracle: 64 sampled output columns (large-operand rows) are compared with
FP64 sums of the same inputs; FP32 sums of K <= 32 terms stay below 1e-5 in
relative L2, TF32 operand rounding below 5e-3.
"""
import numpy as np
import pytest

from oracle import contraction
from test_gpu_batched import TOL, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3"])
@pytest.mark.parametrize("m,n,k,h", [(1, 19, 0, 0), (3, 19, 1, 0), (2, 19, 2, 0), (5, 19, 3, 0), (3, 19, 4, 0),
                                     (3, 20, 5, 0), (2, 9, 4, 10), (1, 21, 3, 0)])
def test_two_rows_a_thread(prec, m, n, k, h):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    rng = np.random.default_rng(m + n + k + h)
    ml, nl, kl, hl = (list(range(100 * i, 100 * i + d)) for i, d in enumerate((m, n, k, h)))
    al, bl = ([int(x) for x in rng.permutation(x)] for x in (ml + kl + hl, nl + kl + hl))
    # the order the kernel writes: nothing is permuted afterwards
    ol = [x for x in bl if x in nl] + [x for x in al if x in ml] + [x for x in bl if x in hl]
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    A = torch.randn(2 ** len(al), dtype=torch.complex64, device="cuda", generator=g)
    B = torch.randn(2 ** len(bl), dtype=torch.complex64, device="cuda", generator=g)
    C = torch.full((2 ** len(ol),), float("nan"), dtype=torch.complex64, device="cuda")
    ctx = T.Context(0, prec)
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    T.tnq_contract_pair(ctx.h, A, al, B, bl, C, ol, ws, nb)
    assert bool(torch.isfinite(torch.view_as_real(C)).all())
    row_labels = ol[:n] + ol[n + m:]  # one large-operand row of one batch entry
    rows = rng.choice(2 ** (n + h), size=64, replace=False)
    rows[:2] = 0, 2 ** (n + h) - 1
    ref = contraction.sampled_rows(A.cpu().numpy(), al, B.cpu().numpy(), bl, ol, rows, row_labels)
    at = np.array([[(int(r) & (2 ** n - 1)) | j << n | (int(r) >> n) << (n + m) for j in range(2 ** m)] for r in rows])
    got = C[torch.from_numpy(at.reshape(-1)).cuda()].cpu().numpy().reshape(at.shape)
    assert rel(got, ref) <= TOL[prec], rel(got, ref)
