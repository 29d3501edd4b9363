"""GPU parity of the rows kernel (long-K steps with many rows): at the line from the
long-K kernel and on both sides of it, one row of the small side and 32, rows in
one batch entry and in many, half-filled tiles, K of one stage pair and more,
operands in the order it asks for and permuted.  64 sampled rows of the large
operand are compared with FP64 sums; FP32 sums of K <= 2^10 terms stay below 1e-5
in relative L2.

In plain TF32 and BF16x3 plans it takes steps whose sums keep a fixed order, as the
one-launch kernel does, a lane or a warp an output: the amplitudes of such a plan
stay within the modes' bounds (5e-3, and 5e-5 for a deep network) of the FP32 plan's.
"""
import numpy as np
import pytest

from oracle import contraction
from test_gpu_batched import TOL, rel
from workloads import grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["stored", "scattered"])
@pytest.mark.parametrize("m,n,k,h", [  # (log2 M, N, K, H)
    (3, 14, 6, 0), (3, 15, 6, 0), (2, 16, 6, 0), (0, 18, 6, 0), (1, 7, 6, 10), (4, 6, 6, 12), (5, 17, 6, 0), (3, 17, 7, 0),
    (5, 8, 7, 9), (5, 17, 8, 0), (2, 19, 8, 0)])
def test_rows(order, m, n, k, h):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    rng = np.random.default_rng(m + n + k + h)
    ml, nl, kl, hl = (list(range(100 * i, 100 * i + d)) for i, d in enumerate((m, n, k, h)))
    al, bl = kl + ml + hl, kl + nl + hl
    if order == "scattered":
        al, bl = ([int(v) for v in rng.permutation(x)] for x in (al, bl))
    ol = [x for x in bl if x in nl] + [x for x in al if x in ml] + [x for x in bl if x in hl]
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    A, B = (torch.randn(2 ** len(x), dtype=torch.complex64, device="cuda", generator=g) for x in (al, bl))
    C = torch.full((2 ** len(ol),), float("nan"), dtype=torch.complex64, device="cuda")
    ctx = T.Context(0, "fp32")
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS["fp32"], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    T.tnq_contract_pair(ctx.h, A, al, B, bl, C, ol, ws, nb)
    assert bool(torch.isfinite(torch.view_as_real(C)).all())
    row_labels = ol[:n] + ol[n + m:]  # one large-operand row of one batch entry
    rows = rng.choice(2 ** (n + h), size=64, replace=False)
    rows[:2] = 0, 2 ** (n + h) - 1
    ref = contraction.sampled_rows(A.cpu().numpy(), al, B.cpu().numpy(), bl, ol, rows, row_labels)
    at = np.array([[(int(r) & (2 ** n - 1)) | j << n | (int(r) >> n) << (n + m) for j in range(2 ** m)] for r in rows])
    got = C[torch.from_numpy(at.reshape(-1)).cuda()].cpu().numpy().reshape(at.shape)
    assert rel(got, ref) <= TOL["fp32"], rel(got, ref)


@pytest.mark.parametrize("rows,cols,cycles,w,max_log2,seed,shape", [
    (4, 6, 14, 4, 26, 1, lambda H, M, N, K: (M == 4) & (N >= 7) & (K >= 9) & (H + N + K >= 23)),  # rows kernel
    (4, 4, 12, 2, 18, 60, lambda H, M, N, K: (N <= 3) & (K >= 10) & (H + M + N + K <= 18)),       # a warp an output
    (4, 5, 9, 0, 19, 16, lambda H, M, N, K: (N <= 3) & (K >= 10) & (H + M + N + K <= 18))])
def test_ordered_sums(rows, cols, cycles, w, max_log2, seed, shape):
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    n = rows * cols
    plan = T.Plan(T.Circuit(grid_circuit(rows, cols, cycles, seed if seed > 1 else 8)), batch_log2=w, n_candidates=8,
                  seed=seed, max_intermediate_log2=max_log2)
    st = plan.steps()
    assert np.any(shape(st[:, 3], st[:, 4], st[:, 5], st[:, 6]))  # a step it is about
    bits = random_bitstrings(n, max(8, 2 ** w), 3)
    amp = {}
    for prec in ("fp32", "tf32", "bf16x3"):
        ctx = T.Context(0, prec)
        ctx.bind(plan)
        amp[prec] = ctx.amplitudes(plan, bits)
    assert rel(amp["tf32"], amp["fp32"]) <= 5e-3
    assert rel(amp["bf16x3"], amp["fp32"]) <= 5e-5
