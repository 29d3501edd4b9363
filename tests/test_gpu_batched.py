"""GPU parity of short-K contractions with many batch entries and short rows.

The gather kernel serves several batch entries per CTA when the rows of one are
few, and its small operand may have up to 128 rows; the tall-skinny tensor-core
kernel gives each CTA one batch entry when the expanded small operands of all
entries do not fit in shared memory.  Operand and output indices are scattered,
every output entry is compared with the FP64 oracle.  Bounds on the relative L2
error: FP32 arithmetic (also used for short rows in the split modes) at most
K * 2^-24 * sqrt(2) < 1e-5 at K <= 64; TF32 operand rounding 2^-11 per factor,
below 5e-3 in every norm here.
"""
import numpy as np
import pytest

from oracle import contraction

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "tf32x3": 1e-5, "bf16x3": 2e-5, "tf32": 5e-3}


def contract(prec, m, n, k, h, seed, order="scattered", policy=None):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    rng = np.random.default_rng(seed)
    ml, nl, kl, hl = (list(range(100 * i, 100 * i + d)) for i, d in enumerate((m, n, k, h)))
    al, bl, ol = ml + kl + hl, nl + kl + hl, nl + ml + hl
    if order == "scattered":
        al, bl, ol = (list(rng.permutation(x)) for x in (al, bl, ol))
    elif order == "stored":  # the order the kernels ask for: nothing is permuted
        al, bl = kl + ml + hl, kl + nl + hl

    def draw(r):
        return ((rng.standard_normal(2 ** r) + 1j * rng.standard_normal(2 ** r)) / 2 ** (k / 4)).astype(np.complex64)

    A, B = draw(len(al)), draw(len(bl))
    ctx = T.Context(0, prec)
    if policy is not None:
        T.tnq_ctx_set_kernel_policy(ctx.h, policy)
    At, Bt = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((2 ** len(ol),), float("nan"), dtype=torch.complex64, device="cuda")
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    T.tnq_contract_pair(ctx.h, At, al, Bt, bl, C, ol, ws, nb)
    return C.cpu().numpy(), contraction.contract_labeled(A, al, B, bl, ol)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("shape", [  # (log2 M, N, K, H)
    (0, 0, 1, 9), (1, 2, 0, 8), (2, 3, 5, 6), (0, 8, 0, 0), (1, 9, 3, 3), (3, 7, 2, 10), (5, 7, 3, 8), (5, 5, 5, 7),
    (6, 7, 3, 6), (7, 8, 0, 5), (7, 7, 3, 5), (6, 10, 4, 2), (4, 7, 4, 9), (5, 8, 5, 6), (6, 8, 6, 5), (2, 11, 1, 4)])
def test_batched_short_k(prec, shape):
    got, ref = contract(prec, *shape, seed=sum(shape) + 31)
    assert np.all(np.isfinite(got))
    assert rel(got, ref) <= TOL[prec], rel(got, ref)


@pytest.mark.parametrize("prec", ["fp32", "tf32"])
@pytest.mark.parametrize("shape", [(2, 4, 3, 5), (5, 7, 3, 8), (1, 9, 5, 2)])
def test_batched_stored_order(prec, shape):
    got, ref = contract(prec, *shape, seed=5, order="stored")
    assert rel(got, ref) <= TOL[prec], rel(got, ref)


def test_large_small_operand_is_permuted():
    """A small operand beyond 2^22 elements leaves the in-place read."""
    got, ref = contract("fp32", 1, 2, 2, 20, seed=3)
    assert rel(got, ref) <= TOL["fp32"], rel(got, ref)


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
@pytest.mark.parametrize("m,n,k", [(6, 14, 3), (3, 16, 3), (2, 3, 14), (4, 5, 4)])
def test_operands_eight_byte_aligned(prec, m, n, k):
    """Operands and output that start on an odd complex value: the kernels that
    read them in place fall back to 8-byte accesses."""
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    rng = np.random.default_rng(m + n + k)
    al, bl = list(range(k)) + list(range(100, 100 + m)), list(range(k)) + list(range(200, 200 + n))
    ol = list(range(200, 200 + n)) + list(range(100, 100 + m))
    A, B = ((rng.standard_normal(2 ** len(x)) + 1j * rng.standard_normal(2 ** len(x))).astype(np.complex64)
            for x in (al, bl))

    def odd(x):
        t = torch.zeros(x.size + 1, dtype=torch.complex64, device="cuda")
        t[1:] = torch.from_numpy(x).cuda()
        return t[1:]

    C = odd(np.zeros(2 ** len(ol), np.complex64))
    ctx = T.Context(0, prec)
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    T.tnq_contract_pair(ctx.h, odd(A), al, odd(B), bl, C, ol, ws, nb)
    got, ref = C.cpu().numpy(), contraction.contract_labeled(A, al, B, bl, ol)
    assert rel(got, ref) <= TOL[prec], rel(got, ref)
