"""Device tensors that start on an odd complex value (8-byte aligned, no more): the
operand permutes and the output permute that keep the lowest bit in place, and a
plain-TF32 operand handed to the general GEMM in its stored order, against the
FP64 oracle; device outputs of trajectory amplitudes and noisy probabilities at
an odd double, bitwise equal to aligned ones; 4-byte alignment is refused;
workspaces may start at any address.
"""
import numpy as np
import pytest

from oracle import contraction
from test_gpu_batched import TOL, rel
from workloads import noisy_grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


def odd(x, dtype):
    import torch
    t = torch.zeros(x.size + 1, dtype=dtype, device="cuda")
    t[1:] = torch.from_numpy(x).cuda()
    return t[1:]


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("m,n,k,h", [(8, 8, 8, 0), (7, 8, 7, 1), (3, 16, 3, 0), (6, 12, 5, 0)])
@pytest.mark.parametrize("moved", ["nothing", "operands", "output", "all"])
def test_pair_operands_and_output(prec, m, n, k, h, moved):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    rng = np.random.default_rng(m + n + k + h)
    ml, nl, kl, hl = (list(range(100 * i, 100 * i + d)) for i, d in enumerate((m, n, k, h)))
    al, bl, ol = kl + ml + hl, kl + nl + hl, nl + ml + hl  # the order the kernels ask for

    def keep_bit0(x):
        return [x[0]] + [int(v) for v in rng.permutation(x[1:])]

    if moved in ("operands", "all"):
        al, bl = keep_bit0(al), keep_bit0(bl)
    if moved in ("output", "all"):
        ol = keep_bit0(ol)
    A, B = (((rng.standard_normal(2 ** len(x)) + 1j * rng.standard_normal(2 ** len(x))) / 2 ** (k / 4)).astype(
        np.complex64) for x in (al, bl))
    C = odd(np.zeros(2 ** len(ol), np.complex64), torch.complex64)
    ctx = T.Context(0, prec)
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    T.tnq_contract_pair(ctx.h, odd(A, torch.complex64), al, odd(B, torch.complex64), bl, C, ol, ws, nb)
    got, ref = C.cpu().numpy(), contraction.contract_labeled(A, al, B, bl, ol)
    assert rel(got, ref) <= TOL[prec], rel(got, ref)


def test_noisy_device_outputs():
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    plan = T.Plan(T.Circuit(noisy_grid_circuit(2, 3, 4, 1, 0.05, 0.05)), batch_log2=2, traj_log2=3, n_candidates=2)
    ctx = T.Context(0, "fp32")
    ctx.bind(plan)
    bits = torch.from_numpy(random_bitstrings(6, 7, 3)).cuda()

    def buf(n, at):
        return torch.zeros(n + at, dtype=torch.float64, device="cuda")[at:]

    out, amp = [], []
    for at in (0, 1):
        p, se, a = buf(7, at), buf(7, at), buf(2 * 7 * 11, at)
        T.tnq_noisy_probabilities(ctx.h, plan.h, 11, 5, bits, p, se)
        T.tnq_trajectory_amplitudes(ctx.h, plan.h, 5, 0, 11, bits, a)
        out.append(torch.cat([p, se]))
        amp.append(a.clone())
    assert torch.equal(out[0], out[1]) and torch.equal(amp[0], amp[1])
    assert bool((amp[0] != 0).any())


def test_four_byte_alignment_is_refused():
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    ctx = T.Context(0, "fp32")
    x = torch.zeros(64, dtype=torch.float32, device="cuda")
    nb = T.tnq_contract_workspace_bytes(T.PRECISIONS["fp32"], 2, 2, 2)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    for at in range(3):
        s = [16 * i + (1 if i == at else 0) for i in range(3)]
        with pytest.raises(T.TnqError) as e:
            T.tnq_contract_pair(ctx.h, x[s[0]:], [0, 1], x[s[1]:], [1, 2], x[s[2]:], [0, 2], ws, nb)
        assert e.value.status == T.TNQ_ERR_INVALID_ARG


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
@pytest.mark.parametrize("at", [1, 8, 255])
def test_workspace_at_any_address(prec, at):
    """Bitwise what an aligned workspace gives, and nothing written outside it."""
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    from workloads import grid_circuit
    build.build()
    ctx = T.Context(0, prec)
    guard = 512

    def workspace(nb, shift):
        w = torch.full((nb + shift + guard,), 0xa5, dtype=torch.uint8, device="cuda")
        return w, w[shift:shift + nb]

    def untouched(w, nb, shift):
        return bool((w[:shift] == 0xa5).all()) and bool((w[shift + nb:] == 0xa5).all())

    bits = random_bitstrings(12, 9, 3)
    plan = T.Plan(T.Circuit(grid_circuit(3, 4, 8, 1234)), batch_log2=2, n_candidates=4, seed=1)
    nb = int(plan.info["workspace_bytes"])
    got = []
    for shift in (0, at):
        w, ws = workspace(nb, shift)
        T.tnq_plan_bind(ctx.h, plan.h, ws, nb)
        got.append(ctx.amplitudes(plan, bits))
        assert untouched(w, nb, shift)
    assert np.array_equal(got[0], got[1])
    rng = np.random.default_rng(7)
    for m, n, k in ((8, 8, 8), (6, 14, 6), (5, 9, 8)):
        al, bl = ([int(v) for v in rng.permutation(x)] for x in (
            list(range(m)) + list(range(200, 200 + k)), list(range(100, 100 + n)) + list(range(200, 200 + k))))
        ol = [int(v) for v in rng.permutation(list(range(m)) + list(range(100, 100 + n)))]
        A, B = (torch.randn(2 ** len(x), dtype=torch.complex64, device="cuda") for x in (al, bl))
        nb = T.tnq_contract_workspace_bytes(T.PRECISIONS[prec], len(al), len(bl), len(ol))
        out = []
        for shift in (0, at):
            w, ws = workspace(nb, shift)
            C = torch.full((2 ** len(ol),), float("nan"), dtype=torch.complex64, device="cuda")
            T.tnq_contract_pair(ctx.h, A, al, B, bl, C, ol, ws, nb)
            assert untouched(w, nb, shift)
            out.append(C)
        assert torch.equal(out[0], out[1])
    grads = []
    X, t = rng.uniform(size=(40, 16)).astype(np.float32), rng.standard_normal(40).astype(np.float32)
    for shift in (0, at):
        m = T.CostModel(ctx, hidden=64, max_batch=64, seed=3)
        nb = m.ws.numel()
        w, ws = workspace(nb, shift)
        T.check(T.load().tnq_cost_model_bind(ctx.h, m.h, T.C.c_void_p(ws.data_ptr()), nb))
        grads.append(m.gradients(X, t)[0])
        assert untouched(w, nb, shift)
    assert np.array_equal(grads[0], grads[1])
