"""Error flags in mapped host memory and results written straight to the caller:
a bad bitstring in device memory is reported once and leaves the plan usable, a
ragged batch replayed from the graph equals its bitstrings in full batches, and
an output buffer that is not 16-byte aligned receives the same amplitudes.
Equalities are bitwise (the same kernels on the same inputs).
"""
import numpy as np
import pytest

from workloads import grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
def test_flags_ragged_and_alignment(prec):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    circ = grid_circuit(3, 4, 8, 1234)
    plan = T.Plan(T.Circuit(circ), batch_log2=3, n_candidates=4, seed=1)
    ctx = T.Context(0, prec)
    ctx.bind(plan)
    bits = random_bitstrings(12, 16, 3)
    full = ctx.amplitudes(plan, torch.from_numpy(bits).cuda())
    bad = torch.from_numpy(bits).cuda()
    bad[5, 7] = 2
    for _ in range(2):
        with pytest.raises(T.TnqError) as e:
            ctx.amplitudes(plan, bad)
        assert e.value.status == T.TNQ_ERR_INVALID_ARG
        assert torch.equal(ctx.amplitudes(plan, torch.from_numpy(bits).cuda()), full)
    for n in (1, 5, 11):
        assert torch.equal(ctx.amplitudes(plan, torch.from_numpy(bits[:n]).cuda()), full[:n])
        host = ctx.amplitudes(plan, bits[:n])
        assert np.array_equal(host, torch.view_as_complex(full).cpu().numpy()[:n])
    buf = torch.zeros(1 + 2 * 11, dtype=torch.float64, device="cuda")
    T.tnq_amplitudes(ctx.h, plan.h, torch.from_numpy(bits[:11]).cuda(), buf[1:])
    assert torch.equal(buf[1:].view(11, 2), full[:11])
