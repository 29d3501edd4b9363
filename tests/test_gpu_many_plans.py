"""More bound plans than the process has mapped-memory slots for error flags
(4096): the later ones keep their flags in the workspace and behave alike.  The
plans share one workspace (same circuit, same plan, so the same constants).
Equalities are bitwise.
"""
import pytest

from workloads import grid_circuit, noisy_grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


def test_more_plans_than_flag_slots():
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    circ = T.Circuit(grid_circuit(2, 3, 4, 5))
    ctx = T.Context(0, "tf32x3")
    bits = torch.from_numpy(random_bitstrings(6, 6, 3)).cuda()
    bad = bits.clone()
    bad[4, 2] = 7
    plans = []
    ws = None
    for _ in range(4200):
        plan = T.Plan(circ, batch_log2=2, n_candidates=1, seed=1)
        nb = int(plan.info["workspace_bytes"])
        if ws is None:
            ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        T.tnq_plan_bind(ctx.h, plan.h, ws, nb)
        plans.append(plan)
    first, last = plans[0], plans[-1]
    want = ctx.amplitudes(first, bits)
    assert torch.equal(ctx.amplitudes(last, bits), want)
    for _ in range(2):
        with pytest.raises(T.TnqError) as e:
            ctx.amplitudes(last, bad)
        assert e.value.status == T.TNQ_ERR_INVALID_ARG
        assert torch.equal(ctx.amplitudes(last, bits), want)  # reported once, then usable
    T.tnq_plan_autotune(ctx.h, last.h, 1)
    ctx.amplitudes(last, bits)
    noisy = T.Plan(T.Circuit(noisy_grid_circuit(2, 2, 3, 1, 0.01, 0.01)), batch_log2=2, traj_log2=2, n_candidates=1)
    ctx.bind(noisy)
    with pytest.raises(T.TnqError) as e:
        T.tnq_noisy_probabilities(ctx.h, noisy.h, 8, 1, bad[:, :4].contiguous(), torch.zeros(6, device="cuda").double())
    assert e.value.status == T.TNQ_ERR_INVALID_ARG
