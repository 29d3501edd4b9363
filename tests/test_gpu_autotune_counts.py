"""The step counts autotuning returns cover every step that could run on the tensor
cores, in the modes that run small steps several to a launch (TF32x3) as in those
that do not (TF32): the same steps qualify in both.
"""
import pytest

from workloads import grid_circuit

pytestmark = pytest.mark.gpu


def test_counts_cover_the_same_steps():
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    plan = T.Plan(T.Circuit(grid_circuit(4, 4, 10, 7)), batch_log2=4, n_candidates=8, seed=1)
    total = {}
    for prec in ("tf32", "tf32x3"):
        ctx = T.Context(0, prec)
        ctx.bind(plan)
        total[prec] = sum(T.tnq_plan_autotune(ctx.h, plan.h, 1))
    assert total["tf32x3"] == total["tf32"] > 0
