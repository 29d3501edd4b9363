"""Step programs (runs of small steps in one launch) give bitwise what the same
steps give one launch at a time: timed runs launch every step on its own.  Covers programs
of one CTA (outputs of at most 2^3), eight and sixteen (a step of 2^14 outputs),
more than 160 steps (the most a launch takes), sliced plans and noisy,
open-qubit, density-matrix and expectation plans, in FP32 and TF32x3, replayed
from a graph and not.
"""
import numpy as np
import pytest

from workloads import grid_circuit, noisy_grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


def both(T, ctx, call):
    """Equal results with programs and with a launch per step; launches saved."""
    out, n = [], []
    call()  # constant steps are contracted by the first call
    for timing in (False, True):
        T.tnq_ctx_set_timing(ctx.h, timing)
        before = T.tnq_ctx_launch_count(ctx.h)
        out.append(call())
        n.append(T.tnq_ctx_launch_count(ctx.h) - before)
    T.tnq_ctx_set_timing(ctx.h, False)
    assert n[0] < n[1]  # programs ran
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
    assert any(np.any(np.asarray(a) != 0) for a in out[0])
    return n[1] - n[0]


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("rows,cols,cycles,w,max_log2,widest,saved", [
    (2, 3, 4, 0, 28, 3, 1), (3, 4, 8, 6, 28, 12, 1), (3, 4, 8, 3, 8, 8, 1), (4, 5, 10, 2, 14, 13, 1),
    (6, 8, 8, 0, 26, 14, 1), (12, 12, 5, 0, 28, 12, 160)])
def test_amplitudes(prec, graphs, rows, cols, cycles, w, max_log2, widest, saved):
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    plan = T.Plan(T.Circuit(grid_circuit(rows, cols, cycles, 7)), batch_log2=w, n_candidates=4, seed=1,
                  max_intermediate_log2=max_log2)
    st = plan.steps()
    H, M, N, K = st[:, 3], st[:, 4], st[:, 5], st[:, 6]
    assert (H + M + N)[(H + M + N <= 14) & (K <= 10) & (H + M + N + K <= 15)].max() == widest
    ctx = T.Context(0, prec)
    ctx.bind(plan)
    T.tnq_ctx_set_graphs(ctx.h, graphs)
    bits = random_bitstrings(rows * cols, 2 ** w + 1, 3)
    assert both(T, ctx, lambda: [ctx.amplitudes(plan, bits)]) >= saved


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
def test_other_plans(prec):
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    ctx = T.Context(0, prec)
    noisy = T.Circuit(noisy_grid_circuit(3, 4, 6, 3, 0.02, 0.02))
    bits = random_bitstrings(12, 5, 3)
    plan = T.Plan(noisy, batch_log2=3, traj_log2=7, n_candidates=4, seed=1)
    ctx.bind(plan)
    both(T, ctx, lambda: list(ctx.noisy_probabilities(plan, bits, 200, 4)))
    dens = T.Plan(T.Circuit(noisy_grid_circuit(2, 3, 4, 3, 0.02, 0.02)), density=True, batch_log2=4, n_candidates=4)
    ctx.bind(dens)
    both(T, ctx, lambda: [ctx.density_probabilities(dens, random_bitstrings(6, 20, 3))])
    circ = T.Circuit(grid_circuit(3, 4, 8, 9))
    opened = T.Plan(circ, open_qubits=[0, 3, 4, 7, 11], batch_log2=3, n_candidates=4, seed=1)
    ctx.bind(opened)
    b = bits.copy()
    b[:, [0, 3, 4, 7, 11]] = -1
    both(T, ctx, lambda: [ctx.amplitudes(opened, b)])
    terms = ["Z" + "I" * 11, "IXIIYIIIZIII", "Z" * 12]
    expect = T.Plan(circ, paulis=terms, traj_log2=2, n_candidates=4, seed=1)
    ctx.bind(expect)
    both(T, ctx, lambda: [np.asarray(x) for x in ctx.expectation(expect, [1.0, 0.5, -2.0])])
