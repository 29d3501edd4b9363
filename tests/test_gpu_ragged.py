"""Ragged batches and the captured graph.  A single ragged request launches its
kernels directly: it makes as many launches as with graphs off, where a replay
counts the graph's nodes (one more: the clearing of the accumulator).  The second
one captures, later ones replay, and all give the same bits, also after a change
of precision and beside full batches.
"""
import pytest

from workloads import grid_circuit, random_bitstrings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
def test_single_ragged_batch_is_not_captured(prec):
    import torch
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    circ = T.Circuit(grid_circuit(3, 4, 8, 1234))
    bits = torch.from_numpy(random_bitstrings(12, 8, 3)).cuda()

    def fresh(graphs):
        plan = T.Plan(circ, batch_log2=3, n_candidates=4, seed=1, max_intermediate_log2=9)
        ctx = T.Context(0, prec)
        T.tnq_ctx_set_graphs(ctx.h, graphs)
        ctx.bind(plan)
        return plan, ctx

    def call(plan, ctx, n):
        before = T.tnq_ctx_launch_count(ctx.h)
        out = ctx.amplitudes(plan, bits[:n])
        return out, T.tnq_ctx_launch_count(ctx.h) - before

    off = fresh(False)
    want, direct = call(*off, 5)
    _, again = call(*off, 5)  # constant steps are contracted by the first call
    on = fresh(True)
    got, n0 = call(*on, 5)
    assert n0 == direct
    assert torch.equal(got, want)
    counts = []
    for _ in range(3):
        got, n = call(*on, 5)
        assert torch.equal(got, want)
        counts.append(n)
    assert len(set(counts)) == 1 and counts[0] == again + 1  # captured, then replayed
    full, _ = call(*on, 8)
    assert torch.equal(full[:5], want)
    on[1].set_precision("bf16x3")
    a, _ = call(*on, 5)
    b, _ = call(*on, 5)
    assert torch.equal(a, b)
    on[1].set_precision(prec)
    assert torch.equal(call(*on, 5)[0], want)
    assert torch.equal(call(*on, 8)[0], full)
