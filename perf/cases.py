"""Performance cases: the work a program gives this library through its public calls.

Four kinds of calls:

* ``pair``: one pairwise contraction of complex64 tensors whose indices all have
  dimension 2 (``tnq_contract_pair``), the unit step of every contraction;
* ``amplitudes``: bitstring amplitudes of a grid random circuit through a plan
  made and bound beforehand (``Context.amplitudes``);
* ``noisy``: bitstring probabilities of a noisy grid circuit averaged over Kraus
  trajectories (``tnq_noisy_probabilities``);
* ``cost_gradients``: one forward and backward pass of the path cost model on a
  minibatch of step features (``CostModel.gradients``).

The library contracts in complex64 and FP32 (only sums over slices and
trajectories are FP64) but hands amplitudes and probabilities over as doubles;
the programs here keep them in single precision, which is what they carry.
"""
import math

import numpy as np
import torch

from paper_2104_10523_gb300 import tnq

DEVICE = "cuda:0"
PRECISIONS = ("fp32", "tf32", "tf32x3", "bf16x3")


# ------------------------------------------------------------------ the cases
def _pair(m, n, k, precision, layout, h=0, layout_seed=1):
    """Output 2^m x 2^n per batch entry, 2^k contracted, 2^h batch entries.  layout:
    "scattered" permutes every tensor's indices at random (unrelated producers
    and consumers), "chain" scatters the operands but takes the output in the
    order the contraction writes it (a program that chains contractions)."""
    return {"kind": "pair", "m": m, "n": n, "k": k, "h": h, "precision": precision, "layout": layout,
            "layout_seed": layout_seed}


def _amplitudes(rows, cols, cycles, n_bs, batch_log2, precision, circuit_seed, candidates=16, autotune=False):
    return {"kind": "amplitudes", "rows": rows, "cols": cols, "cycles": cycles, "n_bs": n_bs,
            "batch_log2": batch_log2, "precision": precision, "circuit_seed": circuit_seed,
            "candidates": candidates, "autotune": autotune}


def _noisy(rows, cols, cycles, p, n_traj, n_bs, batch_log2, traj_log2, precision, circuit_seed):
    return {"kind": "noisy", "rows": rows, "cols": cols, "cycles": cycles, "p": p, "n_traj": n_traj, "n_bs": n_bs,
            "batch_log2": batch_log2, "traj_log2": traj_log2, "precision": precision, "circuit_seed": circuit_seed}


def listed():
    return [
        # the smallest contraction of the microbenchmark: one call's latency
        dict(_pair(6, 6, 6, "fp32", "scattered"), name="pair small fp32"),
        # a square contraction, bound by the tensor cores
        dict(_pair(12, 12, 12, "bf16x3", "scattered"), name="pair cube bf16x3"),
        # a gate-sized operand of 16 rows meeting a large tensor: the heaviest step of the amplitude benchmark
        dict(_pair(4, 23, 4, "tf32x3", "chain"), name="pair 16 rows tf32x3"),
        # a merged operand of 64 rows meeting a large tensor, as in the same benchmark
        dict(_pair(6, 20, 6, "tf32x3", "chain"), name="pair 64 rows tf32x3"),
        # plain FP32 with a small operand of 8 rows: bound by memory
        dict(_pair(3, 23, 3, "fp32", "chain"), name="pair 8 rows fp32"),
        # an inner product closing a network: tiny output, long contracted extent, uneven sides
        dict(_pair(2, 3, 20, "fp32", "scattered"), name="pair dot fp32"),
        # many small contractions as one batch (bitstrings and trajectories are batch indices), odd sizes
        dict(_pair(5, 7, 3, "tf32", "scattered", h=11), name="pair batched tf32"),
        # the smallest circuit of the parity suite: every step is tiny
        dict(_amplitudes(3, 4, 8, 64, 6, "fp32", 1234), name="amplitudes 3x4"),
        # a middle-sized circuit, a bitstring count that leaves a ragged last batch
        dict(_amplitudes(5, 5, 14, 100, 6, "tf32x3", 55), name="amplitudes 5x5"),
        # the benchmark circuit, sliced, autotuned as the benchmark does
        dict(_amplitudes(6, 6, 14, 4, 2, "tf32x3", 2104, candidates=32, autotune=True), name="amplitudes 6x6"),
        # the noisy benchmark circuit: trajectories and bitstrings contracted as batch indices
        dict(_noisy(4, 5, 10, 1e-3, 1024, 64, 4, 8, "tf32x3", 2021), name="noisy 4x5"),
        # training the path cost model: gradients of one minibatch
        {"kind": "cost_gradients", "rows": 1024, "name": "cost model gradients"},
    ]


def draw(rng):
    kind = rng.choice(["square", "skinny", "skinny", "dot", "batched", "amplitudes", "amplitudes", "noisy",
                       "cost_gradients"])
    precision = rng.choice(PRECISIONS)
    layout = rng.choice(["scattered", "chain"])
    ls = rng.randrange(1000)
    if kind == "square":
        return _pair(rng.randint(6, 12), rng.randint(6, 12), rng.randint(6, 12), precision, layout, layout_seed=ls)
    if kind == "skinny":
        return _pair(rng.randint(1, 7), rng.randint(12, 20), rng.randint(1, 7), precision, layout, layout_seed=ls)
    if kind == "dot":
        return _pair(rng.randint(0, 3), rng.randint(0, 3), rng.randint(10, 20), precision, layout, layout_seed=ls)
    if kind == "batched":
        return _pair(rng.randint(1, 6), rng.randint(1, 7), rng.randint(1, 6), precision, layout, h=rng.randint(2, 10),
                     layout_seed=ls)
    if kind == "amplitudes":
        return _amplitudes(rng.randint(2, 5), rng.randint(3, 5), rng.randint(6, 14), int(2 ** rng.uniform(0, 7)),
                           rng.randint(0, 6), precision, rng.randrange(10 ** 6))
    if kind == "noisy":
        return _noisy(rng.randint(2, 4), rng.randint(3, 5), rng.randint(6, 10), rng.choice([2e-3, 1e-2]),
                      int(2 ** rng.uniform(6, 9.5)), int(2 ** rng.uniform(3, 7)), rng.randint(2, 5),
                      rng.randint(4, 8), precision, rng.randrange(10 ** 6))
    return {"kind": "cost_gradients", "rows": int(2 ** rng.uniform(5, 12))}


# ------------------------------------------------------------------ circuits
class _Op:
    def __init__(self, kind, qubits, mats):
        self.kind, self.qubits, self.mats = kind, qubits, mats


class _Circuit:
    def __init__(self, n):
        self.n, self.ops = n, []


def _circuit(case):
    """Grid random circuit: per cycle a random gate of {sqrt-X, sqrt-Y, sqrt-W} on
    every qubit, then fSim(pi/2, pi/6) on the couplers of pattern ABCDCDAB; with
    noise, depolarizing(p) on every qubit a gate acted on and amplitude damping
    of the same strength on every qubit at the end of a cycle."""
    s = 1 / math.sqrt(2)
    singles = [s * np.array([[1, -1j], [-1j, 1]]), s * np.array([[1, -1], [1, 1]], complex),
               s * np.array([[1, np.exp(-0.75j * np.pi)], [np.exp(-0.25j * np.pi), 1]])]
    c, z, ph = math.cos(math.pi / 2), -1j * math.sin(math.pi / 2), np.exp(-1j * math.pi / 6)
    fsim = np.array([[1, 0, 0, 0], [0, c, z, 0], [0, z, c, 0], [0, 0, 0, ph]])
    p = case.get("p", 0.0)
    depol = [math.sqrt(1 - p) * np.eye(2), math.sqrt(p / 3) * np.array([[0, 1], [1, 0]]),
             math.sqrt(p / 3) * np.array([[0, -1j], [1j, 0]]), math.sqrt(p / 3) * np.diag([1.0, -1.0])]
    damp = [np.diag([1.0, math.sqrt(1 - p)]), np.array([[0, math.sqrt(p)], [0, 0]])]
    rows, cols = case["rows"], case["cols"]
    rng = np.random.default_rng(case["circuit_seed"])
    circ = _Circuit(rows * cols)

    def gate(u, *q):
        circ.ops.append(_Op("gate", q, [np.asarray(u, np.complex128)]))
        if p > 0:
            for x in q:
                circ.ops.append(_Op("channel", (x,), [np.asarray(a, np.complex128) for a in depol]))

    for cycle in range(case["cycles"]):
        for q in range(circ.n):
            gate(singles[int(rng.integers(0, 3))], q)
        letter = "ABCDCDAB"[cycle % 8]
        for r in range(rows):
            for col in range(cols):
                q = r * cols + col
                if letter in "AB" and col + 1 < cols and col % 2 == "AB".index(letter):
                    gate(fsim, q, q + 1)
                if letter in "CD" and r + 1 < rows and r % 2 == "CD".index(letter):
                    gate(fsim, q, q + cols)
        if p > 0:
            for q in range(circ.n):
                circ.ops.append(_Op("channel", (q,), [np.asarray(a, np.complex128) for a in damp]))
    return circ


def _bits(case, seed):
    return np.random.default_rng(seed).integers(0, 2, size=(case["n_bs"], case["rows"] * case["cols"]), dtype=np.int8)


def _plan(case):
    if case["kind"] == "noisy":
        return tnq.Plan(tnq.Circuit(_circuit(case)), batch_log2=case["batch_log2"], traj_log2=case["traj_log2"],
                        n_candidates=16, seed=1)
    return tnq.Plan(tnq.Circuit(_circuit(case)), batch_log2=case["batch_log2"], n_candidates=case["candidates"],
                    seed=7)


# ------------------------------------------------------------------ pairs
def _labels(case):
    """Index lists of A, B and C (entry p names bit p of the flat index)."""
    m, n, k, h = case["m"], case["n"], case["k"], case["h"]
    rng = np.random.default_rng(case["layout_seed"])
    a_free, b_free = list(range(m)), list(range(100, 100 + n))
    shared, batch = list(range(200, 200 + k)), list(range(300, 300 + h))
    a = [int(x) for x in rng.permutation(a_free + shared + batch)]
    b = [int(x) for x in rng.permutation(b_free + shared + batch)]
    if case["layout"] == "scattered":
        return a, b, [int(x) for x in rng.permutation(a_free + b_free + batch)]
    # free indices of the larger operand, then of the smaller, then the batch, each as stored
    small, big = (b, a) if len(a) > len(b) else (a, b)
    return a, b, [x for x in big if x not in small] + [x for x in small if x not in big] + [x for x in big if x >= 300]


def _operands(case, seed):
    """Complex normal entries scaled so that output entries have unit variance."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    a, b, _ = _labels(case)
    scale = 2.0 ** (-0.5 * case["k"])
    A = torch.randn(2 ** len(a), dtype=torch.complex64, device=DEVICE, generator=g).mul_(math.sqrt(scale))
    B = torch.randn(2 ** len(b), dtype=torch.complex64, device=DEVICE, generator=g).mul_(math.sqrt(scale))
    return A, B


def _reorder(x, have, want):
    """The flat tensor x with index order `have`, rewritten in the order `want`."""
    i = torch.arange(x.numel(), device=x.device)
    at = torch.zeros_like(i)
    for p, label in enumerate(want):
        at |= ((i >> p) & 1) << have.index(label)
    return x[at]


# ------------------------------------------------------------------ the cost model
def _rows(case, seed):
    """Step features (sizes over 32, 0/1 kernel flags), log times and parameters."""
    rng = np.random.default_rng(seed)
    d = 16
    X = rng.uniform(0, 1, size=(case["rows"], d)).astype(np.float32)
    X[:, 8:14] = X[:, 8:14] > 0.5
    t = rng.normal(3.0, 2.0, size=case["rows"]).astype(np.float32)
    hid = 256

    def u(fan, count):
        return rng.uniform(-1, 1, count) * math.sqrt(6.0 / fan)

    params = np.concatenate([u(d, d * hid), 0.1 * u(1, hid), u(hid, hid * hid), 0.1 * u(1, hid), u(hid, hid),
                             0.1 * u(1, 1)]).astype(np.float32)
    return X, t, params


# ------------------------------------------------------------------ prepare, run, work
def prepare(case, seed):
    kind = case["kind"]
    if kind == "pair":
        A, B = _operands(case, seed)
        a, b, c = _labels(case)
        nbytes = tnq.tnq_contract_workspace_bytes(tnq.PRECISIONS[case["precision"]], len(a), len(b), len(c))
        return {"kind": kind, "ctx": tnq.Context(0, case["precision"]), "A": A, "B": B, "a": a, "b": b, "c": c,
                "C": torch.empty(2 ** len(c), dtype=torch.complex64, device=DEVICE),
                "ws": torch.empty(nbytes, dtype=torch.uint8, device=DEVICE), "nbytes": nbytes}
    if kind == "cost_gradients":
        X, t, params = _rows(case, seed)
        ctx = tnq.Context(0, "fp32")
        model = tnq.CostModel(ctx, hidden=256, max_batch=4096)
        model.set_params(params)
        return {"kind": kind, "model": model, "X": X, "t": t}
    plan = _plan(case)
    ctx = tnq.Context(0, case["precision"])
    ctx.bind(plan)
    bits = torch.from_numpy(_bits(case, seed)).to(DEVICE)
    if kind == "noisy":
        return {"kind": kind, "ctx": ctx, "plan": plan, "bits": bits, "n_traj": case["n_traj"], "seed": seed,
                "p": torch.empty(case["n_bs"], dtype=torch.float64, device=DEVICE),
                "se": torch.empty(case["n_bs"], dtype=torch.float64, device=DEVICE)}
    if case["autotune"]:
        tnq.tnq_plan_autotune(ctx.h, plan.h, 3)
    return {"kind": kind, "ctx": ctx, "plan": plan, "bits": bits}


def run(state):
    kind = state["kind"]
    if kind == "pair":
        tnq.tnq_contract_pair(state["ctx"].h, state["A"], state["a"], state["B"], state["b"], state["C"], state["c"],
                              state["ws"], state["nbytes"])
        return state["C"]
    if kind == "amplitudes":
        return torch.view_as_complex(state["ctx"].amplitudes(state["plan"], state["bits"])).to(torch.complex64)
    if kind == "noisy":
        tnq.tnq_noisy_probabilities(state["ctx"].h, state["plan"].h, state["n_traj"], state["seed"], state["bits"],
                                    state["p"], state["se"])
        return state["p"].float(), state["se"].float()
    return state["model"].gradients(state["X"], state["t"])


def work(case):
    kind = case["kind"]
    if kind == "pair":
        m, n, k, h = case["m"], case["n"], case["k"], case["h"]
        return {"bytes": 8 * 2 ** h * (2 ** (m + k) + 2 ** (n + k) + 2 ** (m + n)), "flops": 8 * 2 ** (h + m + n + k)}
    if kind == "cost_gradients":
        d, hid = 16, 256
        params = d * hid + hid + hid * hid + hid + hid + 1
        per_row = 2 * (2 * (d * hid + hid * hid + hid)) + 2 * (hid * hid + hid)
        return {"bytes": 4 * (case["rows"] * (d + 1) + 2 * params + 1), "flops": case["rows"] * per_row}
    # flops of the contraction along the plan's path (the operation count of the
    # method); intermediates count no bytes
    passes = math.ceil(case["n_bs"] / 2 ** case["batch_log2"])
    n = case["rows"] * case["cols"]
    if kind == "noisy":
        picks, _ = _distinct(_picks(case, 1))
        passes *= math.ceil(len(picks) / 2 ** case["traj_log2"])
        return {"bytes": case["n_bs"] * (n + 16), "flops": passes * _plan(case).info["flops_per_batch"]}
    return {"bytes": case["n_bs"] * (n + 16), "flops": passes * _plan(case).info["flops_per_batch"]}


# ------------------------------------------------------------------ 64-bit values
def _picks(case, seed):
    """Kraus index of every (trajectory, channel): SplitMix64 draws as include/tnq.h states them."""
    chans = [op.mats for op in _circuit(case).ops if op.kind == "channel"]
    golden = 0x9E3779B97F4A7C15
    mask = (1 << 64) - 1
    t = np.arange(case["n_traj"], dtype=np.uint64)
    out = np.zeros((case["n_traj"], len(chans)), dtype=np.int64)
    with np.errstate(over="ignore"):
        for c, ops in enumerate(chans):
            z = np.uint64(seed & mask) + ((t << np.uint64(32)) + np.uint64(c + 1)) * np.uint64(golden)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z ^= z >> np.uint64(31)
            x = (z >> np.uint64(11)).astype(np.float64) / 2.0 ** 53
            cum = np.cumsum([np.trace(a.conj().T @ a).real / 2 for a in ops])
            out[:, c] = np.minimum(np.searchsorted(cum, x, side="right"), len(ops) - 1)
    return out


def _distinct(picks):
    return np.unique(picks, axis=0, return_counts=True)


def _apply(psi, n, qubits, u):
    """psi [T, 2^n] with u [T or 1, 2^k, 2^k] applied (qubit 0 is the most significant bit)."""
    q = sorted(qubits)
    shape, at = [psi.shape[0]], 0
    for x in q:
        shape += [2 ** (x - at), 2]
        at = x + 1
    v = psi.view(shape + [2 ** (n - at)])

    def part(t, r):
        for j, x in enumerate(qubits):
            axis = 2 + 2 * q.index(x)
            t = t.narrow(axis, (r >> (len(qubits) - 1 - j)) & 1, 1)
        return t

    out = torch.zeros_like(v)
    live = (u != 0).any(dim=0).tolist()
    ones = [1] * (v.dim() - 1)
    for r in range(2 ** len(qubits)):
        for c in range(2 ** len(qubits)):
            if live[r][c]:
                part(out, r).addcmul_(part(v, c), u[:, r, c].view(-1, *ones))
    return out.view(psi.shape)


def _states(case, picks):
    """Final states [T, 2^n] for T pick sequences; one-qubit operators are multiplied up until a pair gate needs them."""
    circ = _circuit(case)
    T, n = len(picks), circ.n
    psi = torch.zeros(T, 2 ** n, dtype=torch.complex128, device=DEVICE)
    psi[:, 0] = 1
    pending = {q: None for q in range(n)}
    chan = 0

    def flush(q):
        if pending[q] is not None:
            nonlocal psi
            psi = _apply(psi, n, (q,), torch.from_numpy(pending[q]).to(DEVICE))
            pending[q] = None

    for op in circ.ops:
        if op.kind == "channel":
            scaled = np.stack([a / math.sqrt(np.trace(a.conj().T @ a).real / 2) for a in op.mats])
            u = scaled[picks[:, chan]]
            chan += 1
        else:
            u = op.mats[0][None]
        if len(op.qubits) == 2:
            for q in op.qubits:
                flush(q)
            psi = _apply(psi, n, op.qubits, torch.from_numpy(u).to(DEVICE))
        else:
            q = op.qubits[0]
            pending[q] = u if pending[q] is None else u @ pending[q]
    for q in range(n):
        flush(q)
    return psi


def exact(case, seed):
    kind = case["kind"]
    if kind == "pair":
        a, b, c = _labels(case)
        A, B = _operands(case, seed)
        k = [x for x in a if 200 <= x < 300]
        h = [x for x in a if x >= 300]
        m, n = [x for x in a if x < 100], [x for x in b if 100 <= x < 200]
        A = _reorder(A, a, k + m + h).to(torch.complex128).view(2 ** len(h), 2 ** len(m), 2 ** len(k))
        B = _reorder(B, b, k + n + h).to(torch.complex128).view(2 ** len(h), 2 ** len(n), 2 ** len(k))
        return _reorder(torch.matmul(A, B.transpose(1, 2)).reshape(-1), n + m + h, c)
    if kind == "cost_gradients":
        X, t, params = _rows(case, seed)
        X, t, p = (torch.from_numpy(x).to(DEVICE, torch.float64) for x in (X, t, params))
        d, hid = 16, 256
        sizes = [d * hid, hid, hid * hid, hid, hid, 1]
        W1, b1, W2, b2, W3, b3 = torch.split(p, sizes)
        W1, W2, W3 = (w.to(torch.bfloat16).to(torch.float64) for w in (W1, W2, W3))  # weights are held as BF16
        W1, W2, W3 = W1.view(d, hid), W2.view(hid, hid), W3.view(hid, 1)
        z1 = X @ W1 + b1
        z2 = z1.relu() @ W2 + b2
        y = (z2.relu() @ W3 + b3)[:, 0]
        dy = (2 / len(t) * (y - t))[:, None]
        dz2 = (dy @ W3.T) * (z2 > 0)
        dz1 = (dz2 @ W2.T) * (z1 > 0)
        g = [X.T @ dz1, dz1.sum(0), z1.relu().T @ dz2, dz2.sum(0), z2.relu().T @ dy, dy.sum(0)]
        return torch.cat([x.reshape(-1) for x in g]).cpu().numpy(), float(((y - t) ** 2).mean())
    n = case["rows"] * case["cols"]
    if n > 25:
        return None  # no state vector of that size
    bits = torch.from_numpy(_bits(case, seed).astype(np.int64)).to(DEVICE)
    at = (bits << torch.arange(n - 1, -1, -1, device=DEVICE)).sum(1)
    if kind == "amplitudes":
        return _states(case, np.zeros((1, 0), dtype=np.int64))[0, at]
    picks, mult = _distinct(_picks(case, seed))
    at_once = max(1, 2 ** 25 // 2 ** n)
    p = torch.cat([_states(case, picks[i:i + at_once])[:, at].abs().square() for i in range(0, len(picks), at_once)])
    w = torch.from_numpy(mult).to(DEVICE, torch.float64)[:, None]
    nt = case["n_traj"]
    mean = (w * p).sum(0) / nt
    var = ((w * (p - mean) ** 2).sum(0) / nt).clamp(min=0)
    return mean, (var / (nt - 1)).sqrt()
