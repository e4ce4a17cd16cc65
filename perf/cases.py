"""What is timed: the calls that programs built on this framework make, over the sizes they make them at.

A case names an entry point (``call``), a workload and its sizes.  The circuits are the
evaluated programs of the method (GHZ, Deutsch-Jozsa, QFT), random layered circuits (U3 on
every qubit, CNOTs on seeded pairs) and random mixed steps, drawn here with numpy so that
making thousands of circuits takes no longer than running them.  ``exact`` applies the same
gates in complex128 with plain torch.

Floors (``work``): every input read once, every output written once, and the real
operations of the per-gate update on 2^n amplitudes (14 per amplitude for a dense 2x2
gate, half of that under a control, 6 and 3 for phases, 2 for a Hadamard, none for X, CNOT
and SWAP).
"""
import math

import numpy as np
import torch

from paper_2305_14398_gb300 import binding as B

ID = B.GATE_IDS
X, H, U3, CX, CP, SWAP = ID["x"], ID["h"], ID["u3"], ID["cx"], ID["cp"], ID["swap"]
# random mixed steps draw uniformly from these; the last three take a second qubit
MIXED = np.array([ID[g] for g in ("h", "x", "y", "z", "s", "t", "rx", "ry", "rz", "cx", "cz", "cp")], dtype=np.int32)
TWO = (ID["cx"], ID["cz"], ID["cp"], ID["cu"], ID["swap"])
PRECS = {"fp32": B.PREC_FP32_SIMT, "bf16x3": B.PREC_TC_BF16X3, "tf32x3": B.PREC_TC_TF32X3}


def listed():
    return [
        # The smallest whole call: a 5-qubit QFT on a basis state with probabilities and norm,
        # what a program asks for interactively or inside a parameter loop: latency.
        {"name": "simulate_qft_5", "call": "simulate", "kind": "qft", "n": 5, "layers": 0, "probs": True},
        # One 11-qubit QFT on a basis state (the evaluated size): an ordinary single call.
        {"name": "simulate_qft_11", "call": "simulate", "kind": "qft", "n": 11, "layers": 0, "probs": True},
        # One circuit at the fused kernels' limit of 16 qubits, dense layers: the largest single call there.
        {"name": "simulate_layered_16", "call": "simulate", "kind": "layered", "n": 16, "layers": 10, "probs": False},
        # The benchmark's batch: the evaluated 11-qubit programs, states, probabilities and norms.
        {"name": "batch_paper_11", "call": "batch", "kind": "paper", "count": 16384, "n_lo": 11, "n_hi": 11, "probs": True},
        # A batch of random circuits of uneven size and depth (4 to 14 qubits, 5 to 40 steps): full states.
        {"name": "batch_mixed_4_14", "call": "batch", "kind": "mixed", "count": 4096, "n_lo": 4, "n_hi": 14, "probs": False},
        # A batch of wide random circuits only: arithmetic, one circuit per CTA.
        {"name": "batch_mixed_14", "call": "batch", "kind": "mixed", "count": 1024, "n_lo": 14, "n_hi": 14, "probs": False},
        # Measurement statistics of a batch: 64 shots from each of 16384 11-qubit states.
        {"name": "sample_11", "call": "sample", "n": 11, "count": 16384, "shots": 64},
        # Probabilities and norm of one large state.
        {"name": "probabilities_24", "call": "probabilities", "n": 24, "zeros": 0},
        # A wide circuit on a state held in memory (512 MB), dense layers.
        {"name": "fsv_layered_26", "call": "fsv", "kind": "layered", "n": 26, "layers": 10},
        # The unitary of a 12-qubit circuit on the tensor cores, three layers (at 8 the BF16
        # split's own error, 2e-5, is as much as two correct results may differ by: deeper
        # circuits take the other precisions).
        {"name": "unitary_bf16x3_12", "call": "unitary", "prec": "bf16x3", "kind": "layered", "n": 12, "layers": 3},
        # The unitary of a 10-qubit circuit in full FP32, for those who check others against it.
        {"name": "unitary_fp32_10", "call": "unitary", "prec": "fp32", "kind": "layered", "n": 10, "layers": 20},
        # One step's dense matrix (Kronecker product of its gates), as programs export operators.
        {"name": "step_matrix_12", "call": "step", "kind": "layered", "n": 12, "layers": 1, "step": 0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    call = rng.choice(["simulate", "batch", "batch", "sample", "probabilities", "fsv", "unitary", "step"])
    if call == "simulate":
        kind = rng.choice(["dj", "qft", "layered"])
        layers = rng.randint(1, 20) if kind == "layered" else 0
        return {"call": call, "kind": kind, "n": rng.randint(5, 16), "layers": layers, "probs": kind != "layered"}
    if call == "batch":
        if rng.random() < 0.5:
            n = rng.randint(4, 13)
            return {"call": call, "kind": "paper", "count": _log_int(rng, 16, min(20000, (1 << 25) >> n)), "n_lo": n, "n_hi": n, "probs": True}
        hi = rng.randint(5, 16)
        lo = rng.randint(4, hi)
        return {"call": call, "kind": "mixed", "count": _log_int(rng, 8, min(4096, (1 << 24) >> hi)), "n_lo": lo, "n_hi": hi, "probs": False}
    if call == "sample":
        n = rng.randint(5, 20)
        return {"call": call, "n": n, "count": _log_int(rng, 1, min(16384, (1 << 25) >> n)), "shots": _log_int(rng, 1, 1000)}
    if call == "probabilities":
        n = rng.randint(8, 26)
        return {"call": call, "n": n, "zeros": rng.choice([0, rng.randint(1, n - 1)])}
    if call == "fsv":
        kind = rng.choice(["layered", "layered", "qft"])
        return {"call": call, "kind": kind, "n": rng.randint(14, 26), "layers": rng.randint(2, 10) if kind == "layered" else 0}
    if call == "unitary":
        prec = rng.choice(["fp32", "bf16x3", "bf16x3", "tf32x3"])
        kind = "layered" if prec == "bf16x3" else rng.choice(["layered", "qft"])
        layers = 0 if kind == "qft" else rng.randint(2, {"fp32": 20, "tf32x3": 8, "bf16x3": 3}[prec])
        return {"call": call, "prec": prec, "kind": kind, "n": rng.randint(7, 10 if prec == "fp32" else 12), "layers": layers}
    layers = rng.randint(2, 40)
    return {"call": call, "kind": "mixed", "n": rng.randint(6, 13), "layers": layers, "step": rng.randrange(layers)}


# ---------------------------------------------------------------- circuits
# A circuit is four arrays (kind, qubits [G, 2], params [G, 8]) in program order.

def _gates(rows):
    g = len(rows)
    kind, qub, par = np.zeros(g, np.int32), np.zeros((g, 2), np.int32), np.zeros((g, 8))
    for i, (k, q, p) in enumerate(rows):
        kind[i] = k
        qub[i, : len(q)] = q
        par[i, : len(p)] = p
    return kind, qub, par


def _ghz(n):
    return _gates([(H, (0,), ())] + [(CX, (i, i + 1), ()) for i in range(n - 1)])


def _qft(n):
    rows = []
    for j in range(n - 1, -1, -1):
        rows.append((H, (j,), ()))
        rows += [(CP, (k, j), (math.pi / (1 << (j - k)),)) for k in range(j - 1, -1, -1)]
    return _gates(rows + [(SWAP, (i, n - 1 - i), ()) for i in range(n // 2)])


def _xs(qubits):
    qubits = np.asarray(qubits, np.int32)
    g = len(qubits)
    qub = np.zeros((g, 2), np.int32)
    qub[:, 0] = qubits
    return np.full(g, X, np.int32), qub, np.zeros((g, 8))


def _join(*parts):
    return tuple(np.concatenate(a) for a in zip(*parts))


def _basis(n, x):
    return _xs([q for q in range(n) if (x >> q) & 1])


def _hs(m):
    k, q, p = _xs(np.arange(m))
    return np.full_like(k, H), q, p


def _dj(n, balanced, g):
    anc = n - 1
    if not balanced:
        oracle = _xs([anc] if g.random() < 0.5 else [])
    else:
        chosen = np.flatnonzero(g.random(n - 1) < 0.5)
        if not len(chosen):
            chosen = np.array([int(g.integers(0, n - 1))])
        mask = _xs(np.flatnonzero(g.random(n - 1) < 0.5))
        qub = np.stack([chosen, np.full(len(chosen), anc)], 1).astype(np.int32)
        oracle = _join(mask, (np.full(len(chosen), CX, np.int32), qub, np.zeros((len(chosen), 8))), mask)
    return _join(_xs([anc]), _hs(n), oracle, _hs(n - 1))


def _layered(n, layers, g, cnots=True):
    rows = []
    for _ in range(layers):
        ang = g.uniform(0.0, 2.0 * math.pi, size=(n, 3))
        rows += [(U3, (q,), ang[q]) for q in range(n)]
        if cnots:
            perm = g.permutation(n)
            for p in range(n // 2):
                a, b = int(perm[2 * p]), int(perm[2 * p + 1])
                rows.append((CX, (a, b) if g.random() < 0.5 else (b, a), ()))
    return _gates(rows)


def _mixed_steps(n, steps, g):
    """`steps` random dense steps of n qubits: (step of each gate, kind, qubits, params)."""
    perm = np.argsort(g.random((steps, n)), axis=1).astype(np.int32)
    at, rows = np.zeros(steps, np.int64), np.arange(steps)
    got = []
    for _ in range(n):
        on = at < n
        pick = g.integers(0, len(MIXED), steps)
        pick = np.where((pick >= 9) & (at + 1 >= n), g.integers(0, 9, steps), pick)
        kind, ang = MIXED[pick], g.uniform(0.0, 2.0 * math.pi, steps)
        two = pick >= 9
        q = perm[rows, np.minimum(at, n - 1)]
        t = np.where(two, perm[rows, np.minimum(at + 1, n - 1)], 0)
        par = np.where((pick == 11) | ((pick >= 6) & (pick <= 8)), ang, 0.0)
        got.append((rows[on], at[on], kind[on], np.stack([q, t], 1)[on], par[on]))
        at = at + np.where(two, 2, 1)
    step, pos, kind, qub, par0 = (np.concatenate(a) for a in zip(*got))
    o = np.lexsort((pos, step))
    par = np.zeros((len(o), 8))
    par[:, 0] = par0[o]
    return step[o], kind[o], qub[o].astype(np.int32), par


def _circuit(case, g):
    n, kind = case["n"], case["kind"]
    if kind == "dj":
        return _dj(n, True, g)
    if kind == "qft":
        if case["call"] == "simulate":
            return _join(_basis(n, int(g.integers(0, 1 << n))), _qft(n))
        return _join(_layered(n, 1, g, cnots=False), _qft(n))  # every entry differs with the seed
    return _layered(n, case["layers"], g)


def _steps(case, g):
    """A circuit whose steps are dense: (step of each gate, kind, qubits, params)."""
    if case["kind"] == "layered":
        gates = _layered(case["n"], 1, g, cnots=False)
        return np.zeros(len(gates[0]), np.int64), *gates
    return _mixed_steps(case["n"], case["layers"], g)


def _batch(case, g):
    """(qubits of each circuit, gate offsets, kind, qubits, params)."""
    count, lo, hi = case["count"], case["n_lo"], case["n_hi"]
    if case["kind"] == "paper":
        n, ghz, qft, parts = lo, _ghz(lo), _qft(lo), []
        for i in range(count):
            kind = i % 4
            if kind == 0:
                parts.append(ghz)
            elif kind == 3:
                parts.append(_basis(n, int(g.integers(0, 1 << n))))
                parts.append(qft)
            else:
                parts.append(_dj(n, kind == 2, g))
        size, k = np.zeros(count, np.int64), 0
        for i in range(count):
            for _ in range(2 if i % 4 == 3 else 1):
                size[i] += len(parts[k][0])
                k += 1
        return np.full(count, n, np.int32), np.concatenate([[0], np.cumsum(size)]), *_join(*parts)
    sizes = np.random.default_rng([3, count, lo, hi])  # sizes and depths are the case's, the gates the seed's
    ns = np.minimum(hi, np.exp(sizes.uniform(math.log(lo), math.log(hi + 1), count)).astype(np.int32)).astype(np.int32)
    depth = sizes.integers(5, 41, count)
    owner, parts = [], []
    for n in np.unique(ns):
        mine = np.flatnonzero(ns == n)
        step, *gates = _mixed_steps(int(n), int(depth[mine].sum()), g)
        owner.append(np.repeat(mine, depth[mine])[step])
        parts.append(gates)
    owner = np.concatenate(owner)
    o = np.argsort(owner, kind="stable")
    off = np.concatenate([[0], np.cumsum(np.bincount(owner, minlength=count))])
    return ns, off, *(a[o] for a in _join(*parts))


# ---------------------------------------------------------------- state

class Owned:
    """A library handle, destroyed with the state that holds it."""

    def __init__(self, handle, destroy):
        self.h, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.h)


def _handle(n, gates):
    c = B.tqs_circuit_create(n)
    for k, q, p in zip(*gates):
        k = int(k)
        B.tqs_add_gate(c, k, [int(q[0]), int(q[1])] if k in TWO else [int(q[0])], [float(v) for v in p])
    return Owned(c, B.tqs_circuit_destroy)


def _rng(seed):
    return np.random.default_rng([14398, int(seed)])


def _normal(seed, *shape):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)


def _state(seed, n):
    """A random normalised state of n qubits."""
    v = _normal(seed, 1 << n, 2)
    v /= torch.linalg.vector_norm(v)
    return torch.view_as_complex(v)


def _sample_inputs(case, seed):
    """Probabilities of `count` random states and one uniform per shot."""
    p = _normal(seed, case["count"], 1 << case["n"], 2).square().sum(-1).double()
    p /= p.sum(-1, keepdim=True)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    u = torch.rand(case["count"] * case["shots"], generator=gen, device="cuda", dtype=torch.float64)
    return p.reshape(-1), u


def prepare(case, seed):
    call, g = case["call"], _rng(seed)
    c64 = {"dtype": torch.complex64, "device": "cuda"}
    f64 = {"dtype": torch.float64, "device": "cuda"}
    st = {"case": case}
    if call in ("batch", "sample"):
        if call == "batch":
            st["b"] = Owned(B.tqs_batch_create_packed(*_batch(case, g)), B.tqs_batch_destroy)
            count, total, _ = B.tqs_batch_info(st["b"].h)
            st["states"] = torch.empty(total, **c64)
            st["probs"] = torch.empty(total, **f64) if case["probs"] else None
            st["norms"] = torch.empty(count, **f64) if case["probs"] else None
        else:
            # the sampled batch: its circuits fix the layout, the probabilities are given
            one = _hs(case["n"])
            m, g1 = case["count"], len(one[0])
            packed = [np.full(m, case["n"], np.int32), np.arange(m + 1) * g1, *(np.tile(a, (m,) + (1,) * (a.ndim - 1)) for a in one)]
            st["b"] = Owned(B.tqs_batch_create_packed(*packed), B.tqs_batch_destroy)
            st["probs"], st["u"] = _sample_inputs(case, seed)
            st["out"] = torch.empty(m * case["shots"], dtype=torch.int64, device="cuda")
        return st
    n = case["n"]
    if call == "probabilities":
        st["state"] = _state(seed, n)
        st["probs"], st["total"] = torch.empty(1 << n, **f64), torch.empty(1, **f64)
        st["zero"] = torch.empty(1, **f64) if case["zeros"] else None
        return st
    st["c"] = _handle(n, _steps(case, g)[1:] if call == "step" else _circuit(case, g))
    if call == "simulate":
        st["out"] = torch.empty(1 << n, **c64)
        st["probs"] = torch.empty(1 << n, **f64) if case["probs"] else None
        st["norm"] = torch.empty(1, **f64) if case["probs"] else None
    elif call == "fsv":
        st["init"] = _state(seed, n)
        st["state"] = torch.empty_like(st["init"])
    else:
        st["U"] = torch.empty((1 << n, 1 << n), **c64)
    return st


def run(st):
    case = st["case"]
    call = case["call"]
    if call == "simulate":
        B.tqs_simulate(st["c"].h, st["out"], probs=st["probs"], norm=st["norm"])
        return [st["out"], st["probs"], st["norm"]] if case["probs"] else [st["out"]]
    if call == "batch":
        B.tqs_batch_run(st["b"].h, st["states"], st["probs"], st["norms"])
        return [st["states"], st["probs"], st["norms"]] if case["probs"] else [st["states"]]
    if call == "sample":
        B.tqs_batch_sample(st["b"].h, st["probs"], case["shots"], st["u"], st["out"])
        return [st["out"]]
    if call == "probabilities":
        B.tqs_probabilities(st["state"], case["n"], st["probs"], st["total"])
        if not case["zeros"]:
            return [st["probs"], st["total"]]
        # the probability that a register (the lowest qubits) reads 0
        B.tqs_marginal_zero(st["state"], case["n"], (1 << case["zeros"]) - 1, st["zero"])
        return [st["probs"], st["total"], st["zero"]]
    if call == "fsv":
        st["state"].copy_(st["init"])  # the call works in place: the program keeps its input state
        B.tqs_simulate_fsv(st["c"].h, st["state"])
        return [st["state"]]
    if call == "unitary":
        B.tqs_circuit_unitary(st["c"].h, PRECS[case["prec"]], st["U"])
        return [st["U"]]
    B.tqs_materialize_step(st["c"].h, case["step"], st["U"])
    return [st["U"]]


# ---------------------------------------------------------------- floors

_FLOPS = {ID["h"]: 2, ID["x"]: 0, ID["y"]: 0, ID["z"]: 0, ID["s"]: 0, ID["t"]: 3, ID["rx"]: 8, ID["ry"]: 6, ID["rz"]: 6,
          U3: 14, CX: 0, ID["cz"]: 0, CP: 1.5, SWAP: 0}


def _gate_flops(kind):
    """Operations per amplitude of a gate list."""
    table = np.zeros(max(_FLOPS) + 1)
    for k, v in _FLOPS.items():
        table[k] = v
    return table[kind]


def work(case):
    call, g = case["call"], _rng(1)
    gate_bytes = 12  # kind and qubits, one angle
    if call == "batch":
        ns, off, kind, _, _ = _batch(case, g)
        per = _gate_flops(kind)
        amps = (1 << ns.astype(np.int64))
        flops = float((np.add.reduceat(np.append(per, 0.0), off[:-1]) * amps).sum())
        out = int(amps.sum()) * (16 if case["probs"] else 8) + (8 * len(ns) if case["probs"] else 0)
        return {"bytes": out + gate_bytes * len(kind), "flops": flops}
    n = case["n"]
    N = 1 << n
    if call == "sample":
        m, s = case["count"], case["shots"]
        return {"bytes": 8 * m * N + 16 * m * s, "flops": m * (N + s * n)}
    if call == "probabilities":
        return {"bytes": 16 * N + 8, "flops": 4 * N + (N >> case["zeros"]) * (case["zeros"] > 0)}
    if call == "step":
        # the dense matrix is the output; an entry is a product of 2x2 entries shared along rows and columns
        return {"bytes": 8 * N * N, "flops": 6 * N * N}
    kind = _circuit(case, g)[0]
    flops = float(_gate_flops(kind).sum()) * N
    if call == "simulate":
        return {"bytes": N * (16 if case["probs"] else 8) + gate_bytes * len(kind), "flops": flops}
    if call == "fsv":
        return {"bytes": 16 * N + gate_bytes * len(kind), "flops": flops}
    # every column of the unitary is the circuit applied to a basis state
    return {"bytes": 8 * N * N + gate_bytes * len(kind), "flops": flops * N}


# ---------------------------------------------------------------- exact values

def _mat(kind, p):
    """2x2 matrices [G, 2, 2] of gates (the controlled matrix of a controlled gate)."""
    G = len(kind)
    m = np.zeros((G, 2, 2), np.complex128)
    m[:, 0, 0] = m[:, 1, 1] = 1.0
    th = p[:, 0]
    is_ = lambda *names: np.isin(kind, [ID[x] for x in names])  # noqa: E731
    r = 1.0 / math.sqrt(2.0)
    m[is_("h")] = [[r, r], [r, -r]]
    m[is_("x", "cx")] = [[0, 1], [1, 0]]
    m[is_("y")] = [[0, -1j], [1j, 0]]
    m[is_("z", "cz"), 1, 1] = -1
    m[is_("s"), 1, 1] = 1j
    m[is_("t"), 1, 1] = np.exp(0.25j * math.pi)
    k = is_("cp")
    m[k, 1, 1] = np.exp(1j * th[k])
    k = is_("rz")
    m[k, 0, 0], m[k, 1, 1] = np.exp(-0.5j * th[k]), np.exp(0.5j * th[k])
    c, s = np.cos(th / 2), np.sin(th / 2)
    k = is_("rx")
    m[k, 0, 0] = m[k, 1, 1] = c[k]
    m[k, 0, 1] = m[k, 1, 0] = -1j * s[k]
    k = is_("ry")
    m[k, 0, 0] = m[k, 1, 1] = c[k]
    m[k, 0, 1], m[k, 1, 0] = -s[k], s[k]
    k = is_("u3")
    m[k, 0, 0], m[k, 0, 1] = c[k], -np.exp(1j * p[k, 2]) * s[k]
    m[k, 1, 0], m[k, 1, 1] = np.exp(1j * p[k, 1]) * s[k], np.exp(1j * (p[k, 1] + p[k, 2])) * c[k]
    return m


def _expand(kind, qub, par):
    """(matrices, target masks, control masks); a SWAP becomes three CNOTs."""
    sw = np.flatnonzero(kind == SWAP)
    rep = np.where(kind == SWAP, 3, 1)
    kind2, qub2, par2 = np.repeat(kind, rep), np.repeat(qub, rep, axis=0).copy(), np.repeat(par, rep, axis=0)
    kind2[kind2 == SWAP] = CX
    mid = (np.cumsum(rep) - rep)[sw] + 1
    qub2[mid] = qub2[mid][:, ::-1]
    two = np.isin(kind2, TWO)
    tq = np.where(two, qub2[:, 1], qub2[:, 0])
    return _mat(kind2, par2), 1 << tq.astype(np.int64), np.where(two, 1 << qub2[:, 0].astype(np.int64), 0)


def _apply(psi, mats, tmask, cmask):
    """Apply gate slot after gate slot to psi [C, 2^n]: mats [C or 1, G, 2, 2], masks [C or 1, G]."""
    N = psi.shape[1]
    idx = torch.arange(N, device="cuda")[None]
    mats, tmask, cmask = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda") for a in (mats, tmask, cmask))
    for k in range(mats.shape[1]):
        t, c, m = tmask[:, k, None], cmask[:, k, None], mats[:, k]
        other = idx ^ t
        flip = torch.gather(psi, 1, other.expand(psi.shape)) if other.shape[0] == psi.shape[0] else psi[:, other[0]]
        bit = (idx & t) != 0
        on = (idx & c) == c
        one = torch.ones((), dtype=psi.dtype, device="cuda")
        same = torch.where(on, torch.where(bit, m[:, 1, 1, None], m[:, 0, 0, None]), one)
        cross = torch.where(on, torch.where(bit, m[:, 1, 0, None], m[:, 0, 1, None]), 0 * one)
        psi = psi.mul_(same).add_(flip.mul_(cross))
    return psi


def _zero_states(count, n):
    psi = torch.zeros((count, 1 << n), dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1.0
    return psi


def _exact_batch(case, seed):
    ns, off, kind, qub, par = _batch(case, _rng(seed))
    amps = np.concatenate([[0], np.cumsum(1 << ns.astype(np.int64))])
    out = torch.empty(int(amps[-1]), dtype=torch.complex128, device="cuda")
    for n in np.unique(ns):
        mine = np.flatnonzero(ns == n)
        parts = [_expand(kind[off[i]:off[i + 1]], qub[off[i]:off[i + 1]], par[off[i]:off[i + 1]]) for i in mine]
        most = max(len(p[1]) for p in parts)
        mats = np.zeros((len(mine), most, 2, 2), np.complex128)
        mats[:, :, 0, 0] = mats[:, :, 1, 1] = 1.0
        tm, cm = np.ones((len(mine), most), np.int64), np.zeros((len(mine), most), np.int64)
        for i, (m, t, c) in enumerate(parts):
            mats[i, : len(t)], tm[i, : len(t)], cm[i, : len(t)] = m, t, c
        room = max(1, (1 << 25) >> int(n))  # states at a time
        for a in range(0, len(mine), room):
            psi = _apply(_zero_states(len(mine[a:a + room]), int(n)), mats[a:a + room], tm[a:a + room], cm[a:a + room])
            for j, i in enumerate(mine[a:a + room]):
                out[amps[i]:amps[i + 1]] = psi[j]
    if not case["probs"]:
        return [out]
    p = torch.view_as_real(out).square().sum(-1)
    norms = torch.stack([v.sum() for v in torch.split(p, (1 << ns.astype(np.int64)).tolist())])
    return [out, p, norms]


def exact(case, seed):
    call, g = case["call"], _rng(seed)
    if call == "batch":
        return _exact_batch(case, seed)
    if call == "sample":
        return None  # whole numbers
    n = case["n"]
    if call == "probabilities":
        p = torch.view_as_real(_state(seed, n)).double().square().sum(-1)
        return [p, p.sum().reshape(1)] + ([p[:: 1 << case["zeros"]].sum().reshape(1)] if case["zeros"] else [])
    if call == "step":
        step, *gates = _steps(case, g)
        gates = [a[step == case["step"]] for a in gates]
    else:
        gates = _circuit(case, g)
    args = tuple(a[None] for a in _expand(*gates))
    if call == "simulate":
        psi = _apply(_zero_states(1, n), *args).reshape(-1)
        if not case["probs"]:
            return [psi]
        p = torch.view_as_real(psi).square().sum(-1)
        return [psi, p, p.sum().reshape(1)]
    if call == "fsv":
        return [_apply(_state(seed, n).to(torch.complex128)[None], *args).reshape(-1)]
    return [_apply(torch.eye(1 << n, dtype=torch.complex128, device="cuda"), *args).T.contiguous()]
