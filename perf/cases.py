"""What users of the simulator have it do, as cases that can be timed.

Each case is one whole piece of work through the public entry points
(``Simulator``, ``Batch``, ``MLP``): a circuit applied to a register, the reads
of an energy estimate, a measurement-conditioned loop, a batch of variational
circuits, a training run of the planner's cost model.  Sizes are those of the
repository's configurations, tests and benchmark, up to 30 qubits (8 GiB of
complex64 amplitudes, 64 times L2).

Results of complex64 registers are handed on as float32, the precision their
amplitudes have; those of complex128 registers as float64.
"""
import cmath
import math

import numpy as np
import torch

import circuitgen as cg
import paper_1612_08091_gb300 as q
from paper_1612_08091_gb300.qsim import MLP


def listed():
    return [
        # the 12-qubit check of a new circuit in full precision: 20 layers gate
        # by gate, the amplitudes, every read, one sample.  Calls and launches
        # count, hardly any bytes
        {"name": "check12_c128", "kind": "check", "n": 12, "depth": 20},
        # order finding of Shor's algorithm: emulated modular multiplications
        # under one recycled control qubit that is measured and reset, 22
        # rounds for an 11-bit modulus.  The shortest calls, each waited for
        {"name": "order_finding_12q", "kind": "order", "modulus": 2021, "base": 5},
        # a medium register (8 MiB, inside L2), fused: planning and launches
        # against short passes
        {"name": "random20_c64", "kind": "fused", "n": 20, "depth": 20},
        # the fused path at full size: random U3 + CNOT brickwork
        {"name": "random30_c64", "kind": "fused", "n": 30, "depth": 10},
        # one launch per gate in full precision, the path every other result is
        # checked against
        {"name": "random26_c128", "kind": "plain", "n": 26, "depth": 4, "df": False},
        # complex128 in pairs of FP32, fused at its fastest width
        {"name": "random26_c128_df", "kind": "plain", "n": 26, "depth": 8, "df": True},
        # the Fourier transform of a basis state: phase ladders between
        # Hadamards, swaps at the end
        {"name": "qft30_c64", "kind": "qft", "n": 30},
        # Grover's search: many-controlled phases between layers of H and X
        {"name": "grover28_c64", "kind": "grover", "n": 28, "iterations": 8},
        # a CNOT / Toffoli adder on a superposition of inputs
        {"name": "adder28_c64", "kind": "adder", "m": 13, "reps": 2},
        # the energy and the occupations of a trial state (the transverse-field
        # Ising sum: a chain of ZZ terms and an X on every qubit)
        {"name": "energy29_c64", "kind": "energy", "n": 29, "precision": "c64"},
        # one evaluation of a batch of variational circuits of uneven sizes
        {"name": "batch4096", "kind": "batch", "count": 4096, "nmin": 10, "nmax": 20, "lmin": 2, "lmax": 8},
        # training the planner's cost model on its timings
        {"name": "train_cost_model", "kind": "train", "samples": 11646, "hidden": 64, "batch": 256, "epochs": 10},
    ]


def _log(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["check", "order", "fused", "fused", "plain", "plain", "qft", "grover", "adder", "energy",
                       "batch", "train"])
    if kind == "check":
        return {"kind": kind, "n": rng.randint(5, 14), "depth": rng.randint(4, 24)}
    if kind == "order":
        # bases coprime to every odd modulus of this form: powers of two
        return {"kind": kind, "modulus": 2 * _log(rng, 8, 1900) + 1, "base": rng.choice([2, 4, 8])}
    if kind == "fused":
        n = rng.randint(13, 30)
        return {"kind": kind, "n": n, "depth": rng.randint(3, 10 if n > 26 else 20)}
    if kind == "plain":
        n = rng.randint(13, 26)
        return {"kind": kind, "n": n, "depth": rng.randint(2, 4 if n > 24 else 8), "df": rng.random() < 0.5}
    if kind == "qft":
        return {"kind": kind, "n": rng.randint(13, 30)}
    if kind == "grover":
        return {"kind": kind, "n": rng.randint(13, 28), "iterations": rng.randint(2, 8)}
    if kind == "adder":
        return {"kind": kind, "m": rng.randint(6, 13), "reps": rng.randint(1, 2)}
    if kind == "energy":
        precision = rng.choice(["c64", "c64", "c128"])
        return {"kind": kind, "n": rng.randint(11, 29 if precision == "c64" else 28), "precision": precision}
    if kind == "batch":
        nmin = rng.randint(4, 12)
        return {"kind": kind, "count": _log(rng, 40, 4096), "nmin": nmin, "nmax": rng.randint(nmin, 20),
                "lmin": 2, "lmax": rng.randint(2, 8)}
    batch = rng.choice([64, 100, 256, 512])
    return {"kind": kind, "samples": _log(rng, 700, 11000), "hidden": rng.choice([16, 32, 48, 64]),
            "batch": batch, "epochs": rng.randint(1, 4)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _ops(case, seed):
    """The gate list of a circuit case and the basis state it starts from."""
    kind = case["kind"]
    if kind in ("check", "fused", "plain"):
        return cg.random_u3_brickwork(case["n"], case["depth"], seed), 0
    if kind == "qft":
        return cg.qft_ops(case["n"]), cg.random_basis_state(case["n"], seed)
    if kind == "grover":
        return cg.grover_ops(case["n"], cg.grover_marked(case["n"], seed), iterations=case["iterations"]), 0
    m = case["m"]
    ang = np.random.default_rng(seed).uniform(0.2, 1.4, 2 * m + 2)
    return [cg.op("RY", (i,), (), (float(t),)) for i, t in enumerate(ang)] + cg.ripple_adder_ops(m, case["reps"]), 0


def _qubits(case):
    return 2 * case["m"] + 2 if case["kind"] == "adder" else case["n"]


def _order_inputs(case, seed):
    """Multiplication tables x -> base^(2^k) x mod N, the highest power first, and the draws."""
    N, m = case["modulus"], (case["modulus"] - 1).bit_length()
    x = np.arange(1 << m, dtype=np.uint64)
    tables = []
    for k in range(2 * m - 1, -1, -1):
        f = x.copy()
        f[:N] = (x[:N] * np.uint64(pow(case["base"], 1 << k, N))) % np.uint64(N)
        tables.append(f)
    return m, tables, np.random.default_rng(seed).uniform(0.0, 1.0, 2 * m)


def _trial_state(case, seed):
    """A product of tilted spins with a tenth of noise, normalised, as the register holds it."""
    n = case["n"]
    real = torch.float32 if case["precision"] == "c64" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    psi = torch.ones(1, dtype=real, device="cuda")
    for t in np.random.default_rng(seed).uniform(0.2, 0.8, n):
        psi = torch.outer(torch.tensor([math.cos(t / 2), math.sin(t / 2)], dtype=real, device="cuda"), psi).reshape(-1)
    out = torch.randn((1 << n, 2), generator=g, dtype=real, device="cuda").mul_(0.1 * 2.0 ** (-0.5 * (n + 1)))
    out[:, 0] += psi
    del psi
    return torch.view_as_complex(out.div_(torch.linalg.vector_norm(out.view(-1))))


def _batch_inputs(case, seed):
    # the sizes are the batch's own; the angles change from call to call
    sizes = np.random.default_rng(2016)
    nq = sizes.integers(case["nmin"], case["nmax"] + 1, case["count"])
    nl = sizes.integers(case["lmin"], case["lmax"] + 1, case["count"])
    return nq, nl, np.random.default_rng(seed).uniform(-math.pi, math.pi, int(np.sum(2 * nq * nl)))


def _train_inputs(case, seed):
    """Features and log times as the simulator's own records have them: scaled features, a smooth target with noise."""
    r = np.random.default_rng(seed)
    X = r.uniform(0.0, 1.0, (case["samples"], 16)).astype(np.float32)
    X[:, 2] = X[:, 2] > 0.5
    X[:, 15] = 1.0
    y = 3.0 * X[:, 0] + X[:, 4] * X[:, 2] - 2.0 * X[:, 11] + 0.05 * r.standard_normal(case["samples"]) - 1.0
    return X, y.astype(np.float32)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
class _Amplitudes:
    """A register's amplitudes as a device array without a copy; keeps the register alive."""

    def __init__(self, sim, typestr):
        self.sim = sim
        self.__cuda_array_interface__ = {"shape": (1 << sim.n,), "typestr": typestr, "data": (sim.state_ptr(), False),
                                         "version": 3, "strides": None}


def _view(sim):
    return torch.as_tensor(_Amplitudes(sim, "<c8" if sim.precision == q.qsim.C64 else "<c16"), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        nq, nl, angles = _batch_inputs(case, seed)
        return {"kind": kind, "batch": q.Batch(nq, nl, h=0.7), "angles": angles}
    if kind == "train":
        X, y = _train_inputs(case, seed)
        net = MLP(hidden=case["hidden"], seed=7)
        return {"kind": kind, "case": case, "net": net, "start": net.params, "X": X, "y": y}
    if kind == "order":
        m, tables, draws = _order_inputs(case, seed)
        sim = q.Simulator(m + 1, precision="c128")
        return {"kind": kind, "sim": sim, "tables": tables, "work": list(range(1, m + 1)), "draws": draws}
    if kind == "energy":
        sim = q.Simulator(case["n"], precision=case["precision"], fusion="greedy")
        _view(sim).copy_(_trial_state(case, seed))
        return {"kind": kind, "sim": sim, "terms": cg.tfim_terms(case["n"]),
                "dtype": torch.float32 if case["precision"] == "c64" else torch.float64}
    if kind in ("check", "plain"):
        df = case.get("df", False)
        sim = q.Simulator(case["n"], precision="c128", fusion="greedy" if df else "none", kmax=4, c128_df=df)
    else:
        sim = q.Simulator(_qubits(case), precision="c64", fusion="greedy")
    ops, basis = _ops(case, seed)
    return {"kind": kind, "sim": sim, "psi": _view(sim), "ops": ops, "basis": basis,
            "terms": cg.zz_chain_terms(_qubits(case)), "u": float(cg.uniform_draws(seed + 1, 1)[0])}


def _run_order(s):
    sim, bits, probs = s["sim"], [], []
    rounds = len(s["draws"])
    sim.reset(2)  # the work register holds 1, the control |0>
    for j in range(rounds):
        sim.apply_op(cg.op("H", (0,)))
        sim.apply_permutation(s["tables"][j], s["work"], [0])
        phi = -math.pi * sum(b / float(1 << (j - i)) for i, b in enumerate(bits))
        sim.apply_op(cg.op("R", (0,), (), (phi,)))
        sim.apply_op(cg.op("H", (0,)))
        b, p = sim.measure(0, s["draws"][j])
        bits.append(b)
        probs.append(p)
        if b:
            sim.apply_op(cg.op("X", (0,)))
    return {"bits": np.array(bits, dtype=np.int64), "probs": np.array(probs), "psi": sim.get_amplitudes()}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return torch.tensor(state["batch"].run(state["angles"]), dtype=torch.float32)
    if kind == "train":
        net, c = state["net"], state["case"]
        net.params = state["start"]
        loss = net.train(state["X"], state["y"], epochs=c["epochs"], batch=c["batch"], lr=3e-3)
        return {"loss": np.float32(loss), "params": net.params}
    if kind == "order":
        return _run_order(state)
    sim = state["sim"]
    if kind == "energy":
        p1, norm2 = sim.probs_all()
        return {"energy": torch.tensor(sim.expect(state["terms"]), dtype=state["dtype"]),
                "p1": torch.tensor(p1, dtype=state["dtype"]), "norm2": torch.tensor(norm2, dtype=state["dtype"])}
    sim.reset(state["basis"])
    sim.run(state["ops"])
    sim.flush()
    if kind != "check":
        return state["psi"]
    psi = sim.get_amplitudes()
    p1, norm2 = sim.probs_all()
    zz = sim.expect(state["terms"])
    return {"psi": psi, "p1": p1, "norm2": np.float64(norm2), "zz": np.float64(zz), "outcome": sim.measure_all(state["u"])}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "batch":
        nq, nl, angles = _batch_inputs(case, 0)
        # two FMAs an amplitude for each RY, one complex product for the RZ of a layer
        return {"bytes": 8 * len(angles) + 8 * len(nq), "flops": float(np.sum(2.0 ** nq * nl * (4 * nq + 6)))}
    if kind == "train":
        H, P = case["hidden"], case["hidden"] * (case["hidden"] + 19) + 1
        return {"bytes": 4 * (case["samples"] * 17 + 2 * P), "flops": 6.0 * case["epochs"] * case["samples"] * H * (H + 17)}
    if kind == "order":
        m = (case["modulus"] - 1).bit_length()
        return {"bytes": 2 * m * 8 * (1 << m) + 16 * (1 << (m + 1)), "flops": 2.0 * m * (1 << (m + 1)) * 20}
    if kind == "energy":
        N = 1 << case["n"]
        # weights, P(q=1), one product of a pair per X term, the ZZ sum
        return {"bytes": (8 if case["precision"] == "c64" else 16) * N, "flops": N * (3.0 + 4.0 * case["n"])}
    n = _qubits(case)
    ops, _ = _ops(case, 0)
    per = {"X": 0.0, "SWAP": 0.0, "H": 4.0, "RY": 4.0, "U3": 14.0, "R": 3.0, "Z": 1.0}
    flops = sum(per[o.kind] * 2.0 ** (n - len(o.controls)) for o in ops)
    return {"bytes": (16 if kind in ("check", "plain") else 8) << n, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _matrix(o):
    r, p = math.sqrt(0.5), o.params
    if o.kind == "H":
        return [[r, r], [r, -r]]
    if o.kind == "RY":
        c, s = math.cos(0.5 * p[0]), math.sin(0.5 * p[0])
        return [[c, -s], [s, c]]
    if o.kind == "U3":
        c, s = math.cos(0.5 * p[0]), math.sin(0.5 * p[0])
        return [[c, -cmath.exp(1j * p[2]) * s], [cmath.exp(1j * p[1]) * s, cmath.exp(1j * (p[1] + p[2])) * c]]
    raise ValueError(o.kind)


def _apply(psi, n, o):
    """One gate (X with controls, or a one-qubit matrix) on a complex128 vector, in place."""
    want = {o.targets[0]: None, **{c: 1 for c in o.controls}}
    at = sorted(want, reverse=True)
    shape, idx, top = [], [], n
    for b in at:
        shape += [1 << (top - b - 1), 2]
        idx += [slice(None), want[b]]
        top = b
    shape.append(1 << top)
    v = psi.view(shape)
    a, b = (v[tuple(k if i is None else i for i in idx)] for k in (0, 1))
    if o.kind == "X":
        t = a.clone()
        a.copy_(b)
        b.copy_(t)
        return
    m = _matrix(o)
    t = (a * m[0][0]).add_(b, alpha=m[0][1])
    u = (a * m[1][0]).add_(b, alpha=m[1][1])
    a.copy_(t)
    b.copy_(u)


def _circuit(case, seed):
    n = _qubits(case)
    ops, basis = _ops(case, seed)
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[basis] = 1.0
    for o in ops:
        _apply(psi, n, o)
    return psi


def _half_sums(w, n):
    """sum of w over the indices with bit b set, for every b."""
    return torch.stack([w.view(-1, 2, 1 << b)[:, 1].sum() for b in range(n)])


def _zz(w, n):
    """sum_i w_i sum_k (-1)^(bit k + bit k+1 of i)."""
    total = 0.0
    for b in range(n - 1):
        v = w.view(-1, 2, 2, 1 << b)
        total += float((v[:, 0, 0].sum() + v[:, 1, 1].sum() - v[:, 0, 1].sum() - v[:, 1, 0].sum()))
    return total


def _exact_check(case, seed):
    n, psi = case["n"], _circuit(case, seed)
    w = psi.real ** 2 + psi.imag ** 2
    total = float(w.sum())
    c = np.cumsum(w.cpu().numpy())
    j = int(np.searchsorted(c, float(cg.uniform_draws(seed + 1, 1)[0]) * total, side="right"))
    return {"psi": psi, "p1": _half_sums(w, n), "norm2": np.float64(total), "zz": np.float64(_zz(w, n)), "outcome": j}


def _exact_order(case, seed):
    m, tables, draws = _order_inputs(case, seed)
    r = math.sqrt(0.5)
    psi = np.zeros((1 << m, 2), dtype=np.complex128)  # [work, control]
    psi[1, 0] = 1.0
    bits, probs = [], []
    for j, u in enumerate(draws):
        a, b = (psi[:, 0] + psi[:, 1]) * r, (psi[:, 0] - psi[:, 1]) * r
        moved = np.empty_like(b)
        moved[tables[j].astype(np.int64)] = b
        b = moved * cmath.exp(-1j * math.pi * sum(x / float(1 << (j - i)) for i, x in enumerate(bits)))
        a, b = (a + b) * r, (a - b) * r
        s = [float(np.sum(np.abs(a) ** 2)), float(np.sum(np.abs(b) ** 2))]
        x = 0 if u * (s[0] + s[1]) < s[0] else 1
        bits.append(x)
        probs.append(s[x] / (s[0] + s[1]))
        psi = np.zeros_like(psi)
        psi[:, 0] = (b if x else a) / math.sqrt(s[x])
    return {"bits": np.array(bits, dtype=np.int64), "probs": np.array(probs), "psi": psi.reshape(-1)}


def _exact_energy(case, seed):
    n, psi = case["n"], _trial_state(case, seed).to(torch.complex128)
    v = torch.view_as_real(psi)
    x = 0.0
    for b in range(n):
        p = v.view(-1, 2, 1 << b, 2)
        x += 2.0 * float(torch.sum(p[:, 0] * p[:, 1]))
    w = v.square().sum(-1)
    return {"energy": np.float64(-_zz(w, n) - 0.7 * x), "p1": _half_sums(w, n), "norm2": np.float64(float(w.sum()))}


def _exact_batch(case, seed):
    nq, nl, angles = _batch_inputs(case, seed)
    off = np.concatenate([[0], np.cumsum(2 * nq * nl)])
    energy = np.zeros(len(nq))
    for n, L in sorted(set(zip(nq.tolist(), nl.tolist()))):
        ids = np.flatnonzero((nq == n) & (nl == L))
        y = torch.arange(1 << n, device="cuda")
        src = (y ^ (y << 1)) & ((1 << n) - 1)
        zz = torch.full((1 << n,), float(n - 1), dtype=torch.float64, device="cuda")
        for b in range(n - 1):
            zz -= 2.0 * (((y >> b) ^ (y >> (b + 1))) & 1)
        for lo in range(0, len(ids), max(1, (1 << 26) >> n)):
            part = ids[lo:lo + max(1, (1 << 26) >> n)]
            B = len(part)
            ang = torch.tensor(np.stack([angles[off[i]:off[i + 1]] for i in part]), device="cuda").view(B, L, 2, n)
            psi = torch.zeros((B, 1 << n), dtype=torch.complex128, device="cuda")
            psi[:, 0] = 1.0
            for l in range(L):
                v = torch.view_as_real(psi)
                phase = torch.zeros((B, 1 << n), dtype=torch.float64, device="cuda")
                for b in range(n):
                    c = torch.cos(0.5 * ang[:, l, 0, b]).view(B, 1, 1, 1)
                    s = torch.sin(0.5 * ang[:, l, 0, b]).view(B, 1, 1, 1)
                    w = v.view(B, -1, 2, 1 << b, 2)
                    w0, w1 = w[:, :, 0], w[:, :, 1]
                    t = torch.addcmul(w0 * c, w1, s, value=-1.0)
                    w1.copy_(torch.addcmul(w1 * c, w0, s))
                    w0.copy_(t)
                    phi = 0.5 * ang[:, l, 1, b].view(B, 1, 1)
                    f = phase.view(B, -1, 2, 1 << b)
                    f[:, :, 0] -= phi
                    f[:, :, 1] += phi
                psi = (psi * torch.complex(torch.cos(phase), torch.sin(phase)))[:, src]
            v = torch.view_as_real(psi)
            e = -(v.square().sum(-1) @ zz)
            for b in range(n):
                w = v.reshape(B, -1, 2, (1 << b) * 2)
                e -= 0.7 * 2.0 * (w[:, :, 0] * w[:, :, 1]).sum((1, 2))
            energy[part] = e.cpu().numpy()
    return torch.tensor(energy)


def _exact_train(case, seed):
    X, T = (a.astype(np.float64) for a in _train_inputs(case, seed))
    H, n = case["hidden"], case["samples"]
    p = MLP(hidden=H, seed=7).params.astype(np.float64)  # the start, an input
    cut = np.cumsum([16 * H, H, H * H, H, H])
    m, v, step, b1, b2 = np.zeros_like(p), np.zeros_like(p), 0, float(np.float32(0.9)), float(np.float32(0.999))
    lr, eps, loss = float(np.float32(3e-3)), float(np.float32(1e-8)), 0.0
    for ep in range(case["epochs"]):
        total = 0.0
        for s0 in range(0, n, case["batch"]):
            x, t = X[s0:s0 + case["batch"]], T[s0:s0 + case["batch"]]
            W1, c1, W2, c2, w3, c3 = np.split(p, cut)
            W1, W2 = W1.reshape(H, 16), W2.reshape(H, H)
            h1 = np.maximum(x @ W1.T + c1, 0.0)
            h2 = np.maximum(h1 @ W2.T + c2, 0.0)
            r = h2 @ w3 + c3[0] - t
            total += float(np.sum(r * r))
            dy = 2.0 * r / len(t)
            d2 = np.outer(dy, w3) * (h2 > 0)
            d1 = (d2 @ W2) * (h1 > 0)
            g = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), h2.T @ dy, [dy.sum()]])
            step += 1
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            p = p - lr * (m / (1 - b1 ** step)) / (np.sqrt(v / (1 - b2 ** step)) + eps)
        loss = total / n
    return {"loss": np.float64(loss), "params": p}


def exact(case, seed):
    kind = case["kind"]
    if kind == "qft":
        n, x = case["n"], int(_ops(case, seed)[1])
        y = torch.arange(1 << n, device="cuda")
        y = y.mul_(x).bitwise_and_((1 << n) - 1).double().mul_(2.0 * math.pi / float(1 << n))
        return torch.polar(torch.full_like(y, 2.0 ** (-0.5 * n)), y)
    if kind == "grover":
        n, r = case["n"], case["iterations"]
        theta = math.asin(2.0 ** (-0.5 * n))
        rest = math.cos((2 * r + 1) * theta) / math.sqrt(float((1 << n) - 1))
        psi = torch.full((1 << n,), (-1) ** r * rest, dtype=torch.complex128, device="cuda")
        psi[cg.grover_marked(n, seed)] = (-1) ** r * math.sin((2 * r + 1) * theta)
        return psi
    if kind in ("fused", "plain", "adder"):
        return _circuit(case, seed)
    return {"check": _exact_check, "order": _exact_order, "energy": _exact_energy, "batch": _exact_batch,
            "train": _exact_train}[kind](case, seed)
