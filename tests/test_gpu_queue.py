"""Gates queued by name in one call against one call per gate, and the
tensor-core operand images built on the device: gates of every kind inside a
block, blocks whose gates take more room than their matrix, more blocks than
one launch builds, 5-qubit and padded 4-qubit blocks."""
import numpy as np
import pytest

import circuitgen as cg
from helpers import infidelity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1612_08091_gb300 as q

    q.load()
    return q


def mixed_ops(n, count, seed, wires=None):
    """Every named kind and explicit matrices, with and without controls."""
    r = np.random.default_rng(seed)
    wires = list(range(n)) if wires is None else list(wires)
    kinds = ["H", "X", "Y", "Z", "S", "T", "SWAP", "RX", "RY", "RZ", "R", "U3", "MAT"]
    ops = []
    for i in range(count):
        k = kinds[i % len(kinds)]
        t = 2 if k == "SWAP" else int(r.integers(1, 4)) if k == "MAT" else 1
        q = [int(v) for v in r.permutation(wires)[:t + int(r.integers(0, 3))]]
        if len(q) < t:
            continue
        npar = {"RX": 1, "RY": 1, "RZ": 1, "R": 1, "U3": 3}.get(k, 0)
        params = tuple(float(v) for v in r.uniform(-7, 7, npar))
        if k == "MAT":
            params = (cg.random_unitary(1 << t, int(r.integers(1 << 30))),)
        ops.append(cg.op(k, q[:t], q[t:], params))
    return ops


@pytest.mark.parametrize("n", [3, 9])
def test_named_gates_equal_single_calls(qs, n):
    ops = mixed_ops(n, 130, seed=n, wires=range(n))
    ops = [o for o in ops if len(o.targets) + len(o.controls) <= n]
    out = []
    for whole in (True, False):
        with qs.Simulator(n, precision="c128") as sim:
            if whole:
                sim.run(iter(ops))
            else:
                for o in ops:
                    sim.apply_op(o)
            out.append((sim.get_amplitudes(), sim.stats()["gates"]))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1] == len(ops)


@pytest.mark.parametrize("bad,status", [
    (cg.op("H", (9,)), "ERANGE"), (cg.op("X", (1,), (1,)), "EDUP"), (cg.op("H", (-1,)), "ERANGE"),
    (cg.op("RZ", (0,), (), (float("nan"),)), "ENONFINITE"),
])
def test_a_refused_gate_keeps_the_ones_before_it(qs, bad, status):
    ops = [cg.op("H", (0,)), cg.op("X", (1,), (0,)), bad, cg.op("X", (2,))]
    with qs.Simulator(3, precision="c128") as sim:
        with pytest.raises(qs.QsimError) as e:
            sim.run(ops)
        psi = sim.get_amplitudes()
        gates = sim.stats()["gates"]
    assert e.value.status == status and "sim_apply" in str(e.value)
    assert gates == 2
    np.testing.assert_allclose(psi, [np.sqrt(0.5), 0, 0, np.sqrt(0.5), 0, 0, 0, 0], atol=1e-15)


@pytest.mark.parametrize("kind,params", [("NOPE", ()), ("RX", ()), ("RX", (float("inf"),)), ("U3", (0.1,))])
def test_what_was_refused_in_python_still_is(qs, kind, params):
    with qs.Simulator(3, precision="c128") as sim:
        with pytest.raises((ValueError, TypeError)):
            sim.run([cg.op("H", (0,)), cg.op(kind, (1,), (), params)])
        assert sim.stats()["gates"] == 1


@pytest.mark.parametrize("terms", [3, 5])
@pytest.mark.parametrize("kmax", [4, 5, 6])
def test_blocks_of_every_gate_kind(qs, oracle_mod, kmax, terms):
    """One block's wires at a time: low (quad fragments), high and spread."""
    n = 14
    ops = []
    for w in ((0, 1, 2, 3, 4, 5), (8, 9, 10, 11, 12, 13), (0, 3, 6, 8, 11, 13)):
        ops += [o for o in mixed_ops(n, 39, seed=sum(w) + kmax, wires=w[:kmax]) if len(o.targets) + len(o.controls) <= kmax]
    psi = cg.random_state(n, seed=2)
    ref = oracle_mod.OracleSim(n, psi=psi)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision="c64", fusion="greedy", kmax=kmax, tc_terms=terms) as sim:
        sim.set_amplitudes(psi)
        sim.set_profiling(True)
        sim.run(ops)
        got = sim.get_amplitudes()
        kt = sim.kernel_times()
    assert sum(kt.get(c, {}).get("launches", 0) for c in ("block_tc", "block_tc6")) >= 3, kt
    # 2^-17 per element and pass, at random, over some ten passes: 1e-9
    assert infidelity(ref.psi, got) <= 1e-8


def test_more_gates_than_the_blocks_matrix(qs, oracle_mod):
    """A block of 5-qubit gates (16 KB each) whose record is its matrix."""
    n = 13
    w = (1, 4, 6, 9, 12, 2)
    ops = [cg.op("MAT", [w[(i + j) % 6] for j in range(5)], (), (cg.random_unitary(32, i),)) for i in range(9)]
    ref = oracle_mod.OracleSim(n)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision="c64", fusion="greedy") as sim:
        sim.run(ops)
        got = sim.get_amplitudes()
        assert sim.stats()["passes"] == 1
    assert infidelity(ref.psi, got) <= 1e-8


@pytest.mark.parametrize("n,depth", [(13, 60), (18, 60)])
def test_more_blocks_than_one_launch_builds(qs, oracle_mod, n, depth):
    ops = cg.random_u3_brickwork(n, depth, seed=n)
    ref = oracle_mod.OracleSim(n)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision="c64", fusion="greedy") as sim:
        sim.run(ops)
        got = sim.get_amplitudes()
        assert sim.stats()["passes"] > 32
    assert infidelity(ref.psi, got) <= 1e-7
