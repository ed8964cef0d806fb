"""Runs of diagonal blocks in one pass and their device-built tables: 1 to 6
blocks in a row (one pass takes up to 4; 3 in complex128), tables of 1 to 12
qubits on low and high qubits, multi-target diagonal matrices with controls,
tables whose gates outgrow a record, against the oracle."""
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


def phases(n, groups, seed):
    """H on one qubit, then controlled phases between the first group and
    each of the others (a block per pair of groups)."""
    r = np.random.default_rng(seed)
    ops = [cg.op("H", (groups[0][0],))]
    for g in groups[1:]:
        ops += [cg.op("R", (a,), (b,), (float(r.uniform(0, 6)),)) for a in groups[0] for b in g]
    return ops


@pytest.mark.parametrize("prec,df", [("c64", False), ("c128", False), ("c128", True)])
@pytest.mark.parametrize("count", [1, 2, 3, 4, 5, 6])
def test_runs_of_blocks(qs, oracle_mod, prec, df, count):
    n, w = 18, 6 if count < 3 else 5
    first = list(range(n - w, n))
    rest = list(range(n - w))
    groups = [first] + [rest[i::count] for i in range(count)]
    ops = phases(n, groups, count) + [cg.op("H", (0,))] + phases(n, groups[::-1], count + 9)
    psi = cg.random_state(n, seed=count)
    ref = oracle_mod.OracleSim(n, psi=psi)
    oracle_mod.run_ops(ref, ops)
    out = []
    for profiling in (0, 1, 2):
        with qs.Simulator(n, precision=prec, fusion="greedy", c128_df=df) as sim:
            sim.set_amplitudes(psi)
            sim.set_profiling(profiling)
            sim.reset_stats()
            sim.run(ops)
            out.append((sim.get_amplitudes(), sim.stats()["passes"], sim.kernel_times()))
    # item by item and in runs: the same products in the same order
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][0], out[2][0])
    assert out[0][1] == out[1][1] <= out[2][1]
    assert out[1][2]["block_diag"]["launches"] >= 1
    if prec == "c64":
        assert infidelity(ref.psi, out[0][0]) <= 1e-8
    else:
        assert np.max(np.abs(out[0][0] - ref.psi)) <= (1e-13 if df else 1e-14)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [2, 5, 9, 10, 13])
def test_all_kinds_of_diagonal_gates(qs, oracle_mod, prec, n):
    r = np.random.default_rng(n)
    ops = []
    for i in range(60):
        t = int(r.integers(1, min(n, 4) + 1))
        q = [int(v) for v in r.permutation(n)[:min(n, t + int(r.integers(0, 3)))]]
        ops.append(cg.op("MAT", q[:t], q[t:], (np.diag(np.exp(1j * r.uniform(0, 6, 1 << t))),)))
    psi = cg.random_state(n, seed=n)
    ref = oracle_mod.OracleSim(n, psi=psi)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision=prec, fusion="greedy") as sim:
        sim.set_amplitudes(psi)
        sim.run(ops)
        got = sim.get_amplitudes()
    # each gate and each table rounds a few times
    assert np.max(np.abs(got - ref.psi)) <= 240 * (2.0 ** -24 if prec == "c64" else 2.0 ** -53)


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_more_gates_than_a_record_holds(qs, oracle_mod, prec):
    n = 14
    r = np.random.default_rng(8)
    ops = [cg.op("R", (int(a),), (int(b),), (float(r.uniform(0, 6)),)) for a, b in
           (r.permutation(11)[:2] for _ in range(2000))]
    psi = cg.random_state(n, seed=1)
    ref = oracle_mod.OracleSim(n, psi=psi)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision=prec, fusion="greedy") as sim:
        sim.set_amplitudes(psi)
        sim.run(ops)
        got = sim.get_amplitudes()
        assert sim.stats()["passes"] == 1
    assert np.max(np.abs(got - ref.psi)) <= (1e-6 if prec == "c64" else 1e-12)
