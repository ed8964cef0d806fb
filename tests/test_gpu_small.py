"""Gate by gate on small registers: the whole queue in one launch against one
launch per gate (profiling on), the same bits; one CTA and the cluster, gates
on and across the rank qubits, several launches' worth of gates, the largest
register of each precision and the first beyond it, and registers whose
one-qubit kernels take narrow blocks."""
import numpy as np
import pytest

import circuitgen as cg
from test_gpu_queue import mixed_ops

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1612_08091_gb300 as q

    q.load()
    return q


@pytest.mark.parametrize("prec,n,count", [
    ("c128", 1, 8), ("c128", 2, 60), ("c128", 8, 80), ("c128", 9, 80), ("c128", 12, 900), ("c128", 13, 80),
    ("c128", 14, 40), ("c64", 3, 60), ("c64", 9, 80), ("c64", 16, 80), ("c64", 17, 40),
])
def test_one_launch_equals_one_per_gate(qs, oracle_mod, prec, n, count):
    ops = [o for o in mixed_ops(n, count, seed=n) if len(o.targets) + len(o.controls) <= n]
    assert n == 1 or len(ops) >= 3
    psi = cg.random_state(n, seed=3)
    ref = oracle_mod.OracleSim(n, psi=psi)
    oracle_mod.run_ops(ref, ops)
    out = []
    for profiling in (False, True):
        with qs.Simulator(n, precision=prec) as sim:
            sim.set_amplitudes(psi)
            sim.set_profiling(profiling)
            sim.reset_stats()
            sim.run(ops)
            out.append(sim.get_amplitudes())
            st = sim.stats()
        assert st["passes"] == len(ops)
    np.testing.assert_array_equal(out[0], out[1])
    # each gate rounds each amplitude a few times
    eps = 2.0 ** -53 if prec == "c128" else 2.0 ** -24
    assert np.max(np.abs(out[0] - ref.psi)) <= 16 * eps * len(ops)


@pytest.mark.parametrize("n", [10, 13])
def test_gates_in_many_flushes(qs, oracle_mod, n):
    """Short flushes (plain launches) and longer ones (one launch) in turn."""
    ops = mixed_ops(n, 60, seed=n + 1)
    ref = oracle_mod.OracleSim(n)
    oracle_mod.run_ops(ref, ops)
    with qs.Simulator(n, precision="c128") as sim:
        i, k = 0, 1
        while i < len(ops):
            sim.run(ops[i:i + k])
            sim.flush()
            i, k = i + k, k % 7 + 1
        got = sim.get_amplitudes()
    assert np.max(np.abs(got - ref.psi)) <= 1e-12
