"""complex64 queues of gates on one and several qubits on the registers where
some gates are launched on their own and the others together: the same bits as
one launch per gate (profiling on)."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 8, 12, 13, 14, 15, 16])
def test_runs_equal_one_launch_per_gate(n):
    import paper_1612_08091_gb300 as q

    rng = np.random.default_rng(n)
    gates = []
    for _ in range(60):
        t = int(rng.choice([1, 1, 1, 1, 2, 3, 4, 5]))
        qs = [int(v) for v in rng.permutation(n)[:t + int(rng.integers(0, 2))]]
        d = 1 << t
        m = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))[0]
        if t == 1 and rng.random() < 0.4:
            m = [np.array([[0, 1], [1, 0]]), np.diag([1, 1j])][int(rng.integers(2))]
        gates.append((m, qs[:t], qs[t:]))
    out = []
    for profiling in (False, True):
        with q.Simulator(n, precision="c64") as sim:
            sim.set_amplitudes(cg.random_state(n, seed=3))
            sim.set_profiling(profiling)
            sim.reset_stats()
            for g in gates:
                sim.apply(*g)
            out.append(sim.get_amplitudes())
            assert sim.stats()["passes"] == len(gates)
    np.testing.assert_array_equal(out[0], out[1])
