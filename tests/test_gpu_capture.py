"""Plain gates flushed in a stream capture: the graph replays these gates, also
after the handle has run many others."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,precision", [(7, "c128"), (11, "c128"), (11, "c64"), (15, "c128")])
def test_replay_after_other_gates(oracle_mod, n, precision):
    import torch

    import paper_1612_08091_gb300 as q

    ops, other = cg.random_u3_brickwork(n, 3, 1), cg.random_u3_brickwork(n, 20, 2)
    st = torch.cuda.Stream()
    with q.Simulator(n, precision=precision, stream=st) as sim:
        sim.reset(0)
        sim.run(ops)
        sim.flush()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sim.run(ops)
            sim.flush()
        for _ in range(100):
            sim.run(other)
            sim.flush()
        for k in range(3):
            sim.reset(k)
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            ref = oracle_mod.OracleSim(n, basis=k)
            for op in ops:
                ref.apply_op(op)
            tol = 1e-11 if precision == "c128" else 1e-4
            assert np.max(np.abs(sim.get_amplitudes() - ref.psi)) <= tol
