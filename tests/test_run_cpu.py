"""How Simulator.run hands ops to the library, with a recorder in its place (no
GPU): every op as apply_op would queue it, in order, whatever type carries it."""
from collections import namedtuple
from types import SimpleNamespace

import numpy as np
import pytest

import circuitgen as cg
from paper_1612_08091_gb300 import gates, qsim

KINDS = ["H", "X", "Y", "Z", "S", "T", "SWAP", "RX", "RY", "RZ", "R", "U3"]


class Lib:
    """Records (kind or matrix, targets, controls, params) of what is queued."""

    def __init__(self):
        self.queue = []

    def sim_apply_gates(self, h, count, kinds, nt, nc, targets, controls, params, queued):
        it = ic = ip = 0
        for i in range(count):
            k = KINDS[kinds[i]]
            n = 3 if k == "U3" else int(k in ("RX", "RY", "RZ", "R"))
            self.queue.append((k, [targets[it + j] for j in range(nt[i])], [controls[ic + j] for j in range(nc[i])],
                               [params[ip + j] for j in range(n)]))
            it, ic, ip = it + nt[i], ic + nc[i], ip + n
        return 0

    def sim_apply(self, h, m, t, nt, c, nc):
        self.queue.append((np.array([m[i] for i in range(2 * 4 ** nt)]), [t[j] for j in range(nt)],
                           [c[j] for j in range(nc)], None))
        return 0


def simulator():
    sim = object.__new__(qsim.Simulator)
    sim.lib, sim.h = Lib(), None
    return sim


def check(queue, ops):
    """Each queued gate is the op's, with its matrix."""
    assert len(queue) == len(ops)
    for (k, t, c, p), op in zip(queue, ops):
        assert t == [int(v) for v in op.targets] and c == [int(v) for v in op.controls]
        want = gates.gate_matrix(op.kind, op.params).astype(complex)
        got = gates.gate_matrix(k, p) if isinstance(k, str) else k.view(complex).reshape(want.shape)
        np.testing.assert_array_equal(got, want)


OPS = [cg.op("H", (0,)), cg.op("X", (1,), (0, 2)), cg.op("RY", (2,), (), (0.3,)), cg.op("SWAP", (0, 3)),
       cg.op("U3", (1,), (3,), (0.1, 0.2, 0.3)), cg.op("R", (3,), (1,), (-2,))]


def test_lists_and_tuples():
    for ops in (OPS, tuple(OPS), []):
        sim = simulator()
        sim.run(ops)
        check(sim.lib.queue, list(ops))


def test_fields_are_read_by_name():
    Other = namedtuple("Other", "kind controls targets params")
    for make in (lambda o: Other(o.kind, o.controls, o.targets, o.params),
                 lambda o: SimpleNamespace(kind=o.kind, targets=list(o.targets), controls=list(o.controls),
                                           params=list(o.params))):
        # one control and one target each: nothing but the names tells them apart
        for plain in (OPS, [cg.op("X", (1,), (2,)), cg.op("U3", (3,), (0,), (0.1, 0.2, 0.3))]):
            ops = [make(o) for o in plain]
            sim = simulator()
            sim.run(ops)
            check(sim.lib.queue, ops)


def test_an_iterator_sees_its_ops_queued():
    """A generator that reads the handle between its ops, as a measured loop does."""
    sim = simulator()
    seen = []

    def ops():
        for i, o in enumerate(OPS):
            seen.append(len(sim.lib.queue) == i)
            yield o

    sim.run(ops())
    assert all(seen)
    check(sim.lib.queue, OPS)


@pytest.mark.parametrize("bad", [SimpleNamespace(kind=["H"], targets=(0,), controls=(), params=()),
                                 SimpleNamespace(kind="NOPE", targets=(0,), controls=(), params=()),
                                 SimpleNamespace(targets=(0,)), None,
                                 SimpleNamespace(kind="RY", targets=(0,), controls=(), params=("a",)),
                                 SimpleNamespace(kind="RY", targets=(0,), controls=(), params=())])
def test_refused_at_its_place(bad):
    sim = simulator()
    with pytest.raises(Exception):
        sim.run(OPS + [bad] + OPS)
    check(sim.lib.queue, OPS)


@pytest.mark.parametrize("odd", [
    cg.op("H", (0,), (), (0.5,)), cg.op("RX", (1,), (), (np.float32(0.3),)), cg.op("RZ", np.array([2]), (), (True,)),
    cg.op("MAT", (0,), (), (np.eye(2),)), cg.op("U3", (1,), (), tuple(np.float32([0.3, 0.7, 0.1])))])
def test_what_apply_op_takes_is_taken(odd):
    """Parameters that a kind ignores, and numbers of other types, as apply_op has them."""
    ops = [OPS[0], odd, OPS[1]]
    sim = simulator()
    sim.run(ops)
    check(sim.lib.queue, ops)
