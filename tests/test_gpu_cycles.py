"""The cycle walk on registers whose lowest qubit lies inside a slice: pieces
of 64 bytes to 4 KB, with controls between, against numpy (amplitudes only
move: exact), and the tiled kernel just below."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1612_08091_gb300 as q

    q.load()
    return q


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("qubits,controls", [
    ((3, 4, 5, 6), ()), ((3, 9, 5, 12, 17), (8,)), ((4, 6, 7, 10, 13), ()), ((8, 7), (3, 19)), ((9, 10, 18), ()),
    ((18, 5, 9), (6, 7)), ((2, 5, 8, 11), ()), ((3,), (2, 10)), ((5, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16), ()),
])
@pytest.mark.parametrize("kind", ["random", "one_cycle", "fixed_points"])
def test_walks_inside_a_slice(qs, prec, qubits, controls, kind):
    n, m = 20, len(qubits)
    rng = np.random.default_rng(sum(qubits) + m)
    D = 1 << m
    perm = np.arange(D)
    if kind == "random":
        perm = rng.permutation(D)
    elif kind == "one_cycle":
        perm = (perm + 1) % D
    else:
        moved = rng.choice(D, min(D, 3), replace=False)
        perm[moved] = moved[np.roll(np.arange(len(moved)), 1)]
    psi = cg.random_state(n, seed=1).astype(np.complex64 if prec == "c64" else np.complex128)
    i = np.arange(1 << n)
    v = np.zeros_like(i)
    for j, b in enumerate(qubits):
        v |= ((i >> b) & 1) << j
    w, to = perm[v], i.copy()
    for j, b in enumerate(qubits):
        to = (to & ~(1 << b)) | (((w >> j) & 1) << b)
    for c in controls:
        to = np.where((i >> c) & 1, to, i)
    want = np.empty_like(psi)
    want[to] = psi
    with qs.Simulator(n, precision=prec) as sim:
        sim.set_amplitudes(psi.astype(np.complex128))
        sim.apply_permutation(perm, qubits, controls)
        got = sim.get_amplitudes()
    np.testing.assert_array_equal(got, want.astype(np.complex128))
