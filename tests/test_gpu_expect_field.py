"""Transverse-field terms (X on single qubits) of a complex64 register, many
per read: edges of the tile's 13 bits, one and several passes over the high
qubits, sparse sets of qubits, repeated terms, and beside terms of other
kinds, against FP64 sums of the same amplitudes on the host."""
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


def host_x(psi, b):
    v = psi.reshape(-1, 2, 1 << b)
    return 2.0 * float(np.sum(v[:, 0].real * v[:, 1].real + v[:, 0].imag * v[:, 1].imag))


@pytest.mark.parametrize("n,qubits", [
    (12, range(12)),                      # below the tile: one read per term
    (13, range(13)), (14, range(14)),     # one tile; one high qubit
    (14, (13,)), (14, (0, 13)), (15, (13, 14)),
    (23, range(23)), (24, range(24)),     # ten and eleven high qubits: one and two high passes
    (24, (3, 12, 13, 22, 23)), (24, (14, 17, 20, 23)),
])
def test_field_terms_against_host(qs, n, qubits):
    rng = np.random.default_rng(n + len(list(qubits)))
    psi = cg.random_state(n, seed=n).astype(np.complex64)
    psi += np.float32(2.0 ** (-0.5 * n))  # no cancellation to zero
    terms = [(float(rng.uniform(-1, 1)), 1 << b, 0) for b in qubits]
    terms += terms[:2]                                        # the same qubit twice
    other = [(0.3, 0, 3), (0.2, 3, 0), (0.7, 1, 1), (-0.4, 2, 4)]  # ZZ, XX, Y, XZ
    p64 = psi.astype(np.complex128)
    norm = float(np.sum(np.abs(p64) ** 2))
    want = sum(c * host_x(p64, x.bit_length() - 1) for c, x, _ in terms)
    with qs.Simulator(n, precision="c64") as sim:
        sim.set_amplitudes(p64)
        got = sim.expect(terms)
        parts = [sim.expect([t]) for t in other]
        both = sim.expect(terms + other)
    # FP32 sums of at most 32 products, then FP64: (33 + 5) roundings of 2^-24
    # relative to the sum of the magnitudes
    tol = 38 * 2.0 ** -24 * norm
    assert abs(got - want) <= tol * sum(abs(c) for c, _, _ in terms)
    assert abs(both - (got + sum(parts))) <= tol * sum(abs(c) for c, _, _ in terms + other)
