"""complex128 gates on 2 to 4 qubits where the handle allows double-float
accuracy: every result is within a few 2^-45 of its own products, not of the
group's largest amplitude -- amplitudes of very different sizes under matrices
that mix them, mix some of them, or none (controlled gates, permutations, gates
near the identity), sparse states, and states near the ends of the range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def unitary(d, rng):
    return np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))[0]


def near_identity(d, eps, rng):
    h = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    w, v = np.linalg.eigh(h + h.conj().T)
    return (v * np.exp(1j * eps * w)) @ v.conj().T


def matrix(kind, k, rng):
    d = 1 << k
    if kind == "mixing":
        return unitary(d, rng)
    if kind == "permutation":
        return np.eye(d)[rng.permutation(d)].astype(complex)
    if kind == "phases":
        return np.eye(d)[rng.permutation(d)] * np.where(rng.random(d) < 0.5, 1.0, np.exp(1j * rng.uniform(0, 6, d)))
    if kind == "controlled":  # the last qubit's gate where all others are 1
        m = np.eye(d, dtype=complex)
        m[d // 2 - 1::d // 2, d // 2 - 1::d // 2] = unitary(2, rng)
        return m
    if kind == "product":  # one qubit's gate beside identities
        return np.kron(np.eye(d // 2), unitary(2, rng))
    return near_identity(d, float(kind), rng)


@pytest.mark.parametrize("k", [2, 3, 4])
@pytest.mark.parametrize("kind", ["mixing", "permutation", "phases", "controlled", "product", "1e-3", "0.05", "0.3"])
@pytest.mark.parametrize("spread,zeros,scale", [(0, 0.0, 0), (8, 0.0, 0), (40, 0.0, 0), (0, 0.8, 0), (12, 0.5, 0),
                                                (10, 0.2, 900), (10, 0.2, 200), (10, 0.2, -850), (10, 0.2, -200)])
def test_rows(k, kind, spread, zeros, scale):
    import paper_1612_08091_gb300 as q

    rng = np.random.default_rng([k, spread])
    n, D = 12, 1 << k
    psi = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)) * 2.0 ** -rng.integers(0, spread + 1, 1 << n)
    psi[rng.random(1 << n) < zeros] = 0.0
    psi *= 2.0 ** scale
    U = matrix(kind, k, rng)
    for first in (0, 3, n - k):
        with q.Simulator(n, precision="c128", c128_df=True) as sim:
            sim.set_amplitudes(psi)
            sim.apply(U, tuple(range(first, first + k)))
            got = sim.get_amplitudes()
        v = psi.reshape(-1, D, 1 << first).transpose(1, 0, 2).reshape(D, -1).astype(np.clongdouble)
        g = got.reshape(-1, D, 1 << first).transpose(1, 0, 2).reshape(D, -1)
        ref = sum(U.astype(np.clongdouble)[:, c:c + 1] * v[c:c + 1] for c in range(D))
        size = sum(np.abs(U)[:, c:c + 1] * np.abs(v[c:c + 1]) for c in range(D))
        # a product in pairs: inputs cut at 2^-46 and rounded at 2^-48, three
        # roundings and a dropped term at 2^-47 of it; the sums' 2^-47: 2^-44
        tol = 2.0 ** -44 * size
        assert np.all(np.abs(g.real - ref.real) <= tol)
        assert np.all(np.abs(g.imag - ref.imag) <= tol)

