"""complex128 dense gates whose elements are each real or imaginary: the real
and imaginary parts of a result are as exact, each against the components it
comes from, as in FP64 arithmetic, and zeros stay zeros, for components of very
different sizes, one launch a gate and a queue in one launch (both on qubits
of one CTA and across CTAs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

R = np.sqrt(0.5)
GATES = {
    "H": np.array([[R, R], [R, -R]], dtype=complex),
    "RY": np.array([[np.cos(0.4), -np.sin(0.4)], [np.sin(0.4), np.cos(0.4)]], dtype=complex),
    "RX": np.array([[np.cos(0.4), -1j * np.sin(0.4)], [-1j * np.sin(0.4), np.cos(0.4)]]),
    "SH": np.array([[R, R], [1j * R, -1j * R]]),
    "HS": np.array([[R, 1j * R], [R, -1j * R]]),
    "XRX": np.array([[-1j * np.sin(0.4), np.cos(0.4)], [np.cos(0.4), -1j * np.sin(0.4)]]),
    "odd": np.array([[0.6, 0.8], [0.8, 0.6j]]),  # rows that mix the components differently
}


def part(z, i):
    """0 real, 1 imaginary, as extended floats"""
    return (z.real, z.imag)[i].astype(np.longdouble)


def want(psi, U, t):
    """U on qubit t by components, and the sum of the magnitudes of each component's terms"""
    v = psi.reshape(-1, 2, 1 << t)
    out = np.zeros(v.shape + (2,), dtype=np.longdouble)
    size = np.zeros_like(out)
    for r in (0, 1):
        for c in (0, 1):
            imag = U[r, c].real == 0.0
            m = np.longdouble(U[r, c].imag if imag else U[r, c].real)
            for i in (0, 1):
                term = m * part(v[:, c], i ^ imag) * (-1 if imag and i == 0 else 1)
                out[:, r, :, i] += term
                size[:, r, :, i] += abs(term)
    return out.reshape(-1, 2), size.reshape(-1, 2)


def run(psi, U, t, queued):
    import paper_1612_08091_gb300 as q

    n = int(np.log2(len(psi)))
    with q.Simulator(n, precision="c128") as sim:
        sim.set_amplitudes(psi)
        for _ in range(queued):
            sim.apply(np.eye(2), (0,))
        sim.apply(U, (t,))
        return sim.get_amplitudes()


@pytest.mark.parametrize("n,queued", [(7, 3), (11, 3), (11, 0), (15, 0), (19, 0)])
@pytest.mark.parametrize("name", sorted(GATES))
def test_parts_are_those_of_fp64(n, queued, name):
    r = np.random.default_rng(n)
    N = 1 << n
    comp = r.standard_normal((N, 2)) * 2.0 ** -r.integers(0, 120, (N, 2))
    comp[r.random((N, 2)) < 0.2] = 0.0
    comp[r.random((N, 2)) < 0.1] = -0.0
    psi = comp[:, 0] + 1j * comp[:, 1]
    psi.real, psi.imag = comp[:, 0], comp[:, 1]
    for t in (0, 4, n - 1):
        ref, size = want(psi, GATES[name], t)
        got = run(psi, GATES[name], t, queued)
        for i in (0, 1):
            # FP64: two products and a sum, three roundings of at most 2^-53 of the terms
            assert np.all(abs(part(got, i) - ref[:, i]) <= 3 * 2.0 ** -53 * size[:, i])


@pytest.mark.parametrize("n", [7, 11, 15])
def test_real_states_stay_real(n):
    import paper_1612_08091_gb300 as q

    r = np.random.default_rng(3)
    psi = r.standard_normal(1 << n).astype(complex)
    psi.imag[::3] = -0.0
    with q.Simulator(n, precision="c128") as sim:
        sim.set_amplitudes(psi)
        for k in range(4):
            sim.apply(GATES["H"], (k % n,))
            sim.apply(np.diag([1.0, -1.0]), (k % n,))
            sim.apply(GATES["RY"], (n - 1,))
        assert np.all(sim.get_amplitudes().imag == 0.0)
