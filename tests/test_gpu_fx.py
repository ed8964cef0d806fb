"""complex128 one-qubit dense gates in shared-exponent integers: against long
double sums, for amplitudes of equal and of very different sizes, at the edge
of the matrices that take the path, and outside it (zeros, tiny and huge
amplitudes, infinities), on every target of a narrow and a wide launch."""
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


def run(qs, psi, U, t, controls=()):
    n = int(np.log2(len(psi)))
    with qs.Simulator(n, precision="c128") as sim:
        sim.set_amplitudes(psi)
        sim.apply(U, (t,), controls)
        return sim.get_amplitudes()


def want(psi, U, t):
    """U on qubit t in extended precision, with FP64's error bound of each result."""
    L = np.clongdouble
    v = psi.astype(L).reshape(-1, 2, 1 << t)
    out = np.empty_like(v)
    size = np.empty(v.shape, dtype=np.longdouble)
    for r in (0, 1):
        out[:, r] = L(U[r][0]) * v[:, 0] + L(U[r][1]) * v[:, 1]
        size[:, r] = abs(U[r][0]) * np.abs(v[:, 0]) + abs(U[r][1]) * np.abs(v[:, 1])
    return out.reshape(-1), size.reshape(-1)


def u3(th, ph, la):
    c, s = np.cos(th / 2), np.sin(th / 2)
    return np.array([[c, -np.exp(1j * la) * s], [np.exp(1j * ph) * s, np.exp(1j * (ph + la)) * c]])


@pytest.mark.parametrize("spread", [0, 8, 60, 400])
@pytest.mark.parametrize("theta", [1.1, 0.1252, 0.12, 2 * np.pi - 0.1255, np.pi - 0.1251,
                                   0.0626, 0.06, 2 * np.pi - 0.0627])
def test_error_is_that_of_fp64(qs, spread, theta):
    # sin(0.1252 / 2) is just above 2^-4 of cos, 0.12 below (FP64 path)
    n = 15  # two amplitudes a thread; larger registers use the same arithmetic
    r = np.random.default_rng(spread)
    psi = (r.standard_normal(1 << n) + 1j * r.standard_normal(1 << n)) * 2.0 ** -r.integers(0, spread + 1, 1 << n)
    U = u3(theta, 0.7, 2.1)
    for t in (0, 1, 7, n - 1):
        ref, size = want(psi, U, t)
        got = run(qs, psi, U, t)
        # complex FP64: at most four roundings of terms no larger than `size`
        assert np.all(np.abs(got - ref) <= 4 * 2.0 ** -53 * size)


@pytest.mark.parametrize("n", [14, 19, 21])
@pytest.mark.parametrize("controls", [(), (2,)])
def test_narrow_and_wide_launches(qs, oracle_mod, n, controls):
    psi = cg.random_state(n, seed=n)
    U = u3(0.9, 1.2, 0.4)
    for t in (0, 5, n - 1):
        ref = oracle_mod.OracleSim(n, psi=psi)
        ref.apply(U, (t,), controls)
        got = run(qs, psi, U, t, controls)
        assert np.max(np.abs(got - ref.psi)) <= 8 * 2.0 ** -53 * np.max(np.abs(psi))


@pytest.mark.parametrize("n", [11, 15])
def test_values_outside_the_range(qs, n):
    psi = np.zeros(1 << n, dtype=np.complex128)
    h = 1 << (n - 1)
    psi[0], psi[h] = 1e-300, 3e-300j
    psi[1], psi[h + 1] = 1e300, -2e299
    psi[2], psi[h + 2] = 5e-324, 0
    psi[3], psi[h + 3] = 0, 0
    psi[4], psi[h + 4] = 1.0, 5e-324
    for U in (u3(1.0, 0.3, 0.2), 3e5 * u3(1.0, 0.3, 0.2), np.array([[2.0, 1.0], [1.0, -7.0]])):
        ref, size = want(psi, U, n - 1)
        got = run(qs, psi, U, n - 1)
        assert np.all(np.abs(got - ref) <= 4 * 2.0 ** -53 * size + 1e-323)
        assert np.all(got[[3, h + 3]] == 0)


def test_infinities_stay(qs):
    import torch

    n = 15
    with qs.Simulator(n, precision="c128") as sim:
        class A:
            pass

        a = A()
        a.__cuda_array_interface__ = {"shape": (1 << n,), "typestr": "<c16", "data": (sim.state_ptr(), False),
                                      "version": 3, "strides": None}
        view = torch.as_tensor(a, device="cuda")
        view.fill_(0.5)
        view[3] = complex(float("inf"), 0.0)
        view[9] = complex(float("nan"), 0.0)
        sim.apply(np.array([[1.0, 1.0], [1.0, -1.0]]), (2,))
        got = sim.get_amplitudes()
    for i in (3, 7):
        assert not np.isfinite(got[i].real)
    for i in (9, 13):
        assert np.isnan(got[i].real)
    rest = np.delete(np.arange(1 << n), [3, 7, 9, 13])
    assert np.all(np.isfinite(got[rest]))
