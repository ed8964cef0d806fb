"""complex128 dense gates whose results leave the range of a double: infinity,
as FP64 arithmetic gives it, and finite results next to the end of the range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BIG = 2.0 ** 960.5  # just inside the exponents the integer form takes


def apply(matrix, amps, n, df, queue):
    import paper_1612_08091_gb300 as q

    t = int(np.log2(len(matrix)))
    with q.Simulator(n, precision="c128", c128_df=df) as sim:
        psi = np.zeros(1 << n, dtype=np.complex128)
        psi[:len(amps)] = amps
        sim.set_amplitudes(psi)
        for _ in range(queue):
            sim.apply(np.array([[1.0, 0.0], [0.0, 1.0]]), (n - 1,))
        sim.apply(matrix, tuple(range(t)))
        return sim.get_amplitudes()[:len(amps)]


@pytest.mark.parametrize("n,queue", [(10, 0), (10, 3), (15, 0)])  # one launch a gate, a queue in one launch
@pytest.mark.parametrize("e", [40, 55, 56, 60, 63])
def test_one_qubit(n, queue, e):
    got = apply(2.0 ** e * np.array([[1.0, 1.0], [1.0, -1.0]]), [BIG, BIG], n, False, queue)
    with np.errstate(over="ignore"):
        assert got[0] == np.float64(2.0 ** e * BIG) * 2  # infinity for 2^63
    assert got[1] == 0


@pytest.mark.parametrize("t", [2, 3, 4])
@pytest.mark.parametrize("e", [40, 55, 56, 60, 63.9])  # log2 of a row's sum
def test_several_qubits(t, e):
    # 1.9 2^960 times a sum of 2^63.9: beyond a double
    D = 1 << t
    had = np.array([[1.0]])
    for _ in range(t):
        had = np.kron(had, [[1.0, 1.0], [1.0, -1.0]])
    got = apply(2.0 ** e / D * had, [1.9 * 2.0 ** 960] * D, 12, True, 0)
    with np.errstate(over="ignore"):
        ref = np.float64(1.9 * 2.0 ** 960) * 2.0 ** e
    # FP32 pairs or integers: 2^-45 of the result
    assert got[0] == ref if np.isinf(ref) else abs(got[0] - ref) <= 2.0 ** -45 * ref
    scale = min(ref, 1e308)
    assert np.all(np.abs(got[1:] / scale) <= 2.0 ** -44)
