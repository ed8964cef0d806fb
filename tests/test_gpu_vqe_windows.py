"""Window passes of the batched variational kernel against the oracle: the
smallest register above shared memory, every window position, passes that
stop at their step limit, more layers than a window reaches, no layers, and
rotations whose range reduction flips qubits or not."""
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


def oracle_energy(oracle_mod, c, h):
    ref = oracle_mod.OracleSim(c["n"])
    oracle_mod.run_ops(ref, cg.hea_ops(c["n"], c["ry"], c["rz"]))
    return ref.expect(cg.tfim_terms(c["n"], h))


@pytest.mark.parametrize("scale", [0.3, np.pi, 20.0])
def test_windows_against_oracle(qs, oracle_mod, scale):
    rng = np.random.default_rng(int(scale * 10))
    sizes = [(13, 1), (13, 9), (13, 20), (14, 1), (14, 4), (14, 19), (15, 8), (15, 17), (16, 2), (16, 7), (16, 0),
             (17, 3), (17, 8), (18, 5)]
    circuits = [{"n": n, "L": L, "ry": rng.uniform(-scale, scale, (L, n)), "rz": rng.uniform(-scale, scale, (L, n))}
                for n, L in sizes]
    h = 0.7
    with qs.Batch([c["n"] for c in circuits], [c["L"] for c in circuits], h=h) as b:
        b.set_config(256, 12)
        first = b.run(qs.hea_angles(circuits))
        again = b.run(qs.hea_angles(circuits))
    np.testing.assert_array_equal(first, again)
    for c, e in zip(circuits, first):
        # FP32 rotations: some 4 roundings per amplitude and rotation, at
        # random; the energy's scale is its number of terms
        tol = 2.0 ** -24 * 8 * np.sqrt(max(1, c["n"] * c["L"])) * (2 * c["n"])
        assert abs(e - oracle_energy(oracle_mod, c, h)) <= tol, (c["n"], c["L"])


@pytest.mark.parametrize("sizes", [
    [(17, 3)] * 100 + [(13, 2)] * 40,            # clusters of 4, then CTAs alone
    [(18, 2)] * 3 + [(14, 0), (15, 4), (9, 2)],  # clusters of 8
    [(16, 1)] * 330 + [(16, 0)],                 # a CTA per circuit
])
def test_shared_circuits_against_alone(qs, sizes):
    rng = np.random.default_rng(len(sizes))
    angles = [rng.uniform(-np.pi, np.pi, 2 * n * L) for n, L in sizes]
    with qs.Batch([n for n, _ in sizes], [L for _, L in sizes], h=0.7) as b:
        got = b.run(np.concatenate(angles))
        np.testing.assert_array_equal(got, b.run(np.concatenate(angles)))
    for i in {0, len(sizes) // 3, len(sizes) // 2, len(sizes) - 2, len(sizes) - 1}:
        n, L = sizes[i]
        with qs.Batch([n], [L], h=0.7) as b:
            alone = b.run(angles[i])[0]
        # the same FP32 sums per tile, added up in another order in FP64
        assert abs(got[i] - alone) <= 1e-12 * 2 * n, (i, n, L)
