"""Rounding of the transverse-field terms of a complex64 register, many per
read: no further from FP64 than the same terms read one by one (k_expect_x),
on random states and on product states of tilted spins, whose pairs all have
the same sign, with coefficients that FP32 holds and that it does not."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu


def state(n, kind, seed):
    if kind == "random":
        return cg.random_state(n, seed=seed).astype(np.complex64)
    psi = np.ones(1)
    for t in np.random.default_rng(seed).uniform(0.2, 0.8, n):
        psi = np.kron([np.cos(t / 2), np.sin(t / 2)], psi)
    return psi.astype(np.complex64)


def x_sums(psi):
    out = []
    for b in range(int(np.log2(len(psi)))):
        v = psi.reshape(-1, 2, 1 << b)
        out.append(2.0 * float(np.sum(v[:, 0].real * v[:, 1].real + v[:, 0].imag * v[:, 1].imag)))
    return np.array(out)


# 13: one tile; 16: fewer pairs than threads of the one-by-one read; 21, 22: the
# last register whose pairs go to FP64 one by one and the first where eight go together
@pytest.mark.parametrize("n,seeds", [(13, 8), (16, 6), (21, 4), (22, 4)])
@pytest.mark.parametrize("kind", ["random", "tilted"])
@pytest.mark.parametrize("c", [1.0, 0.7])
def test_no_further_from_fp64_than_term_by_term(n, seeds, kind, c):
    import paper_1612_08091_gb300 as q

    field, one = [], []
    with q.Simulator(n, precision="c64") as sim:
        for seed in range(seeds):
            psi = state(n, kind, seed).astype(np.complex128)
            sim.set_amplitudes(psi)
            ref = x_sums(psi)
            single = [sim.expect([(1.0, 1 << b, 0)]) for b in range(n)]
            for b in range(0, n - 1, 2):
                field.append(sim.expect([(c, 1 << b, 0), (c, 2 << b, 0)]) - c * (ref[b] + ref[b + 1]))
                one.append(c * (single[b] + single[b + 1] - ref[b] - ref[b + 1]))
    # sums of at most eight pairs either way, in a tree here and in a chain there:
    # the errors' standard deviations are at most equal.  Each is known from at
    # least 40 samples, to 1 / sqrt(2 * 40) = 0.11 of itself, so their ratio stays
    # below 1 + 3 * 0.16 at three deviations
    assert len(field) >= 40
    assert np.sqrt(np.mean(np.square(field))) <= 1.5 * np.sqrt(np.mean(np.square(one)))


@pytest.mark.parametrize("n", [13, 22])
def test_coefficients_outside_fp32(n):
    import paper_1612_08091_gb300 as q

    psi = state(n, "tilted", 3).astype(np.complex128)
    x = x_sums(psi)
    with q.Simulator(n, precision="c64") as sim:
        sim.set_amplitudes(psi)
        # a pair of FP32 spans 2^-100 .. 2^100 of these; FP32 itself ends at 2^128
        for c in (2.0 ** 120, 2.0 ** 90, 2.0 ** -90, 2.0 ** -120):
            assert abs(sim.expect([(c, 1, 0), (c, 2, 0), (c, 4, 0)]) / c - x[:3].sum()) <= 2.0 ** -20 * n
        # cancelling coefficients leave the others alone
        got = sim.expect([(0.5, 1, 0), (-0.5, 1, 0), (0.25, 2, 0), (0.25, 4, 0)])
        assert abs(got - 0.25 * (x[1] + x[2])) <= 2.0 ** -20 * n
