"""Draws against the oracle, bit for bit, where the running sums are hard: exact
ties in every addition, sums that stay zero or cross binades, equal
probabilities, one block and many, few draws for the blocks and more than two
per block."""
import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_state, rng
from oracle import sim

pytestmark = pytest.mark.gpu


def amplitudes(kind, n):
    N = 1 << n
    if kind == "random":
        return random_state(n, 7 * n)
    if kind == "uniform":
        return np.full(N, 2.0 ** (-n / 2) if n % 2 == 0 else np.sqrt(0.5) * 2.0 ** (-(n - 1) / 2), dtype=complex)
    if kind == "last":       # the sums stay zero, then one
        psi = np.zeros(N, dtype=complex)
        psi[N - 3] = 1.0
        return psi
    # p odd multiples of 2^-54 on top of a sum of 1/2 and more: half-way in every addition
    k = (rng(n).integers(1, int(2 ** (27 - n / 2)), N) | 1).astype(float)
    psi = (k * 2.0 ** -27).astype(complex)
    psi[0] = np.sqrt(0.5) + 2.0 ** -20
    return psi


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("kind", ["random", "uniform", "last", "ties"])
@pytest.mark.parametrize("n,m", [(9, 5000), (10, 1), (10, 5000), (11, 33), (15, 40), (15, 5000), (20, 300), (21, 9000)])
def test_draws_bit_exact(dtype, kind, n, m):
    psi = amplitudes(kind, n)
    if dtype == qs.QS_C64:
        psi = psi.astype(np.complex64).astype(np.complex128)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        got = qs.qs_sample(h, 17 + n, m)
        both, _ = qs.qs_sample_stats(h, 17 + n, m)
    finally:
        qs.qs_free(h)
    assert np.array_equal(got, sim.sample(psi, 17 + n, m))
    assert np.array_equal(both, got)
