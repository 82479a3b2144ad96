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


def below_a_power_of_two(kind, n, dtype):
    """Amplitudes whose p lie below a power of two by a relative 2^-33 or less.  Equal
    ones: "root" 1 / sqrt(2^n) as rounded, "turned" (x + i y) 2^-(n/2), x^2 + y^2 just
    below 1.  "mixed": every other p is 2^-j (1 - d), j and d at random, so that some
    p is just below 20 binades under the sum wherever the sum stands."""
    g, N = rng(n), 1 << n
    if kind == "root":
        a = 1 / np.sqrt(2.0 ** n) if n % 2 else (1 + 1j) / np.sqrt(2.0 ** (n + 1))
        return np.full(N, a, dtype=complex)
    if kind == "turned":
        real = np.float32 if dtype == qs.QS_C64 else np.float64
        x = g.uniform(0.2, 0.8, 1 << 16).astype(real)
        y = np.sqrt(1 - x.astype(float) ** 2).astype(real).astype(float)
        p = x.astype(float) ** 2 + y ** 2
        i = np.flatnonzero((p < 1) & (p > 1 - 2.0 ** -34))[0]
        return np.full(N, (x[i] + 1j * y[i]) * 2.0 ** (-n / 2))
    p, at = g.exponential(size=N), np.arange(0, N, 2)
    near = 2.0 ** -g.integers(n, n + 9, at.size) * (1 - 2.0 ** -g.uniform(30, 52, at.size))
    p[at] = 0
    p *= (1 - near.sum()) / p.sum()
    p[at] = near
    return np.sqrt(p).astype(complex)


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("kind,n,m", [("root", 21, 300), ("root", 21, 9000), ("root", 22, 5000), ("root", 23, 100000),
                                      ("root", 25, 5000), ("root", 25, 70000), ("turned", 22, 300), ("turned", 22, 20000),
                                      ("mixed", 14, 500), ("mixed", 16, 60), ("mixed", 18, 5000), ("mixed", 21, 3000)])
def test_draws_below_a_power_of_two(dtype, kind, n, m):
    """The largest terms of a running sum's integer form: 2^32 units after rounding."""
    psi = below_a_power_of_two(kind, n, dtype)
    if dtype == qs.QS_C64:
        psi = psi.astype(np.complex64).astype(np.complex128)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        got = qs.qs_sample(h, 5 + n, m)
    finally:
        qs.qs_free(h)
    assert np.array_equal(got, sim.sample(psi, 5 + n, m))
