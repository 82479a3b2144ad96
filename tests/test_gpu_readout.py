"""Results read out: amplitudes by index (more and fewer indices than one launch
takes, none, one out of range, qubits moved to other bits) and complex128
probabilities over the whole range of doubles."""
import time

import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_state, rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("count", [0, 1, 4, 5, 31, 480, 481, 65536, 65536 + 481])
def test_gather(dtype, count):
    n = 12
    psi = random_state(n, 3).astype(np.complex64).astype(np.complex128)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        idx = rng(count).integers(0, 1 << n, count)
        for _ in range(2):   # before and after the state has its scratch
            assert np.array_equal(qs.qs_get_amplitudes_at(h, idx), psi[idx])
            qs.qs_norm(h)
        with pytest.raises(qs.QSError):
            qs.qs_get_amplitudes_at(h, np.append(idx, 1 << n))
    finally:
        qs.qs_free(h)


def test_one_index_costs_less_than_a_gather():
    """One amplitude is one copy; a launch and a copy took 1.4 times as long."""
    h = qs.qs_alloc(12, qs.QS_C128)
    try:
        qs.qs_init_uniform(h)
        qs.qs_norm(h)
        best = []
        for count in (1, 8):
            idx, took = np.arange(count), []
            for _ in range(200):
                t = time.perf_counter()
                qs.qs_get_amplitudes_at(h, idx)
                took.append(time.perf_counter() - t)
            best.append(np.median(took))
    finally:
        qs.qs_free(h)
    assert best[0] <= 0.85 * best[1]


def test_gather_after_remapped_circuit():
    n, gates = qs.qs_supremacy_circuit(3, 4, 8, 5)
    sched = qs.qs_schedule_build(n, gates)
    loc = np.arange(n)
    loc[[0, n - 1]] = loc[[n - 1, 0]]
    qs.qs_schedule_remap(sched, loc)
    h = qs.qs_alloc(n, qs.QS_C128)
    try:
        qs.qs_init_basis(h, 0)
        qs.qs_run_circuit(h, sched)
        got = qs.qs_get_amplitudes_at(h, np.arange(1 << n))   # the qubits still moved
        assert np.array_equal(got, qs.qs_get_amplitudes(h))
    finally:
        qs.qs_free(h)
        qs.qs_schedule_free(sched)


@pytest.mark.parametrize("n", [1, 2, 9, 13])
def test_c128_probabilities_over_every_exponent(n):
    """The squares are built from integers and rounded as FP64 products: bit for
    bit numpy's, with ties, subnormals, overflow, signed zeros and infinities."""
    g = np.random.default_rng(11 + n)
    bits = g.integers(0, 1 << 64, size=2 << n, dtype=np.uint64)
    bits[1::3] &= ~np.uint64((1 << 26) - 1)          # exact ties of the 53-bit result among them
    bits[(bits >> np.uint64(52) & np.uint64(0x7FF)) == 0x7FF] &= np.uint64(0x800FFFFFFFFFFFFF)
    special = np.array([0.0, -0.0, 5e-324, -1.0, 1.0, np.inf, 2.0 ** -511, 2.0 ** -512, 2.0 ** 511.5,
                        1.7976931348623157e308, 1.0 + 2.0 ** -52, 1.5 + 2.0 ** -27])[:2 << n]
    bits[:special.size] = special.view(np.uint64)
    f = bits.view(np.float64)
    with np.errstate(over="ignore", under="ignore"):
        want = f[0::2] * f[0::2] + f[1::2] * f[1::2]
    h = qs.qs_alloc(n, qs.QS_C128)
    try:
        qs.qs_set_amplitudes(h, f.view(np.complex128))
        got = qs.qs_probabilities(h)
    finally:
        qs.qs_free(h)
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))


@pytest.mark.parametrize("n", [2, 9, 13])
def test_c64_probabilities_over_every_exponent(n):
    """Pairs of any two exponents (zeros, subnormals, infinities and NaN among them),
    with full, short and single-bit significands: p = x^2 + y^2 rounded once."""
    g, N = rng(n), 1 << n
    bits = g.integers(0, 1 << 32, (N, 2), dtype=np.uint64).astype(np.uint32)
    near = g.random(N) < 0.6      # exponents within 30 of one another: every shift of the smaller square
    e = (bits[:, 0] >> 23) & 255
    other = np.clip(e.astype(int) + g.integers(-30, 31, N), 0, 255).astype(np.uint32)
    bits[near, 1] = (bits[near, 1] & 0x807FFFFF) | (other[near] << 23)
    for keep, mask in ((0.2, 0xFFFFF000), (0.2, 0xFF800001), (0.1, 0xFF800000)):
        bits[g.random(N) < keep] &= np.uint32(mask)
    bits[g.random((N, 2)) < 0.05] = 0
    with np.errstate(all="ignore"):
        psi = bits.view(np.float32).astype(np.float64).view(np.complex128).ravel()
        want = psi.real ** 2 + psi.imag ** 2
    h = qs.qs_alloc(n, qs.QS_C64)
    try:
        qs.qs_set_amplitudes(h, psi)
        assert np.array_equal(qs.qs_probabilities(h), want, equal_nan=True)
    finally:
        qs.qs_free(h)
