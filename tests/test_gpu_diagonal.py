"""Diagonal sweeps at the edges of their tiling: states below a row, one row,
several rows per chunk, chunks of 32 rows; odd coefficients on the lanes' bits,
above them, on both and nowhere."""
import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_diag, random_phase_poly, random_qubits, random_state
from oracle import sim

pytestmark = pytest.mark.gpu

EPS = {qs.QS_C128: 2.0 ** -53, qs.QS_C64: 2.0 ** -24}


def rounded(psi, dtype):
    return psi.astype(np.complex64).astype(np.complex128) if dtype == qs.QS_C64 else psi


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("odd", ["none", "lanes", "above", "both"])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 10, 14, 19, 20, 23])
def test_phase_rows_and_chunks(dtype, odd, n):
    coeff, edges = random_phase_poly(n, 2 * n if n > 1 else 0, 31 * n)
    coeff = np.asarray(coeff) // 2 * 2
    if odd in ("lanes", "both"):
        coeff[min(2, n - 1)] += 1
        coeff[0] += 1
    if odd in ("above", "both"):
        coeff[n - 1] += 1
        coeff[n // 2] += 1
    psi = rounded(random_state(n, n), dtype)
    ref = psi.copy()
    sim.apply_phase(ref, coeff, edges)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        qs.qs_apply_phase(h, coeff, edges)
        out = qs.qs_get_amplitudes(h)
    finally:
        qs.qs_free(h)
    # an odd factor: one rounded sum and one rounded product per component, and
    # the rounding of sqrt(1/2); even ones are exact
    bound = 8 * EPS[dtype] if odd != "none" else 4 * EPS[qs.QS_C128]
    assert np.all(np.abs(out - ref) <= bound * np.abs(psi))


@pytest.mark.parametrize("bits", [(8,), (9,), (8, 9), (9, 12), (10,), (6, 8)])
@pytest.mark.parametrize("n", [9, 10, 13, 18, 19, 21])
def test_phase_odd_rows(n, bits):
    """Odd coefficients on row bits, none on the lanes' bits: rows next to one another or
    two apart make a pair."""
    coeff, edges = random_phase_poly(n, n, n)
    coeff = np.asarray(coeff) // 2 * 2
    coeff[[b for b in bits if b < n]] += 1
    psi = random_state(n, n)
    ref = psi.copy()
    sim.apply_phase(ref, coeff, edges)
    h = qs.qs_alloc(n, qs.QS_C128)
    try:
        qs.qs_set_amplitudes(h, psi)
        qs.qs_apply_phase(h, coeff, edges)
        out = qs.qs_get_amplitudes(h)
    finally:
        qs.qs_free(h)
    assert np.all(np.abs(out - ref) <= 8 * EPS[qs.QS_C128] * np.abs(psi))


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("n", [16, 20, 22])
def test_phase_of_single_factors(n, dtype):
    """Factors on a chunk's own bits, above them and across: chunks that none reaches stay as they are."""
    psi = rounded(random_state(n, n), dtype)
    h = qs.qs_alloc(n, dtype)
    try:
        for bits in [(0,), (9,), (10,), (13,), (n - 1,), (1, 3), (2, n - 1), (9, n - 2), (13, n - 1), (n - 2, n - 1)]:
            coeff, edges = np.zeros(n, dtype=np.int64), [bits] if len(bits) == 2 else []
            coeff[bits[0]] = 0 if edges else 3
            ref = psi.copy()
            sim.apply_phase(ref, coeff, edges)
            qs.qs_set_amplitudes(h, psi)
            qs.qs_apply_phase(h, coeff, edges)
            out = qs.qs_get_amplitudes(h)
            assert np.all(np.abs(out - ref) <= 8 * EPS[dtype] * np.abs(psi)), bits
    finally:
        qs.qs_free(h)


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("n,k", [(1, 1), (2, 2), (8, 3), (9, 9), (10, 1), (14, 12), (19, 6), (20, 12), (23, 5)])
def test_table_rows_and_chunks(dtype, n, k):
    qubits, d = random_qubits(n, k, 5 * n + k), random_diag(k, k)
    psi = rounded(random_state(n, n + 1), dtype)
    ref = psi.copy()
    sim.apply_diag(ref, qubits, d)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        qs.qs_apply_diag(h, qubits, d)
        out = qs.qs_get_amplitudes(h)
    finally:
        qs.qs_free(h)
    # the table's rounding, one rounded product and one rounded sum per component
    assert np.all(np.abs(out - ref) <= 8 * EPS[dtype] * np.abs(psi))


def device_ms(calls, reps=20):
    torch = pytest.importorskip("torch")
    out = []
    for call in calls:
        best = float("inf")
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(reps):
                call()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / reps)
        out.append(best)
    return out


@pytest.mark.parametrize("q", [5, 8, 9, 12, 13, 24])
def test_one_t_gate_costs_no_more_than_the_whole_state(q):
    """complex128: a T gate off the lanes' bits turns half of the amplitudes, so it takes no
    longer than one on bit 0, which reads and writes every sector (it took 1.6 to 1.8
    times as long where the FP64 pipe was given the other half as well, or where half of
    the blocks had no chunk with work)."""
    n = 25
    h = qs.qs_alloc(n, qs.QS_C128)
    try:
        qs.qs_init_uniform(h)
        t = [np.eye(n, dtype=int)[b] for b in (0, q)]
        all_of_it, half = device_ms([lambda c=c: qs.qs_apply_phase(h, c, []) for c in t])
    finally:
        qs.qs_free(h)
    assert half <= 1.25 * all_of_it
