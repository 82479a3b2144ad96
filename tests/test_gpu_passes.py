"""Passes (several CUDA-core ops per read and write of the state) against the
same ops as one sweep each (qs_run_circuit_timed runs every op by itself): the
same bits, at states below, of and above one chunk, with targets everywhere, odd
phases on the lanes' bits and off them, more ops than one pass holds and operands
larger than the CTA's buffer."""
import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_diag, random_phase_poly, random_qubits, random_state, random_unitary

pytestmark = pytest.mark.gpu


def random_ops(n, count, seed, kinds):
    rng = np.random.Generator(np.random.PCG64(seed))
    ops = []
    for i in range(count):
        kind = kinds[rng.integers(len(kinds))]
        if kind == "phase":
            coeff, edges = random_phase_poly(n, int(rng.integers(0, 2 * n)) if n > 1 else 0, seed + i)
            coeff = np.asarray(coeff) * (rng.random(n) < rng.choice([0.1, 0.5, 1.0]))
            if rng.random() < 0.3:
                coeff = coeff // 2 * 2
            ops.append((qs.QS_OP_PHASE, edges, coeff))
        else:
            k = min(n, int(kind))
            q = random_qubits(n, k, seed + i)
            ops.append((qs.QS_OP_DENSE, q, random_unitary(k, seed + i)))
    return ops


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("kinds", [("1", "phase"), ("2", "3", "phase"), ("4", "5"), ("phase",)], ids=lambda k: "".join(k))
@pytest.mark.parametrize("n", [1, 2, 3, 5, 7, 8, 9, 12, 13, 16, 19, 20, 21, 22])
def test_passes_equal_sweeps(dtype, kinds, n):
    psi = random_state(n, n)
    sched = qs.qs_schedule_from_ops(n, random_ops(n, 40 if n <= 20 else 12, 17 * n, kinds))
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_path(h, qs.QS_PATH_CUDA_CORES)
        out = []
        for run in (qs.qs_run_circuit_timed, qs.qs_run_circuit):
            qs.qs_set_amplitudes(h, psi)
            run(h, sched)
            out.append(qs.qs_get_amplitudes(h))
    finally:
        qs.qs_free(h)
        qs.qs_schedule_free(sched)
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("sizes", [(1, 2, 4), (8, 9, 3), (16, 1, 17), (22,)])
def test_batches_from_zero_equal_sweeps(dtype, sizes):
    """Circuits of few ops leave index bits that no pass covers: zeros there, also in a second run."""
    torch = pytest.importorskip("torch")
    scheds = [qs.qs_schedule_from_ops(n, random_ops(n, c, 5 * n + c, ("1", "2", "4", "phase")))
              for n in sizes for c in (1, 9)]
    b = qs.qs_batch_create(scheds, dtype, torch.cuda.Stream())
    try:
        for threads in (128, 512):
            qs.qs_batch_set_config(b, 2, threads)
            for _ in range(2):
                qs.qs_batch_run(b)
            for i, sc in enumerate(scheds):
                n = sizes[i // 2]
                h = qs.qs_alloc(n, dtype)
                qs.qs_set_path(h, qs.QS_PATH_CUDA_CORES)
                qs.qs_init_basis(h, 0)
                qs.qs_run_circuit_timed(h, sc)
                want = qs.qs_get_amplitudes(h)
                qs.qs_free(h)
                assert np.array_equal(qs.qs_batch_get_amplitudes(b, i, n), want), (threads, i)
    finally:
        qs.qs_batch_free(b)
        for sc in scheds:
            qs.qs_schedule_free(sc)


def run_ms(h, n, ops, timed=False, reps=10):
    """Best time of qs_run_circuit on these ops; timed: of the ops as one sweep each."""
    torch = pytest.importorskip("torch")
    sched = qs.qs_schedule_from_ops(n, ops)
    best = float("inf")
    try:
        for _ in range(5):
            if timed:
                ms = np.sum(np.maximum(qs.qs_run_circuit_timed(h, sched), 0))
            else:
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                for _ in range(reps):
                    qs.qs_run_circuit(h, sched)
                b.record()
                b.synchronize()
                ms = a.elapsed_time(b) / reps
            best = min(best, ms)
    finally:
        qs.qs_schedule_free(sched)
    return best


def turn(n, q, eighths):
    return (qs.QS_OP_PHASE, [], eighths * np.eye(n, dtype=np.int64)[q])


def test_even_turns_leave_the_fp64_pipe_alone():
    """complex128: an S gate in a pass swaps and negates, a T gate is four FP64 operations an
    amplitude; a pass of S gates took as long as one of T gates where both went to that pipe."""
    n = 23
    h = qs.qs_alloc(n, qs.QS_C128)
    try:
        qs.qs_init_uniform(h)
        s, t = [run_ms(h, n, [turn(n, q, e) for q in range(20)]) for e in (2, 1)]
    finally:
        qs.qs_free(h)
    assert s <= 0.75 * t


@pytest.mark.parametrize("dtype,n,k", [(qs.QS_C128, 16, 3), (qs.QS_C128, 16, 4), (qs.QS_C128, 20, 1), (qs.QS_C128, 24, 1),
                                       (qs.QS_C64, 23, 2)])
def test_sweeps_in_turn_cost_no_more_than_one_by_one(dtype, n, k):
    """Table diagonals and clusters in turn: blocks of a sweep that starts early pile up on a few SMs
    (2 to 4 times the time in complex128, 1.3 in complex64)."""
    ops = [(qs.QS_OP_DIAG, [0, 3, n - 1], random_diag(3, 1)), (qs.QS_OP_DENSE, [2, 5, 8, 7, n - 1][-k:], random_unitary(k, k))] * 3
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_path(h, qs.QS_PATH_CUDA_CORES)
        qs.qs_init_uniform(h)
        together, apart = run_ms(h, n, ops), run_ms(h, n, ops, timed=True)
    finally:
        qs.qs_free(h)
    assert together <= 1.1 * apart


def few(kind, n):
    if kind == "phases":
        return [(qs.QS_OP_PHASE, *reversed(random_phase_poly(n, n, i))) for i in (1, 2)]
    if kind == "clusters and a phase":
        return few("phases", n)[:1] + [(qs.QS_OP_DENSE, [n - 1], random_unitary(1, 1))]
    return [(qs.QS_OP_PHASE, [pair], np.zeros(n, dtype=np.int64)) for pair in ((n - 2, n - 1), (n - 4, n - 3))]


@pytest.mark.parametrize("kind", ["phases", "pairs", "clusters and a phase"])
@pytest.mark.parametrize("dtype,n", [(qs.QS_C128, 21), (qs.QS_C128, 24), (qs.QS_C64, 24), (qs.QS_C64, 27)])
def test_few_ops_cost_no_more_than_their_sweeps(dtype, n, kind):
    """Two ops that a pass would not pay for (1.4 to 5 times the time of their sweeps)."""
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_path(h, qs.QS_PATH_CUDA_CORES)
        qs.qs_init_uniform(h)
        together, apart = run_ms(h, n, few(kind, n)), run_ms(h, n, few(kind, n), timed=True)
    finally:
        qs.qs_free(h)
    assert together <= 1.1 * apart
