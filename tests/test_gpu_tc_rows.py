"""complex64 tensor-core sweeps that move neighbouring groups together (lowest
target 1 to 4, many tiles): against the CUDA-core sweeps of the same ops, on the
full state, on a support that a sweep widens, and with a folded phase op."""
import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_phase_poly, random_unitary

pytestmark = pytest.mark.gpu

N = 24   # 4096 tiles of 128 groups


def dense(qubits, seed):
    return (qs.QS_OP_DENSE, qubits, random_unitary(len(qubits), seed))


def run(ops, path):
    sched = qs.qs_schedule_from_ops(N, ops)
    h = qs.qs_alloc(N, qs.QS_C64)
    try:
        qs.qs_set_path(h, path)
        qs.qs_init_basis(h, 5)
        qs.qs_run_circuit(h, sched)
        return qs.qs_get_amplitudes(h)
    finally:
        qs.qs_free(h)
        qs.qs_schedule_free(sched)


@pytest.mark.parametrize("low", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", ["full", "widens", "phase"])
def test_neighbouring_rows(low, kind):
    ops = [dense((0, 1, 2, 3, 4), 1), dense((5, 6, 7, 8, 9), 2), dense((10, 11, 12, 13, 14), 3), dense((15, 16, 17, 18, 19), 4)]
    if kind != "widens":
        ops.append(dense((19, 20, 21, 22, 23), 5))
        ops.append(dense((low, low + 1, 11, 20, 23), 6))
    else:
        ops.append(dense((low, 20, 21, 22, 23), 6))
    if kind == "phase":
        coeff, edges = random_phase_poly(N, 30, 7)
        coeff = np.asarray(coeff) // 2 * 2     # even off the targets: it folds into the sweep
        ops.append((qs.QS_OP_PHASE, edges, coeff))
    got, want = run(ops, qs.QS_PATH_TENSOR), run(ops, qs.QS_PATH_CUDA_CORES)
    # rounded FP32 sums of 32 terms, at most seven sweeps: about 1.5e-7 each on either path
    assert np.linalg.norm(got - want) <= 2e-6
    assert np.max(np.abs(got - want)) <= 2e-6
