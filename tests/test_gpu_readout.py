"""Results read out: amplitudes by index (more and fewer indices than one launch
takes, none, one out of range, qubits moved to other bits)."""
import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs
from inputs import random_state, rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
@pytest.mark.parametrize("count", [0, 1, 31, 480, 481, 65536, 65536 + 481])
def test_gather(dtype, count):
    n = 12
    psi = random_state(n, 3).astype(np.complex64).astype(np.complex128)
    h = qs.qs_alloc(n, dtype)
    try:
        qs.qs_set_amplitudes(h, psi)
        idx = rng(count).integers(0, 1 << n, count)
        assert np.array_equal(qs.qs_get_amplitudes_at(h, idx), psi[idx])
        with pytest.raises(qs.QSError):
            qs.qs_get_amplitudes_at(h, np.append(idx, 1 << n))
    finally:
        qs.qs_free(h)


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
