"""Statistics of equal amplitudes, where every thread's sum takes the same steps and
rounding errors add up instead of averaging out: against exact rationals."""
import math
from fractions import Fraction

import numpy as np
import pytest

import paper_1704_01127_gb300.qs as qs

pytestmark = pytest.mark.gpu

# A thread adds its terms 16 at a time in float-float.  After k equal terms the low word
# is at most k 2^-24 of the sum, so its 16 roundings come to 94 2^-48 of the sum at most
# (the sum of k^2 / 16); a term itself errs by 4 2^-48, p^2 and p ln p by about 8 2^-48; and
# the total of T such sums by T 2^-48.  1725 terms a thread (28 qubits, 608 blocks):
# (94 + 8 + 108) 2^-48 = 7.5e-13.  complex64: 32 terms without low parts of their own, so half
# of 358 2^-48 in the place of 94 2^-48: 8.4e-13 with 862 terms.
BOUND = 1e-12


def check(got, n, x, y, c128):
    p, N = Fraction(x) ** 2 + Fraction(y) ** 2, 1 << n
    # complex64: p^2 rounded to 32 bits, p is exact for these x, y; its logarithm has 32 bits only
    pp = p * p if c128 else Fraction(float(np.float32(float(p)) * np.float32(float(p))))
    want = [N * p, -N * p * Fraction(math.log(p)), N * p, N * N * pp]
    for i, (g, w) in enumerate(zip(got, want)):
        if i != 1 or c128:
            assert abs(Fraction(g) / w - 1) <= BOUND, (i, float(Fraction(g) / w - 1))


@pytest.mark.parametrize("dtype,n", [(qs.QS_C128, 24), (qs.QS_C128, 26), (qs.QS_C128, 28), (qs.QS_C64, 25), (qs.QS_C64, 28)])
@pytest.mark.parametrize("pick", range(3))
def test_equal_amplitudes(dtype, n, pick):
    torch = pytest.importorskip("torch")
    if dtype == qs.QS_C128:
        x, y = [(0.57735, 0.0), (0.7234567, 0.3111), (-0.1, 1.3)][pick]
    else:                       # x^2 + y^2 below 2^24 2^-22: exact in 32 bits
        x, y = [(2731 / 2048, 1755 / 2048), (0.0, 3001 / 2048), (-1111 / 2048, 2222 / 2048)][pick]
    x, y = x * 2.0 ** -(n // 2), y * 2.0 ** -(n // 2)
    psi = torch.full((1 << n,), complex(x, y), dtype=torch.complex128 if dtype == qs.QS_C128 else torch.complex64, device="cuda")
    torch.cuda.synchronize()
    c128 = dtype == qs.QS_C128
    h = qs.qs_wrap(psi, n, dtype)
    try:
        check([qs.qs_norm(h)], n, x, y, c128)
        check(qs.qs_stats(h), n, x, y, c128)
        check(qs.qs_sample_stats(h, 3, 16)[1], n, x, y, c128)
        check(qs.qs_stats_static(psi.data_ptr(), n, dtype), n, x, y, c128)
    finally:
        qs.qs_free(h)
