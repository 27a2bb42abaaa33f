"""Marginal probabilities: how a chunk's sums meet, for every kind of measured bit within it."""

import random

import numpy as np
import pytest

import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu

# bits of a 2^12 chunk: those a thread's own sums differ in (complex64: 0, 9..11; complex128: 8..11), the lanes'
# (1..5; 0..4), the warps'; and bits above the chunk
SETS = [[], [0], [9, 11], [0, 9, 10, 11], [8, 10], [1, 2, 3, 4, 5], [0, 1, 2, 3, 4], [2, 5], [6, 7, 8], [5, 6],
        list(range(12)), [12], [11, 12, 3], [13, 0, 7, 12, 10, 4]]


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [12, 14, 17])
def test_marginals(n, dtype):
    r, g = random.Random(n), np.random.default_rng(n)
    npdt = np.complex64 if dtype == qs.QS_C64 else np.complex128
    x = (g.standard_normal(1 << n) + 1j * g.standard_normal(1 << n)).astype(npdt)
    x /= npdt(np.linalg.norm(x))
    x[5] = np.nan
    st = qs.qs_alloc_state(n, dtype)
    try:
        qs.qs_write_state(st, x)
        w = np.abs(x.astype(np.complex128)) ** 2
        for qubits in SETS + [r.sample(range(n), r.randint(1, n)) for _ in range(4)]:
            qubits = [q for q in qubits if q < n]
            r.shuffle(qubits)
            got = qs.qs_measure_probs(st, qubits)
            bins = np.zeros(1 << n, dtype=np.int64)
            for j, q in enumerate(qubits):
                bins |= ((np.arange(1 << n) >> q) & 1) << j
            want = np.bincount(bins, weights=w, minlength=1 << len(qubits))
            bad = np.isnan(want)
            assert bad.sum() == 1 and np.array_equal(np.isnan(got), bad), qubits
            # complex64: the squares are rounded to FP32 (2 roundings of 2^-24 each), the sums compensated
            rel = 2.0 ** -22 if dtype == qs.QS_C64 else 1e-13
            assert np.all(np.abs(got[~bad] - want[~bad]) <= rel * want[~bad]), qubits
    finally:
        qs.qs_free_state(st)
