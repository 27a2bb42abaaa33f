"""Reading a state in logical order: the relabelling undone bit for bit, all exchanges of a set at once."""

import random

import numpy as np
import pytest

import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu


def _perms(n, r):
    yield list(range(n))[::-1]                        # bit reversal
    yield list(range(1, n)) + [0]                     # one cycle over all bits
    yield [x ^ 1 if x ^ 1 < n else x for x in range(n)]  # neighbours
    yield [n - 1] + list(range(1, n - 1)) + [0]       # a single exchange
    if n >= 4:                                        # two exchanges
        yield [n - 1, n - 2] + list(range(2, n - 2)) + [1, 0]
    for _ in range(3 if n < 24 else 1):
        yield r.sample(range(n), n)


# narrower than a tile, a tile, several, many; both amplitude sizes
@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 7, 8, 9, 11, 14, 17, 21, 24])
def test_logical_order_is_exact(n, dtype):
    r = random.Random(n)
    npdt = np.complex64 if dtype == qs.QS_C64 else np.complex128
    x = (np.arange(1 << n) + 1j).astype(npdt)  # below 2^24: exact
    idx = np.arange(1 << n)
    for want in _perms(n, r):
        # SWAPs that leave logical qubit l on bit want[l]
        at, gates = list(range(n)), []
        for l in range(n):
            if at[l] != want[l]:
                k = at.index(want[l])
                gates.append(("swap", [l, k]))
                at[l], at[k] = at[k], at[l]
        st = qs.qs_alloc_state(n, dtype)
        try:
            qs.qs_write_state(st, x)
            qs.qs_apply_circuit(st, qs.gates_to_array(gates), qs.QS_VSWAP)
            assert list(qs.qs_get_perm(st, n)) == want
            got = qs.qs_read_state(st, n, dtype, logical_order=True)
            assert list(qs.qs_get_perm(st, n)) == list(range(n))
        finally:
            qs.qs_free_state(st)
        phys = np.zeros(1 << n, dtype=np.int64)
        for l in range(n):
            phys |= ((idx >> l) & 1) << want[l]
        assert np.array_equal(got, x[phys]), want
