"""Operands of single tensor-core blocks made on the device: more blocks in a call than one launch takes."""

import random

import numpy as np
import pytest

import circuitgen as cg
import oracle
import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu


# a block's error in a direction of its own, and what truncation takes off the norm, of the same sign in every
# block (below the spacing of FP32 numbers at the factor that puts the norm right): 1.2e-7 and 2.4e-8 with FP16
# halves, 1e-16 and none with digit planes; the FP64 oracle's own 1e-16 for each of 13 to 17 gates of a block
@pytest.mark.parametrize("dtype,k,own,common", [
    (qs.QS_C64, 4, 1.2e-7, 2.4e-8), (qs.QS_C64, 5, 1.2e-7, 2.4e-8), (qs.QS_C64, 6, 1.2e-7, 2.4e-8),
    (qs.QS_C128, 4, 4e-16, 0), (qs.QS_C128, 5, 4e-16, 0)])
def test_many_blocks(dtype, k, own, common):
    n, blocks = 2 * k - 1, 1203  # two sets of k qubits that share one: blocks alternate and cannot merge
    r = random.Random(k)
    gates = []
    for b in range(blocks):
        q = list(range(k)) if b % 2 == 0 else list(range(k - 1, n))
        gates += [("u3", [x], [r.uniform(0, 6.28) for _ in range(3)]) for x in q]
        gates += [("cx", [x, y]) for x, y in zip(q, q[1:])]
    st = qs.qs_alloc_state(n, dtype)
    try:
        qs.qs_apply_circuit(st, qs.gates_to_array(gates), qs.QS_FUSE | qs.QS_FUSE_K(k) | qs.QS_TC)
        recs = qs.qs_profile(st)[1]
        assert len(recs) > 1000 and sum(r.tc > 0 for r in recs) > 1000
        got = qs.qs_read_state(st, n, dtype).astype(np.complex128)
    finally:
        qs.qs_free_state(st)
    want, _ = oracle.simulate(cg.to_qasm(n, gates))
    e = np.linalg.norm(got - want)
    assert e <= 1.5 * (own * blocks ** 0.5 + common * blocks)
