"""Narrow states whose blocks share a launch, and batches whose wide circuits
run as cache-blocked passes: against the FP64 oracle at the edges of their
ranges."""

import numpy as np
import pytest

import circuitgen as cg
import oracle
import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu


def _run(n, gates, flags, init, opts=None):
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        qs.qs_write_state(st, init.astype(np.complex64))
        qs.qs_apply_circuit(st, qs.gates_to_array(gates), flags, opts)
        return qs.qs_read_state(st, n, qs.QS_C64, logical_order=True).astype(np.complex128)
    finally:
        qs.qs_free_state(st)


def _diagonal_runs(n, rng):
    """H layers with runs of phases on any pairs between them."""
    gates = []
    for _ in range(3):
        gates += [("h", [q]) for q in range(n)]
        for _ in range(4 * n):
            a, b = cg.random_pair(rng, n)
            gates.append((("rzz", "cp", "crz")[rng.randint(3)], [a, b], [rng.uniform(-6, 6)]))
        gates += [("t", [rng.randint(n)], []), ("rz", [rng.randint(n)], [rng.uniform(-6, 6)])]
    return gates


# 1 and 2 qubits, the fewest threads (9), a change of the thread count (10, 13), the widest (13); circuits whose
# records fill several launches
@pytest.mark.parametrize("n", [1, 2, 3, 9, 10, 11, 13])
@pytest.mark.parametrize("flags", [qs.QS_PGO_RULES, qs.QS_VSWAP | qs.QS_FUSE | qs.QS_FUSE_K(4) | qs.QS_DIAG,
                                   qs.QS_FUSE | qs.QS_FUSE_K(1), qs.QS_DIAG])
def test_narrow_states(n, flags):
    rng = cg.SplitMix64(100 + n)
    gates = [g for g in cg.all_gate_types_circuit(n, 250, rng)]
    if n > 2:
        gates += _diagonal_runs(n, rng)
    init = np.array([rng.uniform(-1, 1) + 1j * rng.uniform(-1, 1) for _ in range(1 << n)])
    init /= np.linalg.norm(init)
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init)
    got = _run(n, gates, flags, init)
    # FP32 blocks one by one take the same gates: a few 1e-8 per block and norm 1
    assert np.linalg.norm(got - want) < 5e-6
    # an explicit CTA size keeps the block-by-block kernels
    opts = qs.qs_default_opts()
    opts.threads = 256
    assert np.linalg.norm(got - _run(n, gates, flags, init, opts)) < 5e-6


def test_batch_of_wide_circuits():
    """From the widest narrow circuit (14) up: every gate type, diagonal runs over all qubits, no gate at
    all, one gate, and passes of one member; each run starts from |0...0>."""
    rng = cg.SplitMix64(9)
    circuits = []
    for n in (14, 15, 16, 18):
        circuits.append((n, cg.all_gate_types_circuit(n, 150, rng)))
        circuits.append((n, _diagonal_runs(n, rng)))
    circuits += [(15, []), (16, [("h", [15])]), (20, cg.ghz(20)), (15, [("swap", [0, 14]), ("x", [14])]),
                 (14, []), (17, [("h", [q]) for q in range(17)] + [("cswap", [16, 3, 14]), ("ccx", [15, 16, 2])])]
    for flags in (qs.QS_VSWAP | qs.QS_DIAG, qs.QS_FUSE | qs.QS_FUSE_K(1), qs.QS_FUSE | qs.QS_FUSE_K(6)):
        states = [qs.qs_alloc_state(n, qs.QS_C64) for n, _ in circuits]
        try:
            for (n, _), st in zip(circuits, states):
                qs.qs_set_basis(st, (1 << n) - 1)
            qs.qs_apply_batch(states, [qs.gates_to_array(g) for _, g in circuits], flags)
            for i, ((n, gates), st) in enumerate(zip(circuits, states)):
                want, _ = oracle.simulate(cg.to_qasm(n, gates))
                got = qs.qs_read_state(st, n, qs.QS_C64, logical_order=True).astype(np.complex128)
                assert np.linalg.norm(got - want) < 5e-6, (flags, i, n)
        finally:
            for st in states:
                qs.qs_free_state(st)


def test_bytes_shipped_are_those_of_the_launches():
    """A narrow state's gate data are its records, in the parameters of its launches."""
    n = 12
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        shipped = []
        for layers in (2, 40):
            gates = qs.gates_to_array(cg.random_layered(n, layers, cg.SplitMix64(layers)))
            qs.qs_apply_circuit(st, gates, qs.QS_PGO_RULES)
            summary, recs = qs.qs_profile(st)
            assert len(recs) > 1 and all(r.tiles == 0 for r in recs)
            shipped.append(summary.h2d_bytes)
        # launch parameters of 32 KB, whole; the matrices of the deeper circuit's blocks take several
        assert 32000 < shipped[0] < 32764 and shipped[1] % shipped[0] == 0 and shipped[1] > shipped[0]
    finally:
        qs.qs_free_state(st)
