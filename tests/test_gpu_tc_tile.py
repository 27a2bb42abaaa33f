"""Tile passes on the tensor cores (complex64, several fused blocks per launch) against the oracle."""

import random

import numpy as np
import pytest

import circuitgen as cg
import oracle
import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu

FLAGS = qs.QS_PGO_RULES


def _layers(n, layers, seed, kinds):
    r = random.Random(seed)
    gates = []
    for _ in range(layers):
        gates += [("u3", [q], [r.uniform(0, 6.28) for _ in range(3)]) for q in range(n)]
        q = r.sample(range(n), n)
        for a, b, c in zip(q[::3], q[1::3], q[2::3]):
            k = r.choice(kinds)
            if k in ("ccx", "cswap"):
                gates.append((k, [a, b, c]))
            elif k in ("cx", "cz", "swap"):
                gates.append((k, [a, b]))
            else:
                gates.append((k, [a, b], [r.uniform(0, 6.28)]))
    return gates


def _random_state(n, seed):
    g = np.random.default_rng(seed)
    x = g.standard_normal(1 << n) + 1j * g.standard_normal(1 << n)
    return x / np.linalg.norm(x)


def _run(n, gates, init, flags=FLAGS, opts=None):
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        qs.qs_write_state(st, init.astype(np.complex64))
        qs.qs_apply_circuit(st, qs.gates_to_array(gates), flags, opts)
        recs = qs.qs_profile(st)[1]
        return qs.qs_read_state(st, n, qs.QS_C64, logical_order=True).astype(np.complex128), recs
    finally:
        qs.qs_free_state(st)


def _bound(n, gates):
    """A member of a tile pass is off by 1.1e-7 of the state (FP16 halves of 22 bits, FP32 sums; a single block of the
    same kind by 1.2e-7), each in a direction of its own: twice the root of their sum of squares."""
    blocks = [r for r in qs.qs_plan(n, qs.gates_to_array(gates), FLAGS)[0] if r.kind not in (2, 3)]
    return 2.4e-7 * len(blocks) ** 0.5


# the narrowest state with tiles, several tiles, one that several CTAs loop over (ctas), many;
# controls and phases on any bit, 3-qubit gates, blocks that are the identity on some tiles
@pytest.mark.parametrize("n,ctas,kinds", [
    (14, 0, ["cx", "cp", "rzz", "swap"]), (14, 1, ["cx", "ccx"]),
    (14, 3, ["ccx", "cswap", "crx"]), (15, 3, ["cx", "cz"]), (16, 5, ["ccx", "cp", "cx"]),
    (18, 0, ["cx", "crx", "ccx"]), (20, 0, ["cx", "cz", "cp"]),
])
def test_against_oracle(n, ctas, kinds):
    gates = _layers(n, 4, 31 * n + ctas, kinds)
    init = _random_state(n, n)
    opts = qs.qs_default_opts()
    opts.tc_max_ctas = ctas
    got, recs = _run(n, gates, init, FLAGS, opts)
    tiles = [r for r in recs if r.kind == 3]
    assert tiles and all(r.tc and r.tiles == 1 << (n - 12) for r in tiles)
    assert all(r.ctas == (min(ctas, r.tiles) if ctas else min(r.tiles, r.ctas)) for r in tiles)
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init)
    assert np.linalg.norm(got - want) <= _bound(n, gates)


def test_errors_of_many_blocks_do_not_add_up():
    """64 dense blocks in a row: a block is off by 1.1e-7 of the state in a direction of its own (FP16 halves of 22
    bits, FP32 sums), so that they grow with the root of the count, to 9e-7. What the accumulation's truncation takes
    off the norm has the same sign in every block: not put right, 2.3e-8 each, 1.5e-6 in all."""
    n, r = 15, random.Random(1)
    gates = []
    for _ in range(64):
        t = r.sample(range(11), 5)
        for _ in range(3):
            gates += [("u3", [q], [r.uniform(0, 6.28) for _ in range(3)]) for q in t]
            q = r.sample(t, 5)
            gates += [("cx", [q[0], q[1]]), ("cx", [q[2], q[3]]), ("cx", [q[4], q[0]])]
    init = _random_state(n, 1)
    got, recs = _run(n, gates, init)
    assert [r.kind for r in recs] == [3, 3]  # 32 blocks a launch
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init.astype(np.complex64).astype(np.complex128))
    assert np.linalg.norm(got - want) <= 1.2e-6


@pytest.mark.parametrize("size", [1e-17, 1e-20, 1e-22, 1e-23, 1e-24, 1e-26, 1e-30, 1e-36, 1e-40])
def test_rows_whose_norm_underflows(size):
    """What cancellations leave behind: amplitudes whose squares are subnormal or zero in FP32. They may come out as
    zero, never larger than they were, and never as NaN."""
    n = 14
    gates = _layers(11, 3, 3, ["cx"])
    init = _random_state(n, 4).reshape(8, 1 << 11)
    init[1:] *= size
    init = init.astype(np.complex64)
    got, recs = _run(n, gates, init.reshape(-1))
    got = got.reshape(8, 1 << 11)
    assert any(r.kind == 3 for r in recs) and np.isfinite(got).all()
    assert np.abs(np.linalg.norm(got[0]) / np.linalg.norm(init[0].astype(np.complex128)) - 1) <= 1e-6
    for i in range(1, 8):
        assert np.linalg.norm(got[i]) <= 1.01 * np.linalg.norm(init[i].astype(np.complex128)) + 1e-44


def test_products_of_a_split_pass():
    """More blocks than a launch takes, most of them with two bits outside the tile that pick one of four products:
    the second launch's products follow the first's."""
    n, r = 14, random.Random(12)
    gates = []
    for _ in range(40):
        for c in (12, 13):
            gates += [("cu3", [c, q], [r.uniform(0, 6.28) for _ in range(3)]) for q in range(11)]
        q = r.sample(range(11), 11)
        gates += [("cx", [a, b]) for a, b in zip(q[::2], q[1::2])]
    init = _random_state(n, 3)
    got, recs = _run(n, gates, init)
    plan = qs.qs_plan(n, qs.gates_to_array(gates), FLAGS)[0]
    passes = [p for p in plan if p.kind == 3]
    members = [[m for m in plan if m.kind != 3 and m.index == p.index] for p in passes]
    outer = [[sum(q in (12, 13) for q in m.qubits) for m in x] for x in members]
    full = [i for i, x in enumerate(members) if len(x) == 32]
    assert full and all(passes[i + 1].qubits[:] == passes[i].qubits[:] for i in full)
    assert all(2 in outer[i] and 2 in outer[i + 1] for i in full)
    assert [p.kind for p in recs] == [p.kind for i, p in enumerate(plan) if i == 0 or p.index != plan[i - 1].index]
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init)
    assert np.linalg.norm(got - want) <= _bound(n, gates)


@pytest.mark.parametrize("n", [13, 14, 17, 23])
def test_the_plan_is_what_runs(n):
    gates = _layers(n, 4, n, ["cx", "cp", "ccx", "swap"])
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        qs.qs_apply_circuit(st, qs.gates_to_array(gates), FLAGS)
        ran = qs.qs_profile(st)[1]
    finally:
        qs.qs_free_state(st)
    plan = qs.qs_plan(n, qs.gates_to_array(gates), FLAGS)[0]
    assert any(r.kind == 3 for r in plan) == (n > 13)
    plan = [r for i, r in enumerate(plan) if i == 0 or r.index != plan[i - 1].index]  # without the passes' members
    assert [(r.kind, r.k, r.tc, r.n_gates, r.cmask, list(r.qubits)) for r in ran] == \
        [(r.kind, r.k, r.tc, r.n_gates, r.cmask, list(r.qubits)) for r in plan]


def test_every_block_controlled_from_outside_the_tile():
    """Blocks that only act where the highest bits are 1: tiles without work are left as they are."""
    n, top = 15, [13, 14]
    r = random.Random(5)
    gates = []
    for _ in range(6):
        gates += [("cu3", [top[q % 2], q], [r.uniform(0, 6.28) for _ in range(3)]) for q in range(11)]
        gates += [("ccx", [top[0], q, q + 1]) for q in range(0, 10, 2)]
    init = _random_state(n, 9)
    got, recs = _run(n, gates, init)
    assert any(r.kind == 3 for r in recs)
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init)
    assert np.linalg.norm(got - want) <= _bound(n, gates)
    quarter = np.arange(1 << n) >> 13 == 0
    assert np.array_equal(got[quarter].astype(np.complex64), init[quarter].astype(np.complex64))


def test_rows_of_any_size():
    """Groups far smaller than the rest, zero groups, NaN in one group: each keeps to itself."""
    n = 14
    gates = _layers(11, 3, 3, ["cx"])  # bits 0..10: one tile pass, whole tiles along the other bits
    init = _random_state(n, 4).reshape(8, 1 << 11)
    init[1] *= 1e-12
    init[2] = 0
    init[3, 5] = np.nan
    got, recs = _run(n, gates, init.reshape(-1))
    got = got.reshape(8, 1 << 11)
    assert any(r.kind == 3 for r in recs)
    text = cg.to_qasm(11, gates)
    for i in (0, 1, 4, 5, 6, 7):
        size = np.linalg.norm(init[i])
        want, _ = oracle.simulate(text, init=init[i] / size)
        assert np.linalg.norm(got[i] / size - want) <= _bound(n, gates), i
    assert (got[2] == 0).all() and np.isnan(got[3]).any()


def test_profiled_calls_scarce_memory_and_explicit_flags_run_block_by_block():
    n = 16
    gates = _layers(n, 5, 8, ["cx", "cz"])
    init = _random_state(n, 2)
    before = qs.qs_memory_in_use()
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        qs.qs_apply_circuit(st, qs.gates_to_array(gates), FLAGS | qs.QS_PROFILE)
        assert not any(r.kind == 3 for r in qs.qs_profile(st)[1])
        single = qs.qs_memory_in_use() - before
    finally:
        qs.qs_free_state(st)
    tiled, recs = _run(n, gates, init)
    assert any(r.kind == 3 for r in recs)
    qs.qs_set_memory_limit(before + single)
    try:
        blocks, recs = _run(n, gates, init)
    finally:
        qs.qs_set_memory_limit(0)
    assert not any(r.kind == 3 for r in recs)
    assert np.linalg.norm(tiled - blocks) <= 1e-5
    # explicit flags run the blocks they ask for
    _, recs = _run(n, gates, init, qs.QS_VSWAP | qs.QS_FUSE | qs.QS_FUSE_K(5) | qs.QS_DIAG | qs.QS_TC)
    assert not any(r.kind == 3 for r in recs)


@pytest.mark.parametrize("t", [[5, 6, 7], [1, 8, 14], [0, 3, 4, 9, 12]])
def test_a_lone_block_runs_by_itself(t):
    """A tile pass pays for several blocks."""
    n, r, gates = 16, random.Random(4), []
    for _ in range(3):
        gates += [("u3", [q], [r.uniform(0, 6.28) for _ in range(3)]) for q in t]
        gates += [("cx", [a, b]) for a, b in zip(t, t[1:])]
    init = _random_state(n, 6)
    got, recs = _run(n, gates, init)
    assert [(r.k, r.tc > 0) for r in recs if r.kind == 0] == [(len(t), len(t) > 3)]
    assert not any(r.kind == 3 for r in recs)
    want, _ = oracle.simulate(cg.to_qasm(n, gates), init=init.astype(np.complex64).astype(np.complex128))
    assert np.linalg.norm(got - want) <= 2.5e-7


def test_blocks_of_up_to_three_targets_keep_their_fp32_arithmetic():
    n = 16
    init = _random_state(n, 6)
    got, recs = _run(n, [("ccx", [0, 5, 9]), ("ccx", [13, 2, 4]), ("ccx", [7, 8, 12])], init)
    assert [(r.kind, r.k, r.nctrl, r.tc) for r in recs if r.kind != 2] == [(0, 1, 2, 0)] * 3
    x = np.arange(1 << n)
    for a, b, t in ((7, 8, 12), (13, 2, 4), (0, 5, 9)):
        x ^= ((x >> a) & (x >> b) & 1) << t
    assert np.array_equal(got.astype(np.complex64), init.astype(np.complex64)[x])


def test_timeout_is_reported():
    n = 14
    gates = qs.gates_to_array(_layers(n, 3, 1, ["cx"]))
    st = qs.qs_alloc_state(n, qs.QS_C64)
    try:
        opts = qs.qs_default_opts()
        opts.test_wait_timeout = 1
        qs.qs_apply_circuit(st, gates, FLAGS, opts)
        with pytest.raises(qs.QsError) as e:
            qs.qs_norm(st)
        assert e.value.status == qs.QS_ETIMEOUT
        opts.test_wait_timeout = 0
        qs.qs_set_basis(st, 0)
        qs.qs_apply_circuit(st, gates, FLAGS, opts)
        assert any(r.kind == 3 for r in qs.qs_profile(st)[1])
        assert abs(qs.qs_norm(st) - 1) < 1e-5
    finally:
        qs.qs_free_state(st)
