"""Tensor-core tile passes as planned (host only): the product of their member blocks, applied in plan order to a
state, against the oracle. Wide states are compressed to the qubits that the circuit and the plan touch."""

import random

import numpy as np
import pytest

import circuitgen as cg
import oracle
import paper_2410_09326_gb300 as qs
from test_host import apply_block


def _layers(qubits, layers, seed, kinds):
    r = random.Random(seed)
    gates = []
    for _ in range(layers):
        gates += [("u3", [q], [r.uniform(0, 6.28) for _ in range(3)]) for q in qubits]
        q = r.sample(qubits, len(qubits))
        for a, b, c in zip(q[::3], q[1::3], q[2::3]):
            k = r.choice(kinds)
            if k in ("ccx", "cswap"):
                gates.append((k, [a, b, c]))
            elif k in ("cx", "cz", "swap"):
                gates.append((k, [a, b]))
            else:
                gates.append((k, [a, b], [r.uniform(0, 6.28)]))
    return gates


def _check(n, gates, seed):
    """The records of the plan under the rules, after its blocks have reproduced the circuit."""
    recs, mats, perm = qs.qs_plan(n, qs.gates_to_array(gates), qs.QS_PGO_RULES)
    used = {q for g in gates for q in g[1]} | {q for r in recs if r.kind != 3 for q in r.qubits if q >= 0}
    used |= {q for r in recs for q in range(n) if r.cmask >> q & 1}
    used = sorted(used)
    assert {int(perm[q]) for q in used} == set(used) and len(used) <= 16
    at = {q: i for i, q in enumerate(used)}
    m = len(used)
    g = np.random.default_rng(seed)
    psi = g.standard_normal(1 << m) + 1j * g.standard_normal(1 << m)
    psi /= np.linalg.norm(psi)
    want, _ = oracle.simulate(cg.to_qasm(m, [(x[0], [at[q] for q in x[1]], *x[2:]) for x in gates]), init=psi)
    tile, index = None, -1
    for r, mat in zip(recs, mats):
        if r.kind == 3:
            # the contiguous low bits and the ones named: members act non-diagonally on no others
            tile = {0, 1, 2, 3} | {q for q in r.qubits if q >= 0}
            index = r.index
            assert r.tc and r.k == 12 and len(tile) == 12
            continue
        q = [r.qubits[j] for j in range(r.k)]
        if r.tc and r.kind == 0 and r.meta == 4 and r.index == index:
            inside = [x for x in q if x in tile]
            assert len(inside) <= 5 and r.k - len(inside) <= 2
            for x in set(q) - set(inside):  # block-diagonal in the bits outside the tile
                bit = (np.arange(1 << r.k) >> q.index(x)) & 1
                assert not mat[bit[:, None] != bit[None, :]].any()
        for j in range(r.k):
            r.qubits[j] = at[q[j]]
        if r.kind == 4:
            mat["qubits"] = np.array([at[int(x)] for x in mat["qubits"]])
        r.cmask = sum(1 << at[x] for x in range(n) if r.cmask >> x & 1)
        psi = apply_block(psi, m, r, mat)
    assert np.linalg.norm(psi - oracle.to_physical(want, [at[int(perm[x])] for x in used])) < 1e-12
    return recs


# where blocks are grouped by first fit, by roll-outs (from 23 qubits on) and passes too (from 26 on)
@pytest.mark.parametrize("n", [14, 18, 22, 23, 25, 26, 30])
@pytest.mark.parametrize("kinds", [["cx", "cz"], ["cx", "cp", "rzz", "swap"], ["ccx", "cswap", "crx", "cz"]])
def test_plan_reproduces_the_oracle(n, kinds):
    # 13 or 14 qubits, low ones and others
    r = random.Random(n)
    qubits = sorted(r.sample(range(5), 4) + r.sample(range(5, n), 9))
    recs = _check(n, _layers(qubits, 5, n, kinds), n)
    assert any(r.kind == 3 for r in recs)


def test_passes_split_at_32_blocks():
    recs = _check(14, _layers(list(range(11)), 60, 1, ["cx"]), 1)
    passes = [r for r in recs if r.kind == 3]
    members = [sum(q.kind != 3 and q.index == p.index for q in recs) for p in passes]
    assert len(passes) >= 2 and members[0] == 32
    assert list(passes[0].qubits) == list(passes[1].qubits)


def test_where_no_tile_passes_are_planned():
    """A lone block, blocks of up to three qubits, narrow states, options that ask for a kernel, timed calls, and
    explicit flags."""
    n = 16
    gates = qs.gates_to_array(_layers(list(range(n)), 4, 2, ["cx"]))
    opts = qs.qs_default_opts()

    def tiles(n, arr, flags=qs.QS_PGO_RULES):
        return any(r.kind == 3 for r in qs.qs_plan(n, arr, flags, opts=opts)[0])

    assert tiles(n, gates)
    assert not tiles(n, gates, qs.QS_PGO_RULES | qs.QS_PROFILE)
    assert not tiles(n, gates, qs.QS_VSWAP | qs.QS_FUSE | qs.QS_FUSE_K(5) | qs.QS_DIAG | qs.QS_TC)
    assert not tiles(n, qs.gates_to_array(_layers([1, 5, 9, 13, 14], 4, 3, ["cx"])))
    assert not tiles(n, qs.gates_to_array([("ccx", [0, 5, 9]), ("ccx", [13, 2, 4]), ("ccx", [7, 8, 12])]))
    assert not tiles(12, qs.gates_to_array(_layers(list(range(12)), 4, 2, ["cx"])))
    for name in ("threads", "tc_exchange", "tc_precision"):
        setattr(opts, name, 1 if name != "threads" else 256)
        assert not tiles(n, gates), name
        setattr(opts, name, 0)
