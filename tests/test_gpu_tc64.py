"""complex128 blocks of 4 and 5 targets on the tensor cores (digit planes):
against the FP64 product of the planned block matrix."""

import random

import numpy as np
import pytest

import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu


def _gates(targets, ctrl, seed):
    """A dense block on `targets`; with a control, only gates controlled by it."""
    r = random.Random(seed)
    g = []
    for _ in range(3):
        for q in targets:
            p = [r.uniform(0, 6.28) for _ in range(3)]
            g.append(("u3", [q], p) if ctrl is None else ("cu3", [ctrl, q], p))
        t = r.sample(targets, len(targets))
        for a, b in zip(t[::2], t[1::2]):
            g.append(("cx", [a, b], []) if ctrl is None else ("ccx", [ctrl, a, b], []))
    return qs.gates_to_array(g)


def _expected(n, rec, mat, x):
    t = [q for q in rec.qubits if q >= 0]
    idx = np.arange(1 << n)
    low = idx[(idx & sum(1 << q for q in t)) == 0]
    low = low[(low & rec.cmask) == rec.cmask]
    off = np.array([sum(((s >> j) & 1) << q for j, q in enumerate(t)) for s in range(1 << len(t))])
    y = x.copy()
    at = low[:, None] + off[None]
    y[at] = x[at] @ mat.T
    return y, at


def _run(n, gates, x, opts=None):
    import torch
    t = torch.from_numpy(x).cuda()
    st = qs.qs_attach_state(t.data_ptr(), n, qs.QS_C128)
    try:
        width = 6 if gates[0]["nq"] > 1 else 5
        qs.qs_apply_circuit(st, gates, qs.QS_FUSE | qs.QS_FUSE_K(width) | qs.QS_TC, opts)
        recs = qs.qs_profile(st)[1]
        qs.qs_norm(st)
        return t.cpu().numpy(), recs, width
    finally:
        qs.qs_free_state(st)


# fewer groups than a tile, one tile, ragged and many tiles; low, high and spread targets; a control below,
# between and above them
@pytest.mark.parametrize("n,targets,ctrl,ctas", [
    (4, [0, 1, 2, 3], None, 0), (5, [0, 1, 2, 3, 4], None, 0), (6, [0, 2, 3, 5], None, 0), (7, [1, 2, 4, 5, 6], 0, 0),
    (11, [7, 8, 9, 10], None, 0), (12, [7, 8, 9, 10, 11], None, 0), (13, [0, 1, 2, 12], 6, 0),
    (15, [0, 1, 2, 3, 4], None, 3), (15, [3, 6, 9, 12, 14], None, 3), (14, [2, 5, 9, 13], None, 3),
    (16, [1, 4, 8, 11, 13], 15, 3), (18, [0, 5, 9, 13, 17], None, 0),
])
def test_blocks_match_the_fp64_product(n, targets, ctrl, ctas):
    gates = _gates(targets, ctrl, n)
    rng = np.random.default_rng(n)
    x = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    x *= np.exp2(rng.integers(-40, 0, 1 << n))  # amplitudes of very different size in one group
    opts = qs.qs_default_opts()
    opts.tc_max_ctas = ctas
    got, recs, width = _run(n, gates, x, opts)
    (plan,), (mat,), _ = qs.qs_plan(n, gates, qs.QS_FUSE | qs.QS_FUSE_K(width))
    (rec,) = recs
    assert rec.tc == 1 and rec.k == len(targets) and rec.nctrl == (ctrl is not None)
    if ctas:
        assert rec.ctas == ctas and rec.tiles > 2 * ctas
    want, at = _expected(n, plan, mat, x)
    # one rounding of the result and digits to 2^-55 of the group's largest, against numpy's 2^(k + 1)
    # roundings of products: both within 2^(k + 1) units of 2^-53 of the group's norm
    bound = 2.0 ** (len(targets) + 1 - 53) * np.linalg.norm(x[at], axis=1)
    assert (np.abs(got[at] - want[at]).max(1) <= bound).all()
    rest = np.ones(1 << n, dtype=bool)
    rest[at.ravel()] = False
    assert np.array_equal(got[rest], x[rest])


@pytest.mark.parametrize("k", [4, 5])
def test_extreme_scales(k):
    """Group norms from subnormal to near the largest number; zero groups; infinities and NaN."""
    n = 11
    gates = _gates(list(range(n - k, n)), None, 3)
    rng = np.random.default_rng(2)
    g = 1 << (n - k)
    x = (rng.standard_normal((1 << k, g)) + 1j * rng.standard_normal((1 << k, g))) * 2.0 ** -3
    e = np.linspace(-1060, 1020, g).astype(int)
    x = np.ldexp(np.ldexp(x.view(np.float64).reshape(1 << k, g, 2), (e // 2)[None, :, None]),
                 (e - e // 2)[None, :, None]).view(np.complex128)[..., 0]
    x[:, 5] = 0
    x[1, 9] = np.inf
    x[3, 11] = np.nan
    got, recs, _ = _run(n, gates, np.ascontiguousarray(x.reshape(-1)))
    got = got.reshape(1 << k, g)
    assert [r.tc for r in recs] == [1]
    _, (mat,), _ = qs.qs_plan(n, gates, qs.QS_FUSE | qs.QS_FUSE_K(5))
    fine = np.ones(g, dtype=bool)
    fine[[9, 11]] = False
    assert np.isnan(got[:, ~fine]).all() and (got[:, 5] == 0).all()
    # scaled by powers of two into the middle of the range and back, so that numpy's products are exact there
    y = np.ldexp(np.ldexp(x.copy().view(np.float64).reshape(1 << k, g, 2)[:, fine], (-e[fine] // 2)[None, :, None]),
                 (-e[fine] - (-e[fine] // 2))[None, :, None]).view(np.complex128)[..., 0]
    have = np.ldexp(np.ldexp(got.copy().view(np.float64).reshape(1 << k, g, 2)[:, fine], (-e[fine] // 2)[None, :, None]),
                    (-e[fine] - (-e[fine] // 2))[None, :, None]).view(np.complex128)[..., 0]
    # plus one subnormal unit 2^-1074, scaled the same way
    bound = 2.0 ** (k + 1 - 53) * np.linalg.norm(y, axis=0) + np.exp2(np.maximum(-1072.0 - e[fine], -200))
    assert (np.abs(have - mat @ y).max(0) <= bound).all()


@pytest.mark.parametrize("k", [4, 5])
def test_timeout_is_reported(k):
    n = 14
    gates = _gates(list(range(k)), None, 5)
    st = qs.qs_alloc_state(n, qs.QS_C128)
    try:
        opts = qs.qs_default_opts()
        opts.test_wait_timeout = 1
        flags = qs.QS_FUSE | qs.QS_FUSE_K(5) | qs.QS_TC
        qs.qs_apply_circuit(st, gates, flags, opts)
        with pytest.raises(qs.QsError) as e:
            qs.qs_norm(st)
        assert e.value.status == qs.QS_ETIMEOUT
        opts.test_wait_timeout = 0
        qs.qs_set_basis(st, 0)
        qs.qs_apply_circuit(st, gates, flags, opts)
        assert abs(qs.qs_norm(st) - 1) < 1e-14
    finally:
        qs.qs_free_state(st)


# explicit flags, and the rules (which take blocks of five targets)
@pytest.mark.parametrize("flags", [qs.QS_FUSE | qs.QS_FUSE_K(5) | qs.QS_TC, qs.QS_FUSE | qs.QS_FUSE_K(4) | qs.QS_TC,
                                   qs.QS_PGO_RULES])
def test_small_rotations_keep_their_small_amplitudes(flags):
    """RX(2e-9) on every qubit of |0...0>: an amplitude with j flips is 1e-9 to the j, each exact to FP64."""
    n, t = 10, 2e-9
    st = qs.qs_alloc_state(n, qs.QS_C128)
    try:
        qs.qs_apply_circuit(st, qs.gates_to_array([("rx", [q], [t]) for q in range(n)]), flags)
        assert sum(r.tc for r in qs.qs_profile(st)[1]) >= 2
        got = qs.qs_read_state(st, n, qs.QS_C128, logical_order=True)
    finally:
        qs.qs_free_state(st)
    flips = np.array([bin(i).count("1") for i in range(1 << n)])
    want = (-1j) ** flips * np.sin(t / 2) ** flips * np.cos(t / 2) ** (n - flips)
    # two to three blocks of FP64 products of gates and amplitudes, 2^6 roundings each at most
    assert (np.abs(got - want) <= 3 * 2.0 ** (6 - 53) * np.abs(want)).all()


# part of a tile, one tile, tiles that three CTAs loop over
@pytest.mark.parametrize("n,targets,ctas", [
    (7, [0, 1, 2, 3], 0), (8, [0, 2, 4, 5, 7], 0), (11, [0, 1, 2, 3], 0), (12, [2, 3, 7, 8, 11], 0),
    (15, [1, 4, 6, 9], 3), (16, [0, 1, 2, 3, 4], 3)])
@pytest.mark.parametrize("tiny", [0.0, 1e-7])
def test_groups_of_very_different_amplitudes_take_fp64(n, targets, ctas, tiny):
    """A matrix that mixes one qubit and moves the others about keeps small amplitudes apart from large ones."""
    k = len(targets)
    gates = [("u3", [targets[0]], [1.1, 0.3, 0.7])]
    gates += [("cx", [a, b], []) for _ in range(2) for a, b in zip(targets, targets[1:] + targets[:1])]
    if tiny:  # weights far below 1 between the halves of another qubit
        gates += [("ry", [targets[1]], [tiny])]
    gates = qs.gates_to_array(gates)
    rng = np.random.default_rng(3)
    groups = 1 << (n - k)
    y = (rng.standard_normal((groups, 1 << k)) + 1j * rng.standard_normal((groups, 1 << k)))
    wide = rng.random(groups) < 0.5   # groups that span 2^60; in the others no two amplitudes are more than 2 apart
    y /= np.abs(y)
    y[wide] *= np.exp2(rng.integers(-60, 0, (wide.sum(), 1 << k)))
    y[~wide] *= 1 + rng.random(((~wide).sum(), 1 << k))
    if not tiny:
        y[rng.random(y.shape) < 0.1] = 0  # exact zeros stay out of it
    y[7] = 0
    idx = np.arange(1 << n)
    low = idx[(idx & sum(1 << q for q in targets)) == 0]
    at = low[:, None] + np.array([sum(((s >> j) & 1) << q for j, q in enumerate(targets)) for s in range(1 << k)])
    x = np.zeros(1 << n, dtype=np.complex128)
    x[at] = y
    opts = qs.qs_default_opts()
    opts.tc_max_ctas = ctas
    got, recs, width = _run(n, gates, x, opts)
    assert [(q.k, q.tc) for q in recs] == [(k, 1)] and (not ctas or recs[0].tiles > 2 * recs[0].ctas)
    _, (mat,), _ = qs.qs_plan(n, gates, qs.QS_FUSE | qs.QS_FUSE_K(width))
    m = mat.astype(np.clongdouble)
    want = np.stack([(m * v).sum(1) for v in y.astype(np.clongdouble)])
    size = np.abs(y) @ np.abs(mat).T  # what an FP64 sum's error is relative to
    err = np.abs(got[at] - want).astype(np.float64)
    assert (err[wide] <= 2.0 ** (k + 1 - 53) * size[wide]).all()
    # digits: 2^-54 of the largest amplitude for each of the inputs of a result, and its rounding
    assert (err[~wide] <= (2.0 ** (k / 2 - 54) + 2.0 ** -53) * np.abs(y[~wide]).max(1, initial=0)[:, None] * 2).all()
    assert (got[at][7] == 0).all()


def test_the_other_precision_and_scarce_memory_take_the_fp64_kernel():
    n = 14
    gates = _gates([0, 2, 5, 9, 13], None, 8)
    rng = np.random.default_rng(4)
    x = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    opts = qs.qs_default_opts()
    opts.tc_precision = 1
    want, recs, _ = _run(n, gates, x, opts)
    assert [r.tc for r in recs] == [0]
    digits, recs, _ = _run(n, gates, x)
    assert [r.tc for r in recs] == [1]
    qs.qs_set_memory_limit(qs.qs_memory_in_use() + 40 * 1024)  # the matrix (16 KB), not its digits
    try:
        got, recs, _ = _run(n, gates, x)
    finally:
        qs.qs_set_memory_limit(0)
    assert [r.tc for r in recs] == [0] and np.array_equal(got, want)
    assert np.linalg.norm(digits - want) <= 4e-16 * np.linalg.norm(want)
