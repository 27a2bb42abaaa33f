"""Timed cases of the simulator core: what its users run, from one small circuit to 30 qubits.

Every case goes through the package's public calls. Circuits start from a
basis state and are applied to a state that lives in a torch tensor; their
results are the whole state (with the logical -> physical map), either left on
the device or read back in logical order. Batches, marginals and the
cost-model fit return all of what they compute.

`exact` computes the same results in 64 bits with plain torch / Python.
"""

import math
import random

import numpy as np
import torch

import paper_2410_09326_gb300 as qs


def listed():
    return [
        # the smallest call: a few gates on a small state, where launches and host work count
        {"name": "ghz_10", "kind": "circuit", "family": "ghz", "n": 10, "layers": 1, "swaps": 0, "dtype": "c64",
         "flags": "rules", "read": False},
        # a layered circuit with SWAPs on 12 qubits, the whole state read back in logical order
        {"name": "layered_12_read", "kind": "circuit", "family": "random", "n": 12, "layers": 20, "swaps": 10,
         "dtype": "c64", "flags": "rules", "read": True},
        # a 30-layer random circuit on a state that fits L2 (odd width)
        {"name": "random_19", "kind": "circuit", "family": "random", "n": 19, "layers": 30, "swaps": 20,
         "dtype": "c64", "flags": "rules", "read": False},
        # a QFT with its SWAP network, read back in logical order (the map is the bit reversal)
        {"name": "qft_21_read", "kind": "circuit", "family": "qft", "n": 21, "layers": 1, "swaps": 0, "dtype": "c64",
         "flags": "rules", "read": True},
        # plain per-gate application (no passes), as a baseline or for debugging
        {"name": "plain_23", "kind": "circuit", "family": "random", "n": 23, "layers": 6, "swaps": 6, "dtype": "c64",
         "flags": "plain", "read": False},
        # U3 + CX/CZ layers with the widest fused blocks on the tensor cores
        {"name": "u3_27_k6", "kind": "circuit", "family": "u3", "n": 27, "layers": 20, "swaps": 0, "dtype": "c64",
         "flags": "tc6", "read": False},
        # the benchmark's widest random circuit
        {"name": "random_30", "kind": "circuit", "family": "random", "n": 30, "layers": 30, "swaps": 71,
         "dtype": "c64", "flags": "rules", "read": False},
        # complex128 runs, as users take them where single precision is not enough
        {"name": "random_16_c128", "kind": "circuit", "family": "random", "n": 16, "layers": 20, "swaps": 10,
         "dtype": "c128", "flags": "rules", "read": False},
        {"name": "random_24_c128", "kind": "circuit", "family": "random", "n": 24, "layers": 10, "swaps": 8,
         "dtype": "c128", "flags": "rules", "read": False},
        # many QAOA circuits of uneven width in one batch, run again and again
        {"name": "qaoa_batch_192", "kind": "batch", "count": 192, "lo": 10, "hi": 20, "depth": 4},
        # the measured distribution of 16 qubits of a wide state
        {"name": "marginals_29", "kind": "marginals", "n": 29, "m": 16, "dtype": "c64"},
        # the cost model fitted to profiled blocks, then asked about all of them
        {"name": "fit_10000", "kind": "fit", "samples": 10000, "batch": 256, "epochs": 1},
    ]


def draw(rng):
    u = rng.random()
    if u < 0.55:
        family = rng.choice(["ghz", "random", "random", "qft", "u3"])
        n = rng.randint(8, 28)
        flags = rng.choice(["rules", "rules", "rules", "tc4", "tc6", "k3", "plain"])
        if flags == "plain":
            n = min(n, 26)
        layers = rng.randint(2, 30 if flags != "plain" else 6)
        return {"kind": "circuit", "family": family, "n": n, "layers": layers, "swaps": rng.randint(0, n),
                "dtype": "c64", "flags": flags, "read": n <= 22 and rng.random() < 0.4}
    if u < 0.70:
        family = rng.choice(["ghz", "random", "qft", "u3"])
        return {"kind": "circuit", "family": family, "n": rng.randint(8, 24), "layers": rng.randint(2, 10),
                "swaps": rng.randint(0, 10), "dtype": "c128", "flags": rng.choice(["rules", "rules", "k3", "plain"]),
                "read": False}
    if u < 0.82:
        lo = rng.randint(6, 14)
        return {"kind": "batch", "count": int(round(8 * 2 ** rng.uniform(0, 4.5))), "lo": lo,
                "hi": rng.randint(lo, 20), "depth": rng.randint(1, 4)}
    if u < 0.92:
        n = rng.randint(10, 29)
        return {"kind": "marginals", "n": n, "m": rng.randint(0, min(n, 20)),
                "dtype": rng.choice(["c64", "c64", "c128"])}
    # up to 40 updates: over more of them, a sample that rounding moves across a unit's threshold
    # often makes any two implementations differ by 1e-3
    batch, steps = rng.choice([32, 100, 256, 512]), 2 ** rng.uniform(0, 5.3)
    return {"kind": "fit", "samples": max(50, min(20000, int(batch * steps))), "batch": batch, "epochs": 1}


# ---------------------------------------------------------------------------
# Circuits: lists of (name, qubits, params)
# ---------------------------------------------------------------------------

def _matching(rng, n):
    q = list(range(n))
    rng.shuffle(q)
    return [(q[2 * i], q[2 * i + 1]) for i in range(n // 2)]


def _circuit(case, seed):
    """(index of the basis state the circuit starts from, gates)"""
    rng = random.Random(10007 * seed + 31 * case["n"] + 1)
    n, gates, start = case["n"], [], 0
    if case["family"] == "ghz":
        # H on one qubit, a CX chain over all of them in some order
        q = list(range(n))
        rng.shuffle(q)
        start = rng.getrandbits(n)
        gates = [("h", [q[0]], [])] + [("cx", [q[i], q[i + 1]], []) for i in range(n - 1)]
    elif case["family"] == "qft":
        start = rng.getrandbits(n)
        for j in range(n - 1, -1, -1):
            gates.append(("h", [j], []))
            gates += [("cp", [i, j], [math.pi / (1 << (j - i))]) for i in range(j - 1, -1, -1)]
        gates += [("swap", [i, n - 1 - i], []) for i in range(n // 2)]
    else:
        for _ in range(case["layers"]):
            for q in range(n):
                if case["family"] == "u3":
                    gates.append(("u3", [q], [rng.uniform(0, 2 * math.pi) for _ in range(3)]))
                else:
                    name = rng.choice(["h", "x", "rx", "ry", "rz"])
                    gates.append((name, [q], [rng.uniform(0, 2 * math.pi)] if name[0] == "r" else []))
            for a, b in _matching(rng, n):
                gates.append((rng.choice(["cx", "cz"]) if case["family"] == "u3" else "cx", [a, b], []))
    if case["family"] in ("random", "u3"):
        for _ in range(case["swaps"]):
            gates.insert(rng.randint(0, len(gates)), ("swap", rng.sample(range(n), 2), []))
    return start, gates


def _batch_circuits(case, seed):
    """QAOA Max-Cut ansaetze: H on all, then RZZ on the edges of a graph (a cycle through all nodes in
    some order and a matching: at most three edges a node) and RX on every qubit, once per layer."""
    rng = random.Random(7919 * seed + case["count"])
    sizes = random.Random(case["count"])
    out = []
    for _ in range(case["count"]):
        n, layers = sizes.randint(case["lo"], case["hi"]), sizes.randint(1, case["depth"])
        q = list(range(n))
        rng.shuffle(q)
        edges = {tuple(sorted((q[i], q[(i + 1) % n]))) for i in range(n)}
        edges |= {tuple(sorted(e)) for e in _matching(rng, n)}
        gates = [("h", [j], []) for j in range(n)]
        for _ in range(layers):
            gamma, beta = rng.uniform(0, math.pi), rng.uniform(0, math.pi)
            gates += [("rzz", list(e), [gamma]) for e in sorted(edges)]
            gates += [("rx", [j], [beta]) for j in range(n)]
        out.append((n, gates))
    return out


def _flags(name):
    if name == "rules":
        return qs.QS_PGO_RULES
    if name == "plain":
        return qs.QS_PLAIN
    base = qs.QS_VSWAP | qs.QS_FUSE | qs.QS_DIAG | qs.QS_FUSE_K(int(name[-1]))
    return base | (qs.QS_TC if name.startswith("tc") else 0)


def _dtype(case):
    return (qs.QS_C128, torch.complex128) if case["dtype"] == "c128" else (qs.QS_C64, torch.complex64)


class _State:
    """A state in a torch tensor, with its handle."""

    def __init__(self, amps, n, dtype):
        self.amps = amps
        self.handle = qs.qs_attach_state(amps.data_ptr(), n, dtype)

    def __del__(self):
        qs.qs_free_state(self.handle)


class _Batch:
    def __init__(self, states, arrays):
        self.states = states
        self.handle = qs.qs_batch_create([s.handle for s in states], arrays, qs.QS_DIAG)

    def __del__(self):
        if hasattr(self, "handle"):
            qs.qs_batch_free(self.handle)


def _random_state(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    real = torch.float64 if case["dtype"] == "c128" else torch.float32
    x = torch.randn(1 << case["n"], 2, device="cuda", dtype=real, generator=g)
    return torch.view_as_complex(x.mul_(2 ** (-(case["n"] + 1) / 2)))


def _measured(case, seed):
    return random.Random(seed).sample(range(case["n"]), case["m"])


def _fit_data(case, seed):
    """Feature rows like those of profiled blocks (fractions and flags), times that depend on them, and
    the weights the fit starts from."""
    g = np.random.default_rng(seed + 5)
    s, f, h = case["samples"], qs.QS_MLP_FEATURES, qs.QS_MLP_HIDDEN
    x = g.random((s, f))
    x[:, 3:8] = x[:, 3:8] < 0.4
    x[:, 14:] = x[:, 14:] < 0.3
    x[:, 5] = 0.0
    w = g.standard_normal((f, 8))
    y = np.tanh(x @ w) @ g.standard_normal(8) + 0.1 * g.standard_normal(s)
    p = np.zeros(qs.QS_MLP_PARAMS)
    o = 0
    for fan_out, fan_in in ((h, f), (h, h), (1, h)):
        lim = math.sqrt(6.0 / fan_in)
        p[o: o + fan_out * fan_in] = g.uniform(-lim, lim, fan_out * fan_in)
        o += fan_out * fan_in + fan_out
    return x.astype(np.float32), y.astype(np.float32), p.astype(np.float32)


LEARNING_RATE = 2e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        dtype, td = _dtype(case)
        start, gates = _circuit(case, seed)
        st = _State(torch.zeros(1 << case["n"], device="cuda", dtype=td), case["n"], dtype)
        return {"case": case, "state": st, "start": start, "gates": qs.gates_to_array(gates), "dtype": dtype,
                "flags": _flags(case["flags"])}
    if kind == "batch":
        circuits = _batch_circuits(case, seed)
        amps = torch.zeros(sum(1 << n for n, _ in circuits), device="cuda", dtype=torch.complex64)
        states, at = [], 0
        for n, _ in circuits:
            states.append(_State(amps[at: at + (1 << n)], n, qs.QS_C64))
            at += 1 << n
        return {"case": case, "amps": amps, "batch": _Batch(states, [qs.gates_to_array(g) for _, g in circuits])}
    if kind == "marginals":
        dtype, _ = _dtype(case)
        return {"case": case, "state": _State(_random_state(case, seed), case["n"], dtype),
                "qubits": _measured(case, seed)}
    x, y, p = _fit_data(case, seed)
    return {"case": case, "x": x, "y": y, "p": p, "seed": seed}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "circuit":
        st = state["state"]
        qs.qs_set_basis(st.handle, state["start"])
        qs.qs_apply_circuit(st.handle, state["gates"], state["flags"])
        if case["read"]:
            return {"amps": qs.qs_read_state(st.handle, case["n"], state["dtype"], logical_order=True)}
        return {"amps": st.amps, "perm": qs.qs_get_perm(st.handle, case["n"])}
    if kind == "batch":
        qs.qs_batch_run(state["batch"].handle)
        return {"amps": state["amps"]}
    if kind == "marginals":
        return {"probs": qs.qs_measure_probs(state["state"].handle, state["qubits"])}
    m = qs.qs_mlp_create(0)
    qs.qs_mlp_params(m, state["p"])
    loss = qs.qs_mlp_train(m, state["x"], state["y"], epochs=case["epochs"], batch=case["batch"], lr=LEARNING_RATE,
                           seed=state["seed"])
    out = {"loss": loss, "params": qs.qs_mlp_params(m), "times": qs.qs_mlp_predict(m, state["x"])}
    qs.qs_mlp_free(m)
    return out


def _gate_flops(n, gates):
    """Real operations of the gates as they are defined, on 2^n amplitudes."""
    per = {"h": 4, "x": 0, "rx": 6, "ry": 6, "rz": 6, "u3": 14, "cx": 0, "cz": 0.5, "cp": 1.5, "swap": 0, "rzz": 6}
    return sum(per[g[0]] for g in gates) * 2.0 ** n


def work(case):
    kind = case["kind"]
    if kind == "circuit":
        # the state is written once (and read back once where it is read)
        amp = 16 if case["dtype"] == "c128" else 8
        return {"bytes": (2 if case["read"] else 1) * amp * 2 ** case["n"],
                "flops": _gate_flops(case["n"], _circuit(case, 0)[1])}
    if kind == "batch":
        circuits = _batch_circuits(case, 0)
        return {"bytes": sum(8 * 2 ** n for n, _ in circuits), "flops": sum(_gate_flops(n, g) for n, g in circuits)}
    if kind == "marginals":
        return {"bytes": (16 if case["dtype"] == "c128" else 8) * 2 ** case["n"] + 8 * 2 ** case["m"],
                "flops": 4 * 2 ** case["n"]}
    f, h, s = qs.QS_MLP_FEATURES, qs.QS_MLP_HIDDEN, case["samples"]
    layer = 2 * (f * h + h * h + h)
    return {"bytes": 4 * s * (f + 2), "flops": s * layer * (3 * case["epochs"] + 1)}


def tolerance(case):
    """About four times the distance from the 64-bit results, as measured on a GB300: circuits up to
    2.7e-6 (complex64) and 1.1e-14 (complex128), batches 2.8e-7, marginals up to 3e-8 where a bin sums few
    squares, fits up to 8e-4 (mostly 3e-7; more where a sample crosses a unit's threshold)."""
    kind = case["kind"]
    if kind == "circuit":
        return {"rel": 5e-14} if case["dtype"] == "c128" else {"rel": 1e-5}
    if kind == "batch":
        return {"rel": 2e-6}
    if kind == "marginals":
        return {"rel": 1e-7} if case["dtype"] == "c64" else {"rel": 1e-14}
    return {"rel": 3e-3}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _matrix(name, p):
    c, s = (math.cos(p[0] / 2), math.sin(p[0] / 2)) if p else (0, 0)
    if name == "h":
        r = math.sqrt(0.5)
        return [[r, r], [r, -r]]
    if name == "x":
        return [[0, 1], [1, 0]]
    if name == "rx":
        return [[c, -1j * s], [-1j * s, c]]
    if name == "ry":
        return [[c, -s], [s, c]]
    e = lambda a: complex(math.cos(a), math.sin(a))  # noqa: E731
    return [[c, -e(p[2]) * s], [e(p[1]) * s, e(p[1] + p[2]) * c]]  # u3


def _simulate(n, start, gates, device, virtual=True):
    """Amplitudes in physical order and the map: SWAPs relabel (virtual) or move data."""
    a = torch.zeros(1 << n, dtype=torch.complex128, device=device)
    a[start] = 1
    perm = list(range(n))
    for name, q, p in gates:
        if name == "swap" and virtual:
            perm[q[0]], perm[q[1]] = perm[q[1]], perm[q[0]]
            continue
        q = [perm[i] for i in q]
        if len(q) == 1:
            v = a.view(-1, 2, 1 << q[0])
            if name == "rz":
                z = complex(math.cos(p[0] / 2), math.sin(p[0] / 2))
                v[:, 0] *= z.conjugate()
                v[:, 1] *= z
                continue
            m = _matrix(name, p)
            lo, hi = v[:, 0].clone(), v[:, 1].clone()
            v[:, 0] = m[0][0] * lo + m[0][1] * hi
            v[:, 1] = m[1][0] * lo + m[1][1] * hi
            continue
        x, y = max(q), min(q)
        v = a.view(-1, 2, 1 << (x - y - 1), 2, 1 << y)
        at = lambda i, j: v[:, i, :, j] if q[0] == x else v[:, j, :, i]  # noqa: E731  (bits of q[0], q[1])
        if name in ("cx", "swap"):
            i, j = ((1, 0), (1, 1)) if name == "cx" else ((0, 1), (1, 0))
            t = at(*i).clone()
            at(*i).copy_(at(*j))
            at(*j).copy_(t)
        elif name == "rzz":
            z = complex(math.cos(p[0] / 2), math.sin(p[0] / 2))
            for i in (0, 1):
                for j in (0, 1):
                    at(i, j).mul_(z if i != j else z.conjugate())
        else:  # cz, cp
            z = -1.0 if name == "cz" else complex(math.cos(p[0]), math.sin(p[0]))
            at(1, 1).mul_(z)
    return a, perm


def _shuffled_epochs(seed, s, epochs):
    """The sample order of each epoch: a Fisher-Yates shuffle as the C++ standard library of the build
    does it from a 64-bit Mersenne twister (Matsumoto and Nishimura), two positions to a draw, each draw
    reduced to its range by a multiplication (Lemire)."""
    mask = (1 << 64) - 1
    mt = [seed & mask]
    for i in range(1, 312):
        mt.append((6364136223846793005 * (mt[-1] ^ (mt[-1] >> 62)) + i) & mask)
    state = {"at": 312}

    def word():
        if state["at"] == 312:
            for i in range(312):
                x = (mt[i] & ~0x7FFFFFFF & mask) | (mt[(i + 1) % 312] & 0x7FFFFFFF)
                mt[i] = mt[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
            state["at"] = 0
        x = mt[state["at"]]
        state["at"] += 1
        x ^= (x >> 29) & 0x5555555555555555
        x ^= (x << 17) & 0x71D67FFFEDA60000
        x ^= (x << 37) & 0xFFF7EEE000000000
        return x ^ (x >> 43)

    def below(r):
        p = word() * r
        if (p & mask) < r:
            floor = ((1 << 64) - r) % r
            while (p & mask) < floor:
                p = word() * r
        return p >> 64

    order = list(range(s))
    for _ in range(epochs):
        i = 1
        if s % 2 == 0:
            j = below(2)
            order[1], order[j] = order[j], order[1]
            i = 2
        while i < s:
            x, y = divmod(below((i + 1) * (i + 2)), i + 2)
            order[i], order[x] = order[x], order[i]
            order[i + 1], order[y] = order[y], order[i + 1]
            i += 2
        yield np.array(order)


def _exact_fit(case, seed):
    x, y, p = (torch.from_numpy(v.astype(np.float64)) for v in _fit_data(case, seed))
    f, h, s = qs.QS_MLP_FEATURES, qs.QS_MLP_HIDDEN, case["samples"]
    mean, std = x.mean(0), x.std(0, unbiased=False)
    std = torch.where(std > 1e-6, std, torch.ones_like(std))
    xs, ym, ysd = (x - mean) / std, y.mean(), y.std(unbiased=False)
    ys = (y - ym) / ysd
    p = p.clone().requires_grad_(True)

    def forward(v):
        o = 0
        for out, inp, last in ((h, f, False), (h, h, False), (1, h, True)):
            w = p[o: o + out * inp].view(out, inp)
            v = v @ w.t() + p[o + out * inp: o + out * inp + out]
            v = v if last else v.clamp(min=0)
            o += out * inp + out
        return v[:, 0]

    m, v, step, loss = torch.zeros_like(p), torch.zeros_like(p), 0, None
    b = min(case["batch"], s)
    for order in _shuffled_epochs(seed, s, case["epochs"]):
        for at in range(0, s - b + 1, b):
            rows = torch.from_numpy(order[at: at + b])
            loss = ((forward(xs[rows]) - ys[rows]) ** 2).mean()
            g, = torch.autograd.grad(loss, p)
            step += 1
            with torch.no_grad():
                m = 0.9 * m + 0.1 * g
                v = 0.999 * v + 0.001 * g * g
                p -= LEARNING_RATE * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
    with torch.no_grad():
        return {"loss": float(loss), "params": p.detach().numpy(), "times": (forward(xs) * ysd + ym).numpy()}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "circuit":
        n = case["n"]
        start, gates = _circuit(case, seed)
        if len(gates) * 2.0 ** n > 1500 * 2.0 ** 28:
            return None  # takes too long
        a, perm = _simulate(n, start, gates, device, virtual=case["flags"] != "plain")
        if case["read"]:
            return {"amps": a.view([2] * n).permute([n - 1 - perm[n - 1 - i] for i in range(n)]).reshape(-1)}
        return {"amps": a, "perm": np.array(perm, dtype=np.int64)}
    if kind == "batch":
        return {"amps": torch.cat([_simulate(n, 0, g, device)[0] for n, g in _batch_circuits(case, seed)])}
    if kind == "marginals":
        n, q = case["n"], _measured(case, seed)
        w = torch.view_as_real(_random_state(case, seed)).double().square_().sum(1)
        for i in range(n - 1, -1, -1):
            if i not in q:
                w = w.view(-1, 2, 1 << i).sum(1)
        # the kept bits in ascending order; bit j of a bin is qubit q[j]
        up, m = sorted(q), len(q)
        w = w.view([2] * m).permute([m - 1 - up.index(i) for i in reversed(q)]) if m else w
        return {"probs": w.reshape(-1).cpu().numpy()}
    return _exact_fit(case, seed)
