"""Batched circuits whose diagonal gates merge into runs in every way: gates of all kinds in random
order, several RZ on one qubit, parameters shared by gates of one run and of one stage, Z and CZ on
register, lane and warp bits, widths on both sides of the 13-qubit window, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def random_circuit(n, count, seed, shared):
    rng = W.SplitMix64(seed)
    gates, p = [], 0
    for _ in range(count):
        kind = ("RX", "RY", "RZ", "RZ", "RZ", "CZ", "CZ", "CNOT", "H", "X", "Y", "Z")[rng.randint(0, 11)]
        a = rng.randint(0, n - 1)
        b = (a + rng.randint(1, n - 1)) % n
        if kind in ("RX", "RY", "RZ"):
            th = rng.uniform_range(-3.0, 3.0)
            if rng.randint(0, 4) == 0:
                gates.append(W.Gate(kind, (a,), params=(th,)))
            else:
                gates.append(W.Gate(kind, (a,), params=(th,), param_index=p))
                p += 1
        elif kind == "CZ":
            gates.append(W.Gate("CZ", (a, b)))
        elif kind == "CNOT":
            gates.append(W.Gate("CNOT", (a,), controls=(b,), control_values=(1,)))
        else:
            gates.append(W.Gate(kind, (a,)))
    if shared and p > 3:  # three parameters drive all rotations
        th = [rng.uniform_range(-3.0, 3.0) for _ in range(3)]
        gates = [g if g.param_index < 0 else
                 W.Gate(g.name, g.targets, params=(th[g.param_index % 3],), param_index=g.param_index % 3) for g in gates]
        p = 3
    return W.Circuit(n, gates, n_params=p)


def diagonal_layers(n, seed):
    """RZ twice on every qubit and long-range CZ around one layer of RX: runs that fill every bit."""
    rng = W.SplitMix64(seed)
    gates, p = [W.Gate("H", (q,)) for q in range(n)], 0
    for _ in range(2):
        for q in range(n):
            for _ in range(2):
                gates.append(W.Gate("RZ", (q,), params=(rng.uniform_range(-3.0, 3.0),), param_index=p))
                p += 1
        gates += [W.Gate("CZ", (q, r)) for q in range(n) for r in range(q + 1, n) if (q * r + q) % 3 == 0]
        gates += [W.Gate("Z", (q,)) for q in range(0, n, 2)]
        for q in range(n):
            gates.append(W.Gate("RX", (q,), params=(rng.uniform_range(-3.0, 3.0),), param_index=p))
            p += 1
    return W.Circuit(n, gates, n_params=p)


def check(circuits, seed):
    import paper_2011_13524_gb300 as qs
    obs = [W.random_pauli_observable(c.n, 4, seed + i) for i, c in enumerate(circuits)]
    b = qs.Batch(circuits, obs)
    theta = np.concatenate([c.parameters() for c in circuits])
    for use_graph in (True, False):
        e, g = b.run(theta, use_graph=use_graph)
        for c, o, ek, gk in zip(circuits, obs, e, g):
            scale = float(np.abs(o.coef).sum())
            # complex64: 2^-23 per gate on amplitudes of norm 1, at most 200 gates
            assert abs(ek - oracle.energy(c, o)) < 3e-5 * max(scale, 1.0), c.n
            idx = range(c.n_params) if c.n < 13 else range(0, c.n_params, max(1, c.n_params // 5))
            ps = gradient(c, o, idx)
            assert float(np.max(np.abs(gk[list(idx)] - ps))) < 1e-4 * max(scale, 1.0), c.n


def gradient(c, o, idx):
    """Central differences in 64 bits (a shared parameter shifts all of its gates): error about 1e-9."""
    base = c.parameters()
    out = []
    for i in idx:
        d = np.zeros(c.n_params)
        d[i] = 1e-5
        out.append((oracle.energy(c.bind(base + d), o) - oracle.energy(c.bind(base - d), o)) / 2e-5)
    return np.array(out)


@pytest.mark.parametrize("shared", [False, True])
def test_random_gate_orders(shared):
    check([random_circuit(n, 60, 7 * n + i, shared) for n in (4, 5, 6, 8, 9, 10) for i in range(2)], 40)


def test_window_edge_and_beyond():
    check([random_circuit(n, 50, n, False) for n in (11, 12, 13, 14, 15)], 50)


@pytest.mark.parametrize("n", [4, 6, 9, 12, 14])
def test_full_diagonal_layers(n):
    check([diagonal_layers(n, n)], 60)
