"""The simulator's work as its users call it: circuits, gates, energies, overlaps, measurement, time
evolution, gradients and batches, over the sizes of the configured workloads (n = 4 .. 30 qubits,
complex128 and complex64).

A case is a dict of plain values; ``prepare`` makes what a program holds before the call, ``run`` is
one pass through the public entry points, ``exact`` is the same in plain 64-bit torch arithmetic.
"""
import math
import random

import numpy as np
import torch

import paper_2011_13524_gb300 as qs
import workloads as W


def listed():
    return [
        # The smallest circuit run: 12 qubits, depth 10, gate by gate (the default of State.run), then
        # <Z0 Z1>. Launches and host work count.
        {"name": "run_n12_c128", "kind": "run", "n": 12, "depth": 10, "k": 0, "dtype": "c128"},
        # The headline run: 30 qubits (16 GiB), depth 20, fused into 5-qubit blocks, then <Z0 Z1>.
        {"name": "run_n30_c128_fused", "kind": "run", "n": 30, "depth": 20, "k": 5, "dtype": "c128"},
        # The same family as a complex64 state vector in 6-qubit blocks (the precision workload).
        {"name": "run_n28_c64_fused", "kind": "run", "n": 28, "depth": 20, "k": 6, "dtype": "c64"},
        # A program that applies gates one call at a time: every gate kind once, low, high and
        # scattered targets, controls, diagonals, Pauli strings and rotations.
        {"name": "gates_n25_c128", "kind": "gates", "n": 25, "dtype": "c128"},
        # The transverse-field Ising energy of a 28-qubit state: 31 flip groups' worth of terms.
        {"name": "energy_tfim_n28_c128", "kind": "energy", "n": 28, "obs": "tfim", "terms": 0, "dtype": "c128"},
        # A general observable (random Pauli strings over all qubits) on an odd-sized complex64 state.
        {"name": "energy_pauli_n23_c64", "kind": "energy", "n": 23, "obs": "pauli", "terms": 24, "dtype": "c64"},
        # Two states compared: <a|H|b>, <a|b> and the norms.
        {"name": "overlap_tfim_n26_c128", "kind": "overlap", "n": 26, "dtype": "c128"},
        # Measurement of a 28-qubit state: 100 000 shots and a marginal probability.
        {"name": "measure_n28_c128", "kind": "measure", "n": 28, "shots": 100000, "dtype": "c128"},
        # Time evolution under the Ising chain, first-order Trotter.
        {"name": "trotter_tfim_n26_c128", "kind": "trotter", "n": 26, "slices": 2, "dtype": "c128"},
        # Energy and full gradient of a 20-qubit, 20-layer ansatz (800 parameters).
        {"name": "grad_n20_c128", "kind": "grad", "n": 20, "layers": 20, "dtype": "c128"},
        # A small variational step in complex64: latency of one gradient call.
        {"name": "grad_n11_c64", "kind": "grad", "n": 11, "layers": 5, "dtype": "c64"},
        # Many small variational circuits of uneven width and depth, energies and gradients.
        {"name": "batch_512", "kind": "batch", "count": 512, "n_lo": 8, "n_hi": 20, "l_lo": 2, "l_hi": 12},
    ]


def draw(rng: random.Random):
    dtype = rng.choice(["c128", "c64"])
    kind = rng.choice(["run", "run", "gates", "energy", "energy", "overlap", "measure", "trotter", "grad", "grad", "batch"])
    if kind == "run":
        k = rng.choice([0, 0, 2, 3, 4, 5, 5] if dtype == "c128" else [0, 0, 3, 4, 5, 6, 6])
        n = rng.randint(6, 24 if k == 0 else 25 if k < 4 else 28)
        return {"kind": kind, "n": n, "depth": rng.randint(3, 20), "k": k, "dtype": dtype}
    if kind == "gates":
        return {"kind": kind, "n": rng.randint(6, 25), "dtype": dtype}
    if kind == "energy":
        obs = rng.choice(["tfim", "pauli"])
        return {"kind": kind, "n": rng.randint(8, 28 if obs == "tfim" else 25), "obs": obs,
                "terms": 0 if obs == "tfim" else rng.randint(1, 32), "dtype": dtype}
    if kind == "overlap":
        return {"kind": kind, "n": rng.randint(8, 26), "dtype": dtype}
    if kind == "measure":
        return {"kind": kind, "n": rng.randint(8, 28), "shots": int(10 ** rng.uniform(1.0, 5.0)), "dtype": dtype}
    if kind == "trotter":
        return {"kind": kind, "n": rng.randint(6, 25), "slices": rng.randint(1, 3), "dtype": dtype}
    if kind == "grad":
        return {"kind": kind, "n": rng.randint(5, 20), "layers": rng.randint(2, 20), "dtype": dtype}
    n_lo = rng.randint(4, 10)
    n_hi = rng.randint(n_lo + 2, 20)
    count = int(2 ** rng.uniform(2.0, 9.0 if n_hi < 19 else 8.0))
    return {"kind": kind, "count": count, "n_lo": n_lo, "n_hi": n_hi, "l_lo": 2, "l_hi": rng.randint(3, 12)}


# ------------------------------------------------------------------ the calls
def _types(case):
    return (qs.QS_C64, torch.complex64) if case["dtype"] == "c64" else (qs.QS_C128, torch.complex128)


def _random_tensor(n, dtype, seed):
    """A normalised Gaussian random state on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    v = torch.randn(2 << n, dtype=real, device="cuda", generator=g)
    v /= torch.linalg.vector_norm(v.view(1 << max(0, n - 15), -1), dim=1, dtype=torch.float64).norm().item()
    return torch.view_as_complex(v.view(-1, 2))


def _z0z1(n):
    return W.PauliObservable(n, np.array([1.0]), np.array([0], dtype=np.uint64), np.array([3], dtype=np.uint64))


def _observable(case, seed):
    if case.get("obs", "tfim") == "tfim":
        return W.tfim_observable(case["n"], 1.0)
    return W.random_pauli_observable(case["n"], case["terms"], seed + 7)


def _gate_list(case, seed):
    """Every gate kind at seeded placements, and the string of one long Pauli rotation."""
    n = case["n"]
    rng = W.SplitMix64(seed + 11)
    ids = [rng.randint(0, 3) for _ in range(n)]
    x, z = W.pauli_masks(ids, range(n))
    return W.random_gate_suite(n, seed), (x, z, rng.uniform_range(-3.0, 3.0))


def _uniforms(case, seed):
    return np.random.Generator(np.random.PCG64(seed + 3)).random(case["shots"])


def _measured(case, seed):
    """A marginal over about half of the qubits."""
    rng = W.SplitMix64(seed + 5)
    n = case["n"]
    return [2 if q % 2 else (rng.randint(0, 1) if q < 8 else 2) for q in range(n)]


def _batch_items(case, seed):
    """Ansatz circuits of the widths and depths that the case fixes; angles and observables by seed."""
    shape = W.SplitMix64(case["count"] * 1000 + case["n_hi"])
    items = []
    for i in range(case["count"]):
        n, layers = shape.randint(case["n_lo"], case["n_hi"]), shape.randint(case["l_lo"], case["l_hi"])
        items.append(W.BatchItem(W.hea_circuit(n, layers, seed * 100003 + i),
                                 W.random_pauli_observable(n, 4, seed * 100003 + i + 50021)))
    return items


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "batch":
        items = _batch_items(case, seed)
        s["batch"] = qs.Batch([i.circuit for i in items], [i.observable for i in items])
        s["theta"] = np.concatenate([i.circuit.parameters() for i in items])
        return s
    dt, tdt = _types(case)
    n = case["n"]
    if kind == "grad":
        s["circuit"] = W.hea_circuit(n, case["layers"], seed)
        s["obs"] = W.tfim_observable(n, 1.0)
        s["theta"] = s["circuit"].parameters()
        s["dtype"] = dt
        return s
    if kind == "run":
        s["circuit"] = W.u3cz_circuit(n, case["depth"], seed)
        s["obs"] = _z0z1(n)
        s["state"] = qs.State(n, dt)
        return s
    s["state"] = qs.State(n, dt, tensor=_random_tensor(n, tdt, seed))
    if kind == "gates":
        s["gates"], s["rotation"] = _gate_list(case, seed)
    elif kind == "energy":
        s["obs"] = _observable(case, seed)
    elif kind == "overlap":
        s["other"] = qs.State(n, dt, tensor=_random_tensor(n, tdt, seed + 1000003))
        s["obs"] = _observable(case, seed)
    elif kind == "measure":
        s["uniforms"] = _uniforms(case, seed)
        s["measured"] = _measured(case, seed)
    elif kind == "trotter":
        s["obs"] = _observable(case, seed)
    return s


#: evolution time of the Trotter case
TIME = 0.3


def run(s):
    kind = s["kind"]
    if kind == "batch":
        e, g = s["batch"].run(s["theta"])
        return {"energies": e, "gradients": np.concatenate(g)}
    if kind == "grad":
        e, g = qs.adjoint_grad(s["circuit"], s["obs"], s["theta"], s["dtype"])
        return {"energy": np.float64(e), "gradient": g}
    st = s["state"]
    if kind == "run":
        st.set_basis(0)
        st.run(s["circuit"], s["case"]["k"])
        return {"state": st.tensor, "energy": np.float64(st.expectation(s["obs"])[0])}
    if kind == "gates":
        for g in s["gates"]:
            st.apply_gate(g)
        st.apply_pauli_rotation(*s["rotation"])
        return {"state": st.tensor}
    if kind == "energy":
        return {"energy": np.float64(st.expectation(s["obs"])[0])}
    if kind == "overlap":
        t = st.transition_amplitude(s["obs"], s["other"])
        i = st.inner(s["other"])
        return {"transition": np.array([t.real, t.imag]), "inner": np.array([i.real, i.imag]),
                "norms": np.array([st.norm2(), s["other"].norm2()])}
    if kind == "measure":
        return {"samples": st.sample(s["uniforms"]).astype(np.int64), "marginal": np.float64(st.marginal_probability(s["measured"]))}
    st.apply_observable_rotation(s["obs"], TIME, s["case"]["slices"])
    return {"state": st.tensor}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "batch":
        layers = 0.5 * (case["l_lo"] + case["l_hi"])
        flops = byts = 0.0
        widths = range(case["n_lo"], case["n_hi"] + 1)
        for n in widths:
            share = case["count"] / len(widths)
            # per layer and qubit RY on psi (forward, reverse) and lambda with the gradient products,
            # and one diagonal update of each
            flops += share * layers * 2.0 ** n * (n * (3 * 6.0 + 4.0) + 3 * 6.0 + 4.0)
            byts += share * 16.0 * 2 * n * layers
        return {"bytes": byts, "flops": flops}
    n = case["n"]
    amp = 8 if case["dtype"] == "c64" else 16
    size = 2.0 ** n
    if kind == "grad":
        layers = case["layers"]
        return {"bytes": 16.0 * 2 * n * layers, "flops": layers * size * (n * 22.0 + 22.0)}
    if kind == "run":
        u3 = case["depth"] * n
        return {"bytes": 2 * amp * size, "flops": 14.0 * u3 * size}
    if kind == "gates":
        # one call, one pass: 12 named and 6 parametrised one-qubit gates, dense 1..6, diagonals,
        # Pauli strings and rotations read and write the state; controls halve what a gate touches
        return {"bytes": 38 * 2 * amp * size, "flops": size * (18 * 14.0 + sum(8.0 * 2 ** m for m in range(1, 7)))}
    if kind == "energy":
        groups = n + 1 if case["obs"] == "tfim" else case["terms"]
        return {"bytes": amp * size, "flops": 4.0 * groups * size}
    if kind == "overlap":
        return {"bytes": 2 * amp * size, "flops": 8.0 * (n + 2) * size}
    if kind == "measure":
        return {"bytes": amp * size + 16.0 * case["shots"], "flops": 4.0 * size}
    # every slice: one diagonal factor and n rotations about X
    return {"bytes": 2 * amp * size, "flops": case["slices"] * size * (6.0 + 8.0 * n)}


# ------------------------------------------------------------------ the same in plain 64-bit torch
_PAULI = {0: np.eye(2), 1: np.array([[0, 1], [1, 0]]), 2: np.array([[0, -1j], [1j, 0]]), 3: np.diag([1, -1])}


def _kron(ms):
    """Operator on targets[0] (lowest bit), targets[1], ..."""
    out = np.eye(1)
    for m in ms:
        out = np.kron(m, out)
    return out


def _matrix(g):
    """2^m x 2^m matrix of a gate on its targets (rotations exp(+i theta P / 2), U3 as OpenQASM 2)."""
    n, p = g.name, g.params
    h = math.sqrt(0.5)
    if n in ("X", "CNOT", "TOFFOLI"):
        return _PAULI[1]
    if n == "Y":
        return _PAULI[2]
    if n == "Z":
        return _PAULI[3]
    if n == "H":
        return h * np.array([[1, 1], [1, -1]])
    if n in ("S", "Sdag", "T", "Tdag"):
        ph = np.exp((1j if "dag" not in n else -1j) * (math.pi / 2 if n[0] == "S" else math.pi / 4))
        return np.diag([1, ph])
    if n in ("sqrtX", "sqrtXdag", "sqrtY", "sqrtYdag"):
        m = 0.5 * ((1 + 1j) * np.eye(2) + (1 - 1j) * (_PAULI[1] if n[4] == "X" else _PAULI[2]))
        return m.conj().T if n.endswith("dag") else m
    if n in ("RX", "RY", "RZ"):
        P = _PAULI["XYZ".index(n[1]) + 1]
        return math.cos(p[0] / 2) * np.eye(2) + 1j * math.sin(p[0] / 2) * P
    if n == "U1":
        return np.diag([1, np.exp(1j * p[0])])
    if n in ("U2", "U3"):
        th, ph, la = (math.pi / 2, p[0], p[1]) if n == "U2" else p
        c, s = math.cos(th / 2), math.sin(th / 2)
        return np.array([[c, -np.exp(1j * la) * s], [np.exp(1j * ph) * s, np.exp(1j * (ph + la)) * c]])
    if n == "CZ":
        return np.diag([1, 1, 1, -1])
    if n in ("SWAP", "FREDKIN"):
        return np.array([[1, 0, 0, 0], [0, 0, 1, 0], [0, 1, 0, 0], [0, 0, 0, 1]])
    if n == "DENSE":
        return g.matrix
    if n == "DIAG":
        return np.diag(g.matrix)
    P = _kron([_PAULI[i] for i in g.pauli])
    if n == "PAULI":
        return P
    return math.cos(p[0] / 2) * np.eye(len(P)) + 1j * math.sin(p[0] / 2) * P


def _apply(psi, n, g):
    """psi <- g psi in place (complex128 tensor of 2^n)."""
    qubits = sorted(set(g.targets) | set(g.controls), reverse=True)
    shape, axis, top = [], {}, n
    for q in qubits:
        if top - 1 - q:
            shape.append(1 << (top - 1 - q))
        axis[q] = len(shape)
        shape.append(2)
        top = q
    if top:
        shape.append(1 << top)
    v = psi.view(shape)
    vals = tuple(g.control_values) if g.control_values else (1,) * len(g.controls)
    for q, val in zip(g.controls, vals):
        v = v.narrow(axis[q], int(val), 1)
    m = len(g.targets)
    order = [axis[t] for t in reversed(g.targets)]
    w = v.movedim(order, list(range(m)))
    mat = torch.as_tensor(np.ascontiguousarray(_matrix(g), dtype=np.complex128), device=psi.device)
    new = (mat @ w.reshape(1 << m, -1)).view(w.shape)
    w.copy_(new)


def _parity(x):
    for k in (32, 16, 8, 4, 2, 1):
        x = x ^ (x >> k)
    return x & 1


def _pauli_on(psi, x, z):
    """P psi for the string i^{#Y} X^x Z^z."""
    y = torch.arange(psi.numel(), device=psi.device) ^ int(x)
    out = psi[y]
    if int(z):
        out = out * (1 - 2 * _parity(y & int(z)))
    return out * (1j ** (bin(int(x) & int(z)).count("1") % 4))


def _pauli_sum(psi, obs, bra=None):
    """<bra|H|psi>"""
    total = 0j
    bra = psi if bra is None else bra
    for c, x, z in zip(obs.coef, obs.x_mask, obs.z_mask):
        total += float(c) * torch.vdot(bra, _pauli_on(psi, x, z)).item()
    return total


def _hea_exact(circuits, observables):
    """Energies and gradients of HEA circuits of one width (RY, RZ on every qubit, CZ ladder),
    batched; a circuit with fewer layers passes the later ones unchanged."""
    n, B, dev = circuits[0].n, len(circuits), "cuda"
    per = 2 * n
    layers = [c.n_params // per for c in circuits]
    L = max(layers)
    th = torch.zeros(B, L, 2, n, dtype=torch.float64)
    live = torch.zeros(B, L, dtype=torch.float64)
    for b, c in enumerate(circuits):
        p = torch.as_tensor(c.parameters()).view(layers[b], 2, n)
        th[b, :layers[b]] = p
        live[b, :layers[b]] = 1.0
    th, live = th.to(dev), live.to(dev)
    idx = torch.arange(1 << n, device=dev)
    ladder = 1.0 - 2.0 * _parity(idx & (idx >> 1)).to(torch.float64)
    psi = torch.zeros(B, 1 << n, dtype=torch.complex128, device=dev)
    psi[:, 0] = 1.0

    def ry(v, q, t):
        w = v.view(B, -1, 2, 1 << q)
        c, s = torch.cos(t / 2).view(B, 1, 1), torch.sin(t / 2).view(B, 1, 1)
        a, b = w[:, :, 0].clone(), w[:, :, 1].clone()
        w[:, :, 0] = c * a + s * b
        w[:, :, 1] = c * b - s * a

    def diag(v, layer, sign):
        ph = torch.zeros(B, 1 << n, dtype=torch.float64, device=dev)
        for q in range(n):
            w = ph.view(B, -1, 2, 1 << q)
            t = 0.5 * sign * th[:, layer, 1, q].view(B, 1, 1)
            w[:, :, 0] += t
            w[:, :, 1] -= t
        on = live[:, layer].view(B, 1)
        v *= torch.polar((ladder * on + (1.0 - on)).abs(), ph) * (ladder * on + (1.0 - on))

    for layer in range(L):
        for q in range(n):
            ry(psi, q, th[:, layer, 0, q])
        diag(psi, layer, 1.0)
    lam = torch.zeros_like(psi)
    for b, o in enumerate(observables):
        for c, x, z in zip(o.coef, o.x_mask, o.z_mask):
            lam[b] += float(c) * _pauli_on(psi[b], x, z)
    energy = torch.stack([torch.vdot(psi[b], lam[b]).real for b in range(B)])
    grad = torch.zeros(B, L, 2, n, dtype=torch.float64, device=dev)
    for layer in reversed(range(L)):
        w = (lam.conj() * psi).imag
        for q in range(n):
            s = w.view(B, -1, 2, 1 << q).sum(dim=(1, 3))
            grad[:, layer, 1, q] = -(s[:, 0] - s[:, 1])
        diag(psi, layer, -1.0)
        diag(lam, layer, -1.0)
        for q in range(n):
            p, m = psi.view(B, -1, 2, 1 << q), lam.view(B, -1, 2, 1 << q)
            y = (m[:, :, 1].conj() * p[:, :, 0] - m[:, :, 0].conj() * p[:, :, 1]).real  # Im <m|Y|p>
            grad[:, layer, 0, q] = -y.sum(dim=(1, 2))
            ry(psi, q, -th[:, layer, 0, q])
            ry(lam, q, -th[:, layer, 0, q])
    out = [grad[b, :layers[b]].reshape(-1).cpu().numpy() for b in range(B)]
    return energy.cpu().numpy(), out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        items = _batch_items(case, seed)
        e, g = np.zeros(len(items)), [None] * len(items)
        for n in range(case["n_lo"], case["n_hi"] + 1):
            ids = [i for i, it in enumerate(items) if it.circuit.n == n]
            for at in range(0, len(ids), 64):
                part = ids[at:at + 64]
                ee, gg = _hea_exact([items[i].circuit for i in part], [items[i].observable for i in part])
                for i, x, y in zip(part, ee, gg):
                    e[i], g[i] = x, y
        return {"energies": e, "gradients": np.concatenate(g)}
    n = case["n"]
    _, tdt = _types(case)
    if kind == "grad":
        c = W.hea_circuit(n, case["layers"], seed)
        e, g = _hea_exact([c], [W.tfim_observable(n, 1.0)])
        return {"energy": np.float64(e[0]), "gradient": g[0]}
    if kind == "run":
        if n > 28:  # about a minute of 64-bit gates
            return None
        psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
        psi[0] = 1.0
        for g in W.u3cz_circuit(n, case["depth"], seed).gates:
            _apply(psi, n, g)
        return {"state": psi, "energy": np.float64(_pauli_sum(psi, _z0z1(n)).real)}
    psi = _random_tensor(n, tdt, seed).to(torch.complex128)
    if kind == "gates":
        gates, (x, z, angle) = _gate_list(case, seed)
        for g in gates:
            _apply(psi, n, g)
        return {"state": math.cos(angle / 2) * psi + 1j * math.sin(angle / 2) * _pauli_on(psi, x, z)}
    if kind == "energy":
        return {"energy": np.float64(_pauli_sum(psi, _observable(case, seed)).real)}
    if kind == "overlap":
        b = _random_tensor(n, tdt, seed + 1000003).to(torch.complex128)
        t, i = _pauli_sum(b, _observable(case, seed), psi), torch.vdot(psi, b).item()
        return {"transition": np.array([t.real, t.imag]), "inner": np.array([i.real, i.imag]),
                "norms": np.array([torch.vdot(psi, psi).real.item(), torch.vdot(b, b).real.item()])}
    if kind == "measure":
        p = psi.real ** 2 + psi.imag ** 2
        fix = [(q, v) for q, v in enumerate(_measured(case, seed)) if v != 2]
        x = torch.arange(1 << n, device="cuda")
        mask, val = sum(1 << q for q, _ in fix), sum(v << q for q, v in fix)
        # (the shots are whole numbers, the same wherever a draw is not within rounding of an edge)
        return {"samples": None, "marginal": np.float64(p[(x & mask) == val].sum().item())}
    obs = _observable(case, seed)
    for _ in range(case["slices"]):
        for c, x, z in zip(obs.coef, obs.x_mask, obs.z_mask):
            a = TIME / case["slices"] * float(c)
            psi = math.cos(a) * psi + 1j * math.sin(a) * _pauli_on(psi, x, z)
    return {"state": psi}
