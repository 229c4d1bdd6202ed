"""Several gates per pass (gate-by-gate circuit runs) against the same gates applied one call at a
time, over tile edges, low, high and scattered qubits, controls, strings longer than a tile, and the
layout changes folded into the first and last pass."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# per gate 2^-46 (double-float; FP64 below it) or 2^-23 (complex64) of amplitudes <= 1, at most 400 gates
TOL = {"df": 1e-12, "f64": 1e-12, "c64": 1e-5}


def random_tensor(n, dtype, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v = torch.randn(1 << n, dtype=dtype, device="cuda", generator=g)
    return v / torch.linalg.vector_norm(v)


def mixed_circuit(n, seed):
    """Every gate kind twice in shuffled order, long Pauli rotations among them, between layers."""
    rng = W.SplitMix64(seed)
    gates = W.u3cz_circuit(n, 2, seed).gates
    if n >= 6:
        suite = W.random_gate_suite(n, seed) + W.random_gate_suite(n, seed + 1)
        for i in range(len(suite) - 1, 0, -1):
            j = rng.randint(0, i)
            suite[i], suite[j] = suite[j], suite[i]
        gates += suite
        ids = tuple(rng.randint(1, 3) for _ in range(6))
        gates.append(W.Gate("PAULIROT", tuple(range(n - 6, n)), pauli=ids, params=(0.4,)))
    gates += W.hea_circuit(n, 1, seed).gates
    return W.Circuit(n, gates)


@pytest.mark.parametrize("arith", ["df", "f64", "c64"])
@pytest.mark.parametrize("n", [1, 2, 5, 8, 9, 10, 12, 15, 18, 19, 21])
def test_passes_equal_single_gates(n, arith):
    import torch
    import paper_2011_13524_gb300 as qs
    dt, tdt = (qs.QS_C64, torch.complex64) if arith == "c64" else (qs.QS_C128, torch.complex128)
    v = random_tensor(n, tdt, n)
    a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
    math = qs.QS_MATH_FP64 if arith == "f64" else qs.QS_MATH_DF
    a.set_arith(math=math)
    b.set_arith(math=qs.QS_MATH_FP64)
    c = mixed_circuit(n, 3 + n) if n > 1 else W.Circuit(1, [W.Gate("H", (0,)), W.Gate("T", (0,)), W.Gate("RX", (0,), params=(0.3,))])
    a.run(c, 0)
    for g in c.gates:
        b.apply_gate(g)
    a.synchronize()
    b.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL[arith]
    a.close()
    b.close()


@pytest.mark.parametrize("arith", ["df", "c64"])
def test_one_gate_runs(arith):
    """Runs of a single gate of each kind: one pass that changes the layout on both sides."""
    import torch
    import paper_2011_13524_gb300 as qs
    n = 13
    dt, tdt = (qs.QS_C64, torch.complex64) if arith == "c64" else (qs.QS_C128, torch.complex128)
    for i, g in enumerate(W.random_gate_suite(n, 8)):
        v = random_tensor(n, tdt, i)
        a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
        b.set_arith(math=qs.QS_MATH_FP64)
        a.run(W.Circuit(n, [g]), 0)
        b.apply_gate(g)
        a.synchronize()
        b.synchronize()
        assert float((a.tensor - b.tensor).abs().max()) < TOL[arith], g
        a.close()
        b.close()


def test_long_runs_and_many_slices():
    """More gates than the scheduler looks at together, and Trotter slices in batches."""
    import paper_2011_13524_gb300 as qs
    import oracle
    c = W.u3cz_circuit(9, 90, 4)  # 1170 gates
    st = qs.State(9, qs.QS_C128)
    st.run(c, 0)
    assert float(np.max(np.abs(st.get_vector() - oracle.run_circuit(c)))) < 2e-12
    obs = W.random_pauli_observable(9, 9, 5)
    psi = W.random_state(9, 3)
    st.load(psi)
    st.apply_observable_rotation(obs, 0.9, 150)  # 1350 rotations
    assert float(np.max(np.abs(st.get_vector() - oracle.observable_rotation(psi, 9, obs, 0.9, 150)))) < 2e-12
    st.close()


@pytest.mark.parametrize("arith", ["df", "f64", "c64"])
@pytest.mark.parametrize("n", [19, 20])
def test_launches_between_passes(n, arith):
    """Runs of one kind, of one gate to more than a tile pays for, on either side of the size from which a
    pass may be launched gate by gate: as tiles, as launches, and both in one run."""
    import torch
    import paper_2011_13524_gb300 as qs
    dt, tdt = (qs.QS_C64, torch.complex64) if arith == "c64" else (qs.QS_C128, torch.complex128)
    rng = W.SplitMix64(n)
    qubits = [(0, n - 1), (n // 2, 1), (n - 1, 3), (2, n - 2)]
    apart = W.Gate("DENSE", (0, n // 2, n - 1), matrix=W.random_unitary(8, rng))  # in no tile
    kinds = {
        "u3": lambda a, b: W.Gate("U3", (a,), params=(0.3 + a, 0.2, 0.7)),
        "ry": lambda a, b: W.Gate("RY", (a,), (b,), (1,), params=(0.3 + a,)),
        "dense": lambda a, b: W.Gate("DENSE", (a, b), matrix=W.random_unitary(4, rng)),
        "cz": lambda a, b: W.Gate("CZ", (a, b)),
        "rz": lambda a, b: W.Gate("RZ", (a,), params=(0.7,)),
        "diag": lambda a, b: W.Gate("DIAG", (a, b), matrix=np.exp(1j * np.arange(4))),
        "swap": lambda a, b: W.Gate("SWAP", (a, b)),
        "y": lambda a, b: W.Gate("Y", (a,)),
        "rot": lambda a, b: W.Gate("PAULIROT", (a, b), pauli=(1, 2), params=(0.4,)),
    }
    gates = []
    for make in kinds.values():
        for count in (1, 2, 12):
            gates += [make(*qubits[i % 4]) for i in range(count)] + [apart]
    c = W.Circuit(n, gates)
    v = random_tensor(n, tdt, n)
    a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
    a.set_arith(math=qs.QS_MATH_FP64 if arith == "f64" else qs.QS_MATH_DF)
    b.set_arith(math=qs.QS_MATH_FP64)
    a.run(c, 0)
    for g in gates:
        b.apply_gate(g)
    a.synchronize()
    b.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL[arith]
    a.close()
    b.close()


@pytest.mark.parametrize("arith", ["f64", "c64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(bad, arith):
    """An amplitude that is not finite reaches the same amplitudes through passes as through single gates."""
    import torch
    import paper_2011_13524_gb300 as qs
    n = 12
    dt, tdt = (qs.QS_C64, torch.complex64) if arith == "c64" else (qs.QS_C128, torch.complex128)
    v = random_tensor(n, tdt, 3)
    v[77] = complex(bad, 0.5)
    a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
    for s in (a, b):
        s.set_arith(math=qs.QS_MATH_FP64)
    gates = [W.Gate("H", (0,)), W.Gate("RX", (5,), params=(0.3,)), W.Gate("RZ", (1,), params=(0.2,)), W.Gate("CZ", (0, 11)),
             W.Gate("U3", (11,), params=(0.3, 0.2, 0.7)), W.Gate("SWAP", (3, 9)), W.Gate("PAULIROT", (2, 7), pauli=(1, 3), params=(0.4,))]
    a.run(W.Circuit(n, gates), 0)
    for g in gates:
        b.apply_gate(g)
    a.synchronize()
    b.synchronize()
    x, y = torch.view_as_real(a.tensor), torch.view_as_real(b.tensor)
    fine = torch.isfinite(y)
    assert torch.equal(torch.isfinite(x), fine) and 0 < int((~fine).sum()) < y.numel()
    assert float((x - y)[fine].abs().max()) < TOL[arith]
    a.close()
    b.close()


@pytest.mark.parametrize("arith", ["df", "c64"])
@pytest.mark.parametrize("n", [12, 21])
def test_capture(n, arith):
    """A run gate by gate on a new state is launches alone, whether its passes are tiles or launches."""
    import torch
    import paper_2011_13524_gb300 as qs
    dt, tdt = (qs.QS_C64, torch.complex64) if arith == "c64" else (qs.QS_C128, torch.complex128)
    st = torch.cuda.Stream()
    v = random_tensor(n, tdt, n)
    a, b = qs.State(n, dt, tensor=v.clone(), stream=st), qs.State(n, dt, tensor=v)
    torch.cuda.synchronize()
    rot = tuple(1 + q % 3 for q in range(6))
    gates = [W.Gate("RZ", (3,), params=(0.2,)), W.Gate("PAULIROT", tuple(range(0, 12, 2)), pauli=rot, params=(0.3,)),
             W.Gate("DIAG", (1, n - 1), matrix=np.exp(1j * np.arange(4))), W.Gate("CZ", (0, 5)), W.Gate("H", (2,)),
             W.Gate("DENSE", (0, 4, n - 1), matrix=W.random_unitary(8, W.SplitMix64(5))), W.Gate("SWAP", (1, 2))]
    c = W.Circuit(n, gates + W.u3cz_circuit(n, 2, 3).gates)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        a.run(c, 0)
    with torch.cuda.stream(st):
        graph.replay()
    b.run(c, 0)
    a.synchronize()
    b.synchronize()
    torch.cuda.synchronize()
    assert torch.equal(a.tensor, b.tensor)
    a.close()
    b.close()
