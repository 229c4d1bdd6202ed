"""Trotter slices in fused blocks (states of 128 MiB and more) against one pass per term (the same
call with the state's tensor cores off)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# per block 2^-45 (double-float) or 2^-24 (complex64) of the group's largest amplitude, at most 60
# blocks or 200 single rotations a run, amplitudes up to 2^-9 of these states
TOL = {"c128": 1e-12, "c64": 1e-5}


def few_body(n, terms, seed):
    """Strings on 1..6 qubits with X, Y and Z, and an identity term."""
    rng = W.SplitMix64(seed)
    coef, xm, zm = [0.3], [0], [0]
    for _ in range(terms):
        qubits = {rng.randint(0, n - 1) for _ in range(rng.randint(1, 6))}
        x, z = W.pauli_masks([rng.randint(1, 3) for _ in qubits], sorted(qubits))
        coef.append(rng.uniform_range(-1.0, 1.0))
        xm.append(x)
        zm.append(z)
    return W.PauliObservable(n, np.array(coef), np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64))


def joined(n, *obs):
    return W.PauliObservable(n, *(np.concatenate([getattr(o, f) for o in obs]) for f in ("coef", "x_mask", "z_mask")))


@pytest.mark.parametrize("dtype,n", [("c128", 23), ("c64", 24)])
@pytest.mark.parametrize("case", ["chain", "chain_many_slices", "few_body", "long_first", "long_between", "long_only"])
def test_blocks_equal_terms(case, dtype, n):
    import torch
    import paper_2011_13524_gb300 as qs
    long2 = W.random_pauli_observable(n, 2, 5)  # strings over most qubits
    obs, slices = {
        "chain": (W.tfim_observable(n, 0.7), 1),
        "chain_many_slices": (W.tfim_observable(n, 0.7), 8),  # more gates than one plan holds
        "few_body": (few_body(n, 20, 3), 2),
        "long_first": (joined(n, long2, few_body(n, 6, 4)), 2),
        "long_between": (joined(n, few_body(n, 6, 6), long2, few_body(n, 6, 7)), 2),
        "long_only": (long2, 2),
    }[case]
    dt, tdt = (qs.QS_C64, torch.complex64) if dtype == "c64" else (qs.QS_C128, torch.complex128)
    g = torch.Generator(device="cuda")
    g.manual_seed(17)
    v = torch.randn(1 << n, dtype=tdt, device="cuda", generator=g)
    v /= torch.linalg.vector_norm(v)
    a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
    b.set_arith(tensor=0)
    a.apply_observable_rotation(obs, 0.4, slices)
    b.apply_observable_rotation(obs, 0.4, slices)
    a.synchronize()
    b.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL[dtype]
    a.close()
    b.close()


def bodies(n, count, body, seed):
    """Random strings on `body` qubits each."""
    rng = W.SplitMix64(seed)
    coef, xm, zm = [], [], []
    for _ in range(count):
        qubits = set()
        while len(qubits) < body:
            qubits.add(rng.randint(0, n - 1))
        x, z = W.pauli_masks([rng.randint(1, 3) for _ in range(body)], sorted(qubits))
        coef.append(rng.uniform_range(-0.1, 0.1))
        xm.append(x)
        zm.append(z)
    return W.PauliObservable(n, np.array(coef), np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64))


@pytest.mark.parametrize("dtype,n", [("c128", 23), ("c64", 24)])
@pytest.mark.parametrize("case", ["fused_and_not", "more_than_a_plan", "not_fused", "hopping"])
@pytest.mark.parametrize("slices", [1, 2])
def test_parts_of_a_slice(case, slices, dtype, n):
    """Slices whose runs of terms are partly cheaper in blocks and partly by passes, in order."""
    import torch
    import paper_2011_13524_gb300 as qs
    chain = W.tfim_observable(n, 0.7)
    hop = [((1 << i) | (1 << j), sum(1 << k for k in range(i + 1, j))) for i in range(0, n, 3) for j in range(i + 1, min(n, i + 9), 2)]
    obs = {
        "fused_and_not": joined(n, chain, W.random_pauli_observable(n, 1, 5), bodies(n, 20, 4, 3), W.random_pauli_observable(n, 1, 6), chain),
        "more_than_a_plan": joined(n, bodies(n, 250, 2, 8), chain),
        "not_fused": bodies(n, 20, 5, 9),
        "hopping": W.PauliObservable(n, np.full(len(hop), 0.1), *(np.array(m, dtype=np.uint64) for m in zip(*hop))),
    }[case]
    dt, tdt = (qs.QS_C64, torch.complex64) if dtype == "c64" else (qs.QS_C128, torch.complex128)
    g = torch.Generator(device="cuda")
    g.manual_seed(18)
    v = torch.randn(1 << n, dtype=tdt, device="cuda", generator=g)
    v /= torch.linalg.vector_norm(v)
    a, b = qs.State(n, dt, tensor=v.clone()), qs.State(n, dt, tensor=v)
    b.set_arith(tensor=0)
    a.apply_observable_rotation(obs, 0.4, slices)
    b.apply_observable_rotation(obs, 0.4, slices)
    a.synchronize()
    b.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL[dtype]
    a.close()
    b.close()
