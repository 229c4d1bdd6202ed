"""The gradient's forward pass on either side of the size where complex128 goes from gate passes to
fused blocks, with every gate kind between the rotations, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11  # the bound of the other complex128 gradient tests, per qubit


@pytest.mark.parametrize("math", ["df", "f64"])
@pytest.mark.parametrize("n", [6, 13, 16, 17])
def test_forward_of_gradient(n, math):
    import paper_2011_13524_gb300 as qs
    a, b = W.hea_circuit(n, 1, n), W.hea_circuit(n, 1, n + 1)
    shifted = [W.Gate(g.name, g.targets, g.controls, g.control_values, g.params, matrix=g.matrix, pauli=g.pauli,
                      param_index=g.param_index + a.n_params if g.param_index >= 0 else -1) for g in b.gates]
    c = W.Circuit(n, a.gates + W.random_gate_suite(n, 5) + shifted, n_params=a.n_params + b.n_params)
    obs = W.random_pauli_observable(n, 6, 3)
    old = qs.get_c128_math()
    try:
        qs.set_c128_math(qs.QS_MATH_FP64 if math == "f64" else qs.QS_MATH_DF)
        e, g = qs.adjoint_grad(c, obs)
    finally:
        qs.set_c128_math(old)
    assert abs(e - oracle.energy(c, obs)) < TOL * n
    idx = [0, 1, n, 2 * n - 1, 2 * n, 3 * n, 4 * n - 1]
    assert float(np.max(np.abs(g[idx] - oracle.grad_parameter_shift(c, obs, idx)))) < TOL * n


@pytest.mark.parametrize("count", [0, 15, 16, 40])
def test_forward_with_wide_gates(count):
    """Fixed gates of 3..6 targets, fewer and more than gate passes serve, and no gate at all."""
    import paper_2011_13524_gb300 as qs
    n = 9
    rng = W.SplitMix64(count)
    h = W.hea_circuit(n, 2, 3)
    gates = list(h.gates) if count else []
    for j in range(count):
        m = 3 + j % 4
        gates.insert((j * 7) % len(gates), W.Gate("DENSE", tuple((3 * j + 2 * i) % n for i in range(m)), matrix=W.random_unitary(1 << m, rng)))
    c = W.Circuit(n, gates, n_params=h.n_params)
    obs = W.random_pauli_observable(n, 6, 3)
    e, g = qs.adjoint_grad(c, obs)
    assert abs(e - oracle.energy(c, obs)) < TOL * n
    if not count:
        assert not np.any(g)
        return
    idx = [0, 1, n, 2 * n - 1, 2 * n, 3 * n, 4 * n - 1]
    assert float(np.max(np.abs(g[idx] - oracle.grad_parameter_shift(c, obs, idx)))) < TOL * n
