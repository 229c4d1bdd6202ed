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
