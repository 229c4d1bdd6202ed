"""Rotations sharing a pass of the gradient's reverse sweep (k_adj_tile): one to ten per pass, odd
counts, repeated qubits, states smaller than a tile, one tile and many, RX and RY with other gates
between, against the oracle's parameter shift."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"df": 1e-11, "f64": 1e-11, "c64": 1e-4}  # the bounds of the other gradient tests


def circuit(n, counts, seed):
    """Layers of `counts` rotations on random qubits (repeats split a pass), entangled between."""
    rng = W.SplitMix64(seed)
    gates, p = [W.Gate("H", (q,)) for q in range(n)], 0
    for count in counts:
        order = list(range(n))
        for i in range(n - 1, 0, -1):
            j = rng.randint(0, i)
            order[i], order[j] = order[j], order[i]
        for i in range(count):
            q = order[i % n]
            gates.append(W.Gate(("RX", "RY")[rng.randint(0, 1)], (q,), params=(rng.uniform_range(-3, 3),), param_index=p))
            p += 1
        if n > 1:
            gates += [W.Gate("CNOT", (q,), controls=(q + 1,), control_values=(1,)) for q in range(n - 1)]
            gates += [W.Gate("RZ", (q,), params=(0.1 * q + 0.3,)) for q in range(n)]
    return W.Circuit(n, gates, n_params=p)


@pytest.mark.parametrize("arith", ["df", "f64", "c64"])
@pytest.mark.parametrize("n,counts", [(1, (1, 1)), (2, (2, 3)), (3, (3, 1, 4)), (5, (5, 2)), (9, (9, 7)), (10, (10, 3)),
                                      (11, (11, 12)), (12, (12, 1)), (14, (14, 5))])
def test_gradient(n, counts, arith):
    import paper_2011_13524_gb300 as qs
    c = circuit(n, counts, n)
    obs = W.tfim_observable(n, 0.8)
    old = qs.get_c128_math()
    try:
        qs.set_c128_math(qs.QS_MATH_FP64 if arith == "f64" else qs.QS_MATH_DF)
        e, g = qs.adjoint_grad(c, obs, dtype=qs.QS_C64 if arith == "c64" else qs.QS_C128)
    finally:
        qs.set_c128_math(old)
    assert abs(e - oracle.energy(c, obs)) < TOL[arith] * n
    idx = list(range(c.n_params)) if n < 12 else list(range(0, c.n_params, 4))
    ps = oracle.grad_parameter_shift(c, obs, idx)
    assert float(np.max(np.abs(g[idx] - ps))) < TOL[arith] * n
