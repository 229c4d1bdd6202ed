"""Runs of diagonal gates in the gradient's reverse sweep (k_adj_diag): factors on a thread's own bits
alone, on the top bits, across both, conditional ones and signs, in shuffled order, against the
oracle's parameter shift."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"df": 1e-11, "f64": 1e-11, "c64": 1e-4}  # the bounds of the other gradient tests


def circuit(n, seed):
    rng = W.SplitMix64(seed)
    gates, p = [W.Gate("H", (q,)) for q in range(n)], 0
    for layer in range(2):
        run = [W.Gate("CZ", (q, q + 1)) for q in range(n - 1)] + [W.Gate("CZ", (0, n - 1))]
        run += [W.Gate("RZ", (q,), params=(rng.uniform_range(-3, 3),), param_index=p + q) for q in range(n)]
        p += n
        run.append(W.Gate("PAULIROT", (0, n - 1), pauli=(3, 3), params=(0.7,), param_index=p))
        p += 1
        for a, b in ((0, 1), (1, n - 1), (n - 1, n - 2)):
            d = np.exp(1j * np.array([rng.uniform_range(-3, 3) for _ in range(4)]))
            run.append(W.Gate("DIAG", (a, b), matrix=d))
        run += [W.Gate("T", (0,)), W.Gate("S", (n - 1,)), W.Gate("Z", (n - 1,)), W.Gate("Z", (1,))]
        run.append(W.Gate("DIAG", (0,), controls=(n - 1,), control_values=(0,), matrix=np.exp(1j * np.array([0.4, -0.9]))))
        for i in range(len(run) - 1, 0, -1):
            j = rng.randint(0, i)
            run[i], run[j] = run[j], run[i]
        gates += run + [W.Gate("RX", (q,), params=(0.2 + 0.1 * q,)) for q in range(n)]
    return W.Circuit(n, gates, n_params=p)


@pytest.mark.parametrize("arith", ["df", "f64", "c64"])
@pytest.mark.parametrize("n", [3, 8, 9, 10, 13])
def test_diagonal_runs(n, arith):
    import paper_2011_13524_gb300 as qs
    c = circuit(n, n)
    obs = W.tfim_observable(n, 0.8)
    old = qs.get_c128_math()
    try:
        qs.set_c128_math(qs.QS_MATH_FP64 if arith == "f64" else qs.QS_MATH_DF)
        e, g = qs.adjoint_grad(c, obs, dtype=qs.QS_C64 if arith == "c64" else qs.QS_C128)
    finally:
        qs.set_c128_math(old)
    assert abs(e - oracle.energy(c, obs)) < TOL[arith] * n
    idx = [0, 1, n - 2, n - 1, n, n + 1, 2 * n, 2 * n + 1]
    assert float(np.max(np.abs(g[idx] - oracle.grad_parameter_shift(c, obs, idx)))) < TOL[arith] * n
