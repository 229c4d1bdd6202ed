"""Single gate calls in complex128 whose kernels read and write the IEEE layout (double-float dense gates
of 3..6 targets, Pauli rotations) or skip products by zero (real and imaginary one-qubit entries)."""
import math

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-13  # one gate on amplitudes <= 1: double-float 2^-45, FP64 below it


def run(n, math_mode, tensor, act, seed=3):
    import paper_2011_13524_gb300 as qs
    st = qs.State(n, qs.QS_C128)
    st.set_arith(math=math_mode, tensor=tensor)
    st.load(W.random_state(n, seed))
    act(st)
    out = st.get_vector()
    st.close()
    return out


@pytest.mark.parametrize("tensor", [0, 6])
@pytest.mark.parametrize("m", [3, 4, 5, 6])
def test_dense_calls(m, tensor):
    import paper_2011_13524_gb300 as qs
    rng = W.SplitMix64(m)
    U = W.random_unitary(1 << m, rng)
    for n, targets, controls in [(m, tuple(range(m)), ()), (8, tuple(range(8 - m, 8)), ()), (9, tuple(reversed(range(1, 1 + m))), ()),
                                 (11, (0, 10, 4, 7, 2, 5)[:m], ()), (9, tuple(range(m)), (8,))]:
        g = W.Gate("DENSE", targets, controls=controls, control_values=(0,) * len(controls), matrix=U)
        ref = W.random_state(n, 3)
        oracle.apply_gate(ref, n, g)
        got = run(n, qs.QS_MATH_DF, tensor, lambda st: st.apply_gate(g))
        assert float(np.max(np.abs(got - ref))) < TOL, (n, targets)


@pytest.mark.parametrize("mode", ["df", "f64"])
def test_rotation_calls(mode):
    import paper_2011_13524_gb300 as qs
    n = 9
    for x, z in [(1, 0), (1, 1), (0b110, 0b010), (0b111, 0b111), (0b100000001, 0b000010000), (511, 510), (0, 0b1010), (0, 0)]:
        got = run(n, qs.QS_MATH_DF if mode == "df" else qs.QS_MATH_FP64, 6, lambda st: st.apply_pauli_rotation(x, z, 0.77))
        psi = W.random_state(n, 3)
        idx = np.arange(1 << n)
        src = idx ^ x
        sign = np.array([(-1.0) ** bin(int(s) & z).count("1") for s in src])
        ref = math.cos(0.385) * psi + 1j * math.sin(0.385) * (1j ** bin(x & z).count("1")) * sign * psi[src]
        assert float(np.max(np.abs(got - ref))) < TOL, (x, z)


def test_one_qubit_forms():
    import paper_2011_13524_gb300 as qs
    n = 7
    real = np.array([[0.3, -1.2], [0.7, 0.4]])
    imag = np.array([[0.3, -1.2j], [0.7j, 0.4]])
    gates = [W.Gate("H", (2,)), W.Gate("RY", (0,), params=(0.4,)), W.Gate("RX", (6,), params=(1.4,)), W.Gate("U2", (3,), params=(0.2, 0.9)),
             W.Gate("DENSE", (5,), matrix=real), W.Gate("DENSE", (1,), matrix=imag), W.Gate("DENSE", (1,), matrix=real + 0.1j * imag),
             W.Gate("DENSE", (4,), controls=(0, 6), control_values=(1, 0), matrix=imag)]
    for g in gates:
        ref = W.random_state(n, 3)
        oracle.apply_gate(ref, n, g)
        assert float(np.max(np.abs(run(n, qs.QS_MATH_DF, 6, lambda st: st.apply_gate(g)) - ref))) < TOL, g.name
