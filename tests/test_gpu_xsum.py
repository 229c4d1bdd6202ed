"""X strings of one weight (k_xsum) in transition amplitudes, beside the expectations of the same: against the oracle, and
against the tiled reads (the same strings with weights that differ), on tile edges, several tiles,
strings on register, lane and warp bits, with diagonal and other terms beside them."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def observable(n, strings):
    coef, xm, zm = zip(*strings)
    return W.PauliObservable(n, np.array(coef), np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64))


def cases(n):
    chain = [(1.0, 0, 3 << i) for i in range(n - 1)] + [(0.7, 1 << i, 0) for i in range(n)]
    high = [(-0.3, 1 << i, 0) for i in range(n - 5, n)]
    pairs = [(0.4, 3 << i, 0) for i in range(n - 1)] + [(0.4, 1 | (1 << (n - 1)), 0)]
    mixed = chain + [(0.2, 3, 3), (0.5, 1, 2), (0.7, 7, 0), (-0.7, 5, 0), (1.5, 0, 0), (0.25, (1 << n) - 1, 5)]
    few = [(1.0, 1, 0), (1.0, 2, 0), (1.0, 1 << (n - 1), 0)]  # fewer than a read of their own takes
    return {"chain": chain, "high": high, "pairs": pairs, "mixed": mixed, "few": few}


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n", [11, 12, 13, 15])
@pytest.mark.parametrize("case", ["chain", "high", "pairs", "mixed", "few"])
def test_against_the_oracle(case, n, dtype):
    import paper_2011_13524_gb300 as qs
    obs = observable(n, cases(n)[case])
    dt = qs.QS_C64 if dtype == "c64" else qs.QS_C128
    a, b = qs.State(n, dt), qs.State(n, dt)
    a.load(W.random_state_fast(n, 1))
    b.load(W.random_state_fast(n, 2))
    va, vb = a.get_vector().astype(np.complex128), b.get_vector().astype(np.complex128)
    # the tiled reads' bound: 1e-13 of the weights (norm 1 to the storage's rounding)
    tol = 1e-13 * float(np.abs(obs.coef).sum())
    assert abs(a.expectation(obs)[0] - oracle.expectation(va, obs)[0]) < tol
    t = oracle.transition_amplitude(va, vb, n, obs)
    assert abs(a.transition_amplitude(obs, b) - t) < tol
    a.close()
    b.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_against_tiled_reads(dtype):
    """Eight tiles and more per CTA; amplitudes over many magnitudes between tiles."""
    import torch
    import paper_2011_13524_gb300 as qs
    n = 22
    dt, tdt = (qs.QS_C64, torch.complex64) if dtype == "c64" else (qs.QS_C128, torch.complex128)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    states = []
    for _ in range(2):
        v = torch.randn(1 << n, dtype=tdt, device="cuda", generator=g)
        v *= torch.exp2(-(torch.arange(1 << n, device="cuda") >> 14) % 31)
        states.append(qs.State(n, dt, tensor=v / torch.linalg.vector_norm(v)))
    a, b = states
    same = observable(n, [(0.5, 1 << i, 0) for i in range(n)])
    apart = observable(n, [(0.5 + 2.0 ** -20 * i, 1 << i, 0) for i in range(n)])
    back = observable(n, [(-(2.0 ** -20) * i, 1 << i, 0) for i in range(1, n)])
    tol = 1e-13 * n
    assert abs(a.expectation(same)[0] - (a.expectation(apart)[0] + a.expectation(back)[0])) < tol
    t = a.transition_amplitude(apart, b) + a.transition_amplitude(back, b)
    assert abs(a.transition_amplitude(same, b) - t) < tol
    zero = qs.State(n, dt)
    assert a.transition_amplitude(same, a) == pytest.approx(a.expectation(same)[0], abs=tol)
    assert abs(zero.expectation(same)[0]) < tol  # all tiles but one empty
    for s in (a, b, zero):
        s.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("part", [1.0, 1j])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_not_finite(bad, part, dtype):
    """One amplitude of the ket that is not finite: neither part of the sum is a number to go on with."""
    import paper_2011_13524_gb300 as qs
    n = 14
    dt = qs.QS_C64 if dtype == "c64" else qs.QS_C128
    obs = observable(n, [(0.5, 1 << i, 0) for i in range(n)])
    a, b = qs.State(n, dt), qs.State(n, dt)
    v = W.random_state_fast(n, 2)
    v[5000] = complex(bad, 0.25) if part == 1.0 else complex(0.25, bad)
    a.load(W.random_state_fast(n, 1))
    b.load(v)
    t = a.transition_amplitude(obs, b)
    assert not np.isfinite(t.real) and not np.isfinite(t.imag)
    a.close()
    b.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("orders", [10, 40, 90])
def test_small_components_beside_large_ones(orders, dtype):
    """Ket amplitudes over many binary orders within one tile, read out one by one: each sum keeps its own
    accuracy. The bound: components cut at 2^-46 of themselves (complex64: exact), at most 13 of them summed
    with an error of 2^-47 of their magnitudes per addition, one product."""
    import paper_2011_13524_gb300 as qs
    n = 14
    dt = qs.QS_C64 if dtype == "c64" else qs.QS_C128
    obs = observable(n, [(1.0, 1 << i, 0) for i in range(n)])
    a, b = qs.State(n, dt), qs.State(n, dt)
    order = (np.arange(1 << n) * 2654435761 >> 7) % (orders + 1)
    b.load(W.random_state_fast(n, 3) * 2.0 ** (7.0 - order))
    ket = b.get_vector().astype(np.clongdouble)
    for y in (0, 1, 255, 256, 4095, 4096, 9999, (1 << n) - 1):
        near = ket[[y ^ (1 << i) for i in range(n)]]
        bra = np.zeros(1 << n, dtype=np.complex128)
        bra[y] = 1.0
        a.load(bra)
        err = abs(np.clongdouble(a.transition_amplitude(obs, b)) - near.sum())
        assert err < 2.0 ** -42 * np.abs(near).sum()
    # a small answer beside amplitudes of 1 that it does not read
    small = W.random_state_fast(n, 4) * 2.0 ** -orders
    small[[4095, (1 << n) - 1]] = 1.0
    b.load(small)
    ket = b.get_vector().astype(np.clongdouble)
    near = ket[[1 << i for i in range(n)]]
    bra = np.zeros(1 << n, dtype=np.complex128)
    bra[0] = 1.0
    a.load(bra)
    assert abs(np.clongdouble(a.transition_amplitude(obs, b)) - near.sum()) < 2.0 ** -42 * np.abs(near).sum()
    a.close()
    b.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_sums_beyond_the_range(dtype):
    """Ket components whose sums, not whose products with the bra, leave FP32's range."""
    import paper_2011_13524_gb300 as qs
    n = 14
    dt = qs.QS_C64 if dtype == "c64" else qs.QS_C128
    obs = observable(n, [(1.0, 1 << i, 0) for i in range(n)])
    a, b = qs.State(n, dt), qs.State(n, dt)
    a.load(W.random_state_fast(n, 1) * 1e-25)
    b.load(np.full(1 << n, 3e38 - 2.5e38j))
    va, vb = a.get_vector().astype(np.complex128), b.get_vector().astype(np.complex128)
    t = a.transition_amplitude(obs, b)
    assert abs(t - oracle.transition_amplitude(va, vb, n, obs)) < 1e-13 * n * float(np.sum(np.abs(va)) * np.abs(vb[0]))
    a.close()
    b.close()
