"""Terms alone in their flip group (k_expect_singles) against the oracle and against the general
group kernel (the same terms entered twice with half weight, which makes a two-term group)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def observable(n, strings):
    xm, zm = zip(*strings)
    rng = W.SplitMix64(n + len(strings))
    return W.PauliObservable(n, np.array([rng.uniform_range(-1.0, 1.0) for _ in strings]),
                             np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64))


def doubled(obs):
    return W.PauliObservable(obs.n, np.repeat(obs.coef * 0.5, 2), np.repeat(obs.x_mask, 2), np.repeat(obs.z_mask, 2))


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,count", [(1, 1), (2, 1), (4, 2), (13, 1), (14, 30), (16, 100)])
def test_singles_against_the_oracle(n, count, dtype):
    import paper_2011_13524_gb300 as qs
    rng = W.SplitMix64(100 * n + count)
    full = (1 << n) - 1
    strings = [(1 << (n - 1), full), (full, full), (full, 0)][:min(count, n)]
    while len(strings) < count:
        x = rng.next_u64() & full
        if x and x not in [s[0] for s in strings]:
            strings.append((x, rng.next_u64() & full))
    obs = observable(n, strings[:count])
    st = qs.State(n, qs.QS_C64 if dtype == "c64" else qs.QS_C128)
    st.load(W.random_state_fast(n, 7))
    vec = st.get_vector().astype(np.complex128)
    # sums of 2^n products of amplitudes with norm 1, in FP64 on both sides
    tol = 1e-14 * (1.0 + float(np.abs(obs.coef).sum()))
    got = st.expectation(obs)
    assert got[1] == 0.0 and abs(got[0] - oracle.expectation(vec, obs)[0]) < tol
    assert abs(got[0] - st.expectation(doubled(obs))[0]) < 10 * tol  # (tiled double-float: 1e-13)
    st.close()


def test_singles_hold_wide_magnitudes():
    """complex64 amplitudes over 30 binary orders: cancelling contributions stay exact."""
    import paper_2011_13524_gb300 as qs
    n = 15
    v = W.random_state_fast(n, 3) * 2.0 ** -(np.arange(1 << n) % 31)
    st = qs.State(n, qs.QS_C64)
    st.load(v)
    vec = st.get_vector().astype(np.complex128)
    wide = sum(1 << q for q in range(3, 14))
    for x, z in [(wide, 0), (wide | 1, wide), (1, 2), ((1 << n) - 1, 5)]:
        obs = W.PauliObservable(n, np.array([1.0]), np.array([x], dtype=np.uint64), np.array([z], dtype=np.uint64))
        ref = oracle.expectation(vec, obs)[0]
        assert abs(st.expectation(obs)[0] - ref) < 1e-15 * float((np.abs(vec) ** 2).sum())
    st.close()
