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


@pytest.mark.parametrize("scale", [2.0 ** -80, 2.0 ** 70])
@pytest.mark.parametrize("n", [4, 14])
def test_singles_of_scaled_complex64_states(n, scale):
    """Amplitudes whose products leave FP32's range: the sums are those of FP64 products, as in a group of
    its own, to 1e-14 of the summed magnitudes (FP64 on both sides)."""
    import paper_2011_13524_gb300 as qs
    full = (1 << n) - 1
    st = qs.State(n, qs.QS_C64)
    st.load(W.random_state_fast(n, 11) * scale)
    vec = st.get_vector().astype(np.complex128)
    for x, z in [(full, 0), (full, 5), (full, full), (1, 2)]:
        obs = W.PauliObservable(n, np.array([0.75]), np.array([x], dtype=np.uint64), np.array([z], dtype=np.uint64))
        size = float((np.abs(vec) * np.abs(vec[np.arange(1 << n) ^ x])).sum())
        assert abs(st.expectation(obs)[0] - oracle.expectation(vec, obs)[0]) < 1e-14 * size
    st.close()


def test_singles_of_small_pairs_beside_large_ones():
    """A string that joins amplitudes of 2^-70 only, beside one of 1, in complex64; and an amplitude that is
    not finite."""
    import paper_2011_13524_gb300 as qs
    n = 14
    full = (1 << n) - 1
    v = W.random_state_fast(n, 12) * 2.0 ** -70
    v[1000] = 1.0
    v[1000 ^ full] = 0.0
    st = qs.State(n, qs.QS_C64)
    st.load(v)
    vec = st.get_vector().astype(np.complex128)
    obs = W.PauliObservable(n, np.array([1.0]), np.array([full], dtype=np.uint64), np.array([3], dtype=np.uint64))
    size = float((np.abs(vec) * np.abs(vec[::-1])).sum())
    assert abs(st.expectation(obs)[0] - oracle.expectation(vec, obs)[0]) < 1e-14 * size
    for bad in (np.nan, np.inf):
        v[77] = bad
        st.load(v)
        assert not np.isfinite(st.expectation(obs)[0])
    st.close()
