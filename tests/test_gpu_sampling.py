"""Sampling from segment masses (k_sample_pick) against the per-chunk FP64 search (k_sample_find):
the same index for every uniform, and both within rounding of the oracle's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def uniforms(count, seed):
    u = np.random.Generator(np.random.PCG64(seed)).random(count)
    u[:4] = [0.0, 1.0 - 2.0 ** -53, 0.5, 2.0 ** -60]
    return u


def make_vec(kind, n, seed):
    v = W.random_state_fast(n, seed)
    if kind == "sparse":  # whole chunks, segments and most amplitudes empty
        keep = np.zeros(1 << n, dtype=bool)
        keep[np.random.Generator(np.random.PCG64(seed)).integers(0, 1 << n, 97)] = True
        v = np.where(keep, v, 0.0)
    if kind == "skewed":  # masses over 40 orders of magnitude
        v = v * np.exp(-np.arange(1 << n) % 4099 * 0.02)
    if kind == "tiny":  # below the range of FP32 pairs: every sample by the FP64 search
        return v * 2.0 ** -45
    return v / np.linalg.norm(v)


@pytest.mark.parametrize("kind", ["random", "sparse", "skewed", "tiny"])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_segment_search_equals_chunk_search(kind, dtype):
    import paper_2011_13524_gb300 as qs
    n = 26  # 16384 chunks: from 1024 samples on a call takes the segment masses
    st = qs.State(n, qs.QS_C64 if dtype == "c64" else qs.QS_C128)
    v = make_vec(kind, 19, 5)  # a pattern repeated with changing weight
    st.load(np.concatenate([v * (1.0 + 0.01 * k) for k in range(128)]))
    u = uniforms(3000, 9)
    many = st.sample(u)
    few = np.concatenate([st.sample(u[i:i + 750]) for i in range(0, len(u), 750)])
    assert np.array_equal(many, few)
    st.close()


@pytest.mark.parametrize("n", [12, 13, 16])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_segment_search_against_cumulative_sums(n, dtype):
    import paper_2011_13524_gb300 as qs
    st = qs.State(n, qs.QS_C64 if dtype == "c64" else qs.QS_C128)
    st.load(make_vec("random", n, 11))
    p = np.abs(st.get_vector().astype(np.complex128)) ** 2
    cum = np.concatenate([[0.0], np.cumsum(p)])
    u = uniforms(2000, 3)
    got = st.sample(u).astype(np.int64)
    # 2^n positive terms summed in FP64: relative error below 2^n * 2^-53
    tol = 2.0 ** (n - 53) * cum[-1]
    target = u * cum[-1]
    assert np.all(target >= cum[got] - tol) and np.all(target < cum[got + 1] + tol)
    st.close()


def test_marginal_by_insertion_and_by_deposit():
    """Few measured qubits insert bits, many deposit the free ones."""
    import paper_2011_13524_gb300 as qs
    n = 10
    st = qs.State(n, qs.QS_C128)
    st.load(make_vec("random", n, 2))
    p = np.abs(st.get_vector()) ** 2
    x = np.arange(1 << n)
    for mask, val in [(0, 0), (1, 1), (0b1010000001, 0b1000000001), (0b1111011110, 0b0101010100), (1023, 700)]:
        mv = [(val >> q) & 1 if (mask >> q) & 1 else 2 for q in range(n)]
        assert abs(st.marginal_probability(mv) - p[(x & mask) == val].sum()) < 1e-14
    st.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_outside_the_range_of_pairs(dtype):
    """A state of large norm takes the FP64 search (the indices of the same state scaled down), and one
    that is not finite is refused by either search."""
    import paper_2011_13524_gb300 as qs
    n = 14
    st = qs.State(n, qs.QS_C64 if dtype == "c64" else qs.QS_C128)
    v = make_vec("random", n, 3).astype(np.complex64).astype(np.complex128)
    u = uniforms(2000, 4)
    st.load(v)
    ref = st.sample(u)
    st.load(v * 2.0 ** 45)
    assert np.array_equal(st.sample(u), ref)
    v[321] = np.nan
    st.load(v)
    with pytest.raises(qs.QsError) as e:
        st.sample(u)
    assert e.value.code == qs.QS_ERR_NUMERIC
    st.close()
