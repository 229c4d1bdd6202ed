"""Trotter slices of large states where their fused blocks cannot be prepared: under a stream capture,
and without device memory for the block matrices. Both give the result of one pass per term."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N = 23  # 128 MiB in complex128: the size from which slices are fused
TOL = 1e-12  # as for fused blocks against terms


def pair(qs, stream=None):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    v = torch.randn(1 << N, dtype=torch.complex128, device="cuda", generator=g)
    v /= torch.linalg.vector_norm(v)
    a, b = qs.State(N, tensor=v.clone(), stream=stream), qs.State(N, tensor=v, stream=stream)
    torch.cuda.synchronize()
    b.set_arith(tensor=0)
    return a, b


def test_capture():
    import torch
    import paper_2011_13524_gb300 as qs
    obs, st = W.tfim_observable(N, 0.7), torch.cuda.Stream()
    a, b = pair(qs, st)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        a.apply_observable_rotation(obs, 0.4, 1)
    with torch.cuda.stream(st):
        graph.replay()
    b.apply_observable_rotation(obs, 0.4, 1)
    a.synchronize()
    b.synchronize()
    torch.cuda.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL
    a.close()
    b.close()


@pytest.mark.parametrize("slices", [1, 9])  # one plan, and several with a shorter last one
def test_no_memory_for_blocks(slices):
    import paper_2011_13524_gb300 as qs
    obs = W.tfim_observable(N, 0.7)
    a, b = pair(qs)
    a.apply_observable_rotation(obs, 0.0, 1)  # (one-time allocations)
    qs.check(qs.lib().qs_debug_fail_alloc(0, None))
    try:
        a.apply_observable_rotation(obs, 0.4, slices)
    finally:
        qs.check(qs.lib().qs_debug_fail_alloc(-1, None))
    b.apply_observable_rotation(obs, 0.4, slices)
    a.synchronize()
    b.synchronize()
    assert float((a.tensor - b.tensor).abs().max()) < TOL
    a.close()
    b.close()


@pytest.mark.parametrize("n", [5, N])
def test_no_terms_many_slices(n):
    """Without terms a call has nothing to loop over, whatever its slices."""
    import numpy as np
    import torch
    import paper_2011_13524_gb300 as qs
    st = qs.State(n, qs.QS_C128)
    ref = st.tensor.clone()
    none = W.PauliObservable(n, np.array([]), np.array([], dtype=np.uint64), np.array([], dtype=np.uint64))
    st.apply_observable_rotation(none, 0.4, 2 ** 31 - 1)
    st.synchronize()
    assert torch.equal(st.tensor, ref)
    st.close()
