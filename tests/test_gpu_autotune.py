"""Predictions of the fusion autotuner against measured device times."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def measured_ms(qs, c, dtype, k):
    import torch
    st = qs.State(c.n, dtype)
    best = 1e9
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        st.run(c, k)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    st.close()
    return best


@pytest.mark.parametrize("dtype", [2, 1])
def test_small_probe_does_not_serve_large_states(dtype):
    """A circuit of 8 qubits tuned first: its launch-bound costs are not scaled by 2^14."""
    import paper_2011_13524_gb300 as qs
    qs.autotune_fusion(W.u3cz_circuit(8, 4, 1), dtype)
    c = W.u3cz_circuit(22, 4, 2)
    pred = qs.autotune_fusion(c, dtype)[1]
    assert pred[4] < 10.0 * measured_ms(qs, c, dtype, 4)  # (8192 times too long otherwise)


@pytest.mark.parametrize("dtype", [2, 1])
@pytest.mark.parametrize("n", [12, 20, 23])
def test_unfused_prediction_counts_passes(n, dtype):
    """Index 0 follows a run that applies several gates per pass (175 gates in 4 passes at n = 12), within
    the host's share at small sizes and the spread of the gates' costs."""
    import paper_2011_13524_gb300 as qs
    c = W.u3cz_circuit(n, 10, 2)
    pred, got = qs.autotune_fusion(c, dtype)[1][0], measured_ms(qs, c, dtype, 0)
    assert got / 4.0 < pred < 2.0 * got
