"""Tabulated propagators where the difference of two times is no number."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads.generate import Graph  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [0, 1, 2])
def test_nan_times_give_nan_results(schedule):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg

    g = Graph([1, 2, 1], [0, 2, 2], np.array([[0, 1, 0, 1, 0], [0, 2, 0, 0, 1], [1, 3, 0, 1, 0], [2, 3, 0, 0, 1]]), 1, 2)
    t = np.array([[1.0, 2.0], [np.nan, 2.0], [1.0, np.nan], [np.inf, np.inf], [3.0, 2.5]])
    gr = cg.Graph.from_workload_graph(g)
    gr.set_propagator_table(np.random.default_rng(0).normal(size=(1, 2, 9)), 8.0)
    gr.set_tuning(schedule=schedule)
    gr.set_samples(t, np.zeros(1), 8.0, cg.COS_T_HOST | cg.COS_T_SAMPLE_MAJOR)
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    gr.evaluate(0, out=out, want_mean=False)
    assert torch.isnan(out).tolist() == [False, True, True, True, False]
    gr.close()
