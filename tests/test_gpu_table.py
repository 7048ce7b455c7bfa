"""Tabulated propagators by integer arithmetic (work queue, on-chip walk) against the plain
conversions of the level-synchronous kernel, bit for bit: differences on and beside the
nodes, beyond both ends, zero of either sign, infinite and NaN, the shortest table and one of
more than 2^21 nodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import medium  # noqa: E402
from workloads.generate import Graph  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg
    return cg


@pytest.mark.parametrize("T", [1, 2, 17, 256, (1 << 21) + 5])
@pytest.mark.parametrize("mode", [0, 1])
def test_integer_and_plain_interpolation_agree(cg, T, mode):
    g = Graph([1, 2, 1], [0, 2, 2], np.array([[0, 1, 0, 1, 0], [0, 2, 0, 0, 1], [1, 3, 0, 1, 0], [2, 3, 0, 0, 1]]), 1, 2)
    rng = np.random.default_rng(T)
    h = 8.0 / T
    nodes = h * rng.integers(-T, T + 1, 400)
    tau = np.concatenate([nodes, np.nextafter(nodes, 99.0), np.nextafter(nodes, -99.0), rng.uniform(-8.0, 8.0, 1000),
                          rng.uniform(-20.0, 20.0, 200), h * rng.uniform(-2.0, 2.0, 200), 10.0 ** rng.uniform(-300, 0, 100),
                          [0.0, -0.0, 8.0, -8.0, 1e300, -1e300, np.inf, -np.inf, np.nan, 5e-324, -5e-324]])
    t = np.stack([tau, np.zeros_like(tau)])   # differences t_1 - t_0 and t_0 - t_1
    t[1, -1] = -0.0
    S = t.shape[1]
    table = rng.normal(size=(1, 2, T + 1))
    gr = cg.Graph.from_workload_graph(g)
    gr.set_propagator_table(table, 8.0)
    gr.set_samples(np.ascontiguousarray(t), np.zeros(1), 8.0, cg.COS_T_HOST, num_samples=S)
    res = {}
    for schedule in (1, 2, 0):
        gr.set_tuning(schedule=schedule)
        out = torch.full((S,), -7.0, dtype=torch.float64, device="cuda")
        gr.evaluate(mode, out=out, want_mean=False)
        torch.cuda.synchronize()
        res[schedule] = out.cpu().numpy()
    np.testing.assert_array_equal(res[2], res[1])
    np.testing.assert_array_equal(res[0], res[1])
    gr.close()


def test_large_tabulated_evaluations_may_be_captured(cg):
    # enough work for the work queue, which a capturing stream does not get
    S, g = 8192, medium(num_samples=1).graph
    rng = np.random.default_rng(1)
    assert g.num_edges * S >= 3e8
    gr = cg.Graph.from_workload_graph(g)
    gr.set_propagator_table(0.3 * rng.normal(size=(g.num_kinds, 2, 65)), 10.0)
    gr.set_samples(torch.from_numpy(rng.uniform(0.0, 10.0, (S, g.num_times))).cuda(), np.zeros(g.num_kinds), 10.0,
                   cg.COS_T_SAMPLE_MAJOR)
    ref, out = (torch.zeros(S, dtype=torch.float64, device="cuda") for _ in range(2))
    gr.evaluate(0, out=ref, want_mean=False)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gr.evaluate(0, out=out, want_mean=False, stream=torch.cuda.current_stream())
    graph.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), ref.cpu().numpy())
    gr.close()


@pytest.mark.parametrize("schedule", [0, 1, 2])
def test_nan_times_give_nan_results(cg, schedule):
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
