"""On-chip walk against the general kernels and the oracle at the sizes where it can go
wrong: levels around its groups of 64 rows, more than four in-edges per row, rows without
in-edges, two levels, a wide level before the sink, many kinds (several passes of
exponentials), ragged sample counts, few and many blocks of samples, tabulated
propagators, |factor| walks, energies and times outside the float-float range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from workloads import complete_layered_graph, medium, tiny  # noqa: E402
from workloads.generate import BETA, FaninSpec, Graph, make_graph  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5}
ABS = 16


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg
    from paper_2501_00675_gb300 import _build
    _build.build()
    cg.load_library()
    return cg


def _on_chip(cg, gr, mode):
    info = np.zeros(11, dtype=np.int64)
    cg.load_library().cos_graph_info(gr.handle, info.ctypes.data, 11)
    return bool(info[10] >> {0: 0, 1: 1, 2: 2, 1 | ABS: 4}[mode] & 1)


def _evaluate(gr, mode, S, call="evaluate"):
    n = 2 * S if mode & ABS else S
    out = torch.full((n,), -7, dtype=torch.int64 if mode == 2 else torch.float64, device="cuda")
    mean = getattr(gr, call)(mode, out=out, **({"allow_overflow": True} if call == "evaluate" else {}))
    return out.cpu().numpy(), mean


def _both(cg, g, eps, t, modes, call="evaluate", table=None, oracle_rows=64):
    """Every mode on chip (twice: the counters are left as they were found) equals the
    level-synchronous kernel bit for bit; the first samples equal the oracle."""
    S = t.shape[0]
    gr = cg.Graph.from_workload_graph(g)
    if table is not None:
        gr.set_propagator_table(table, BETA)
    gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    for mode in modes:
        gr.set_tuning()
        if mode == 0 and not _on_chip(cg, gr, mode):
            continue   # (FP64: the general kernel may be the faster one, which it then is)
        assert _on_chip(cg, gr, mode), (mode, S)
        first, again = _evaluate(gr, mode, S, call), _evaluate(gr, mode, S, call)
        gr.set_tuning(schedule=1)
        ref = _evaluate(gr, mode, S, call)
        for got in (first, again):
            np.testing.assert_array_equal(got[0], ref[0])
            assert got[1] == ref[1]
        if mode in TOL and table is None and call == "evaluate":
            R, A = oracle.evaluate(g, eps, BETA, t[:oracle_rows])
            assert np.all(np.abs(first[0][:oracle_rows] - R) <= TOL[mode] * A)
    gr.close()


def _inputs(g, S, seed=0, spread=2.0):
    rng = np.random.default_rng(seed)
    return rng.uniform(-spread, spread, g.num_kinds), rng.uniform(0.0, BETA, (S, g.num_times))


GRAPHS = {
    "tiny": lambda r: tiny(num_samples=1).graph,
    "two levels": lambda r: complete_layered_graph([1, 1], 2, 3, r),
    "widths 63, 64, 65, 129": lambda r: make_graph([1, 63, 64, 65, 129, 64, 1], FaninSpec("uniform", 4), 3, 5, r),
    "fan-in 1..9": lambda r: make_graph([1, 9, 200, 333, 40, 1], FaninSpec("uniform", 9), 4, 5, r),
    "40 in-edges": lambda r: complete_layered_graph([1, 40, 33, 1], 3, 4, r),
    "100 rows before the sink": lambda r: make_graph([1, 30, 100, 1], FaninSpec("uniform", 3), 5, 3, r),
    "one time": lambda r: make_graph([1, 5, 70, 3, 1], FaninSpec("uniform", 2), 7, 1, r),
    "300 kinds": lambda r: make_graph([1, 20, 90, 20, 1], FaninSpec("uniform", 4), 300, 12, r),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("S", [1, 31, 1025])
def test_graph_shapes_match_the_general_kernel(cg, name, S):
    g = GRAPHS[name](np.random.default_rng(3))
    _both(cg, g, *_inputs(g, S), modes=(0, 1, 2, 1 | ABS))


def test_rows_without_in_edges_and_loop_signs(cg):
    # level 1 holds 3 nodes; node 2 has no in-edge (value 0); one edge closes a fermion loop
    sign = 1 << 30
    e = np.array([[0, 1, 0, 0, 1], [0, 3, 1 | sign, 1, 0], [1, 4, 1, 1, 1], [2, 4, 0, 0, 1], [3, 4, 0 | sign, 0, 0]], np.int32)
    g = Graph(np.array([1, 3, 1]), np.array([0, 2, 3]), e, 2, 2)
    _both(cg, g, *_inputs(g, 200), modes=(0, 1, 2, 1 | ABS))


@pytest.mark.parametrize("S", [70001, 9000])
def test_many_blocks_of_samples(cg, S):
    g = make_graph([1, 40, 300, 40, 1], FaninSpec("geometric", 6, 0.31), 8, 4, np.random.default_rng(4))
    _both(cg, g, *_inputs(g, S), modes=(1, 2, 1 | ABS))


def test_medium_graph_through_staged_levels(cg):
    w = medium(num_samples=1100)
    _both(cg, w.graph, w.samples.eps, w.samples.t, modes=(0, 1, 2, 1 | ABS))


def test_wide_levels_with_narrow_rows(cg):
    for width in (9000, 30000):   # two samples and one per chunk in FP32
        g = make_graph([1, 100, width, 50, 1], FaninSpec("uniform", 3), 6, 4, np.random.default_rng(5))
        _both(cg, g, *_inputs(g, 300), modes=(1,))


def test_tabulated_propagators(cg):
    g = GRAPHS["widths 63, 64, 65, 129"](np.random.default_rng(6))
    table = 0.5 * np.tanh(np.random.default_rng(7).normal(size=(g.num_kinds, 2, 18)))
    _both(cg, g, *_inputs(g, 777), modes=(0, 1, 1 | ABS), table=table)


def test_absolute_factors(cg):
    g = GRAPHS["fan-in 1..9"](np.random.default_rng(8))
    _both(cg, g, *_inputs(g, 500), modes=(0, 1), call="evaluate_abs")


def test_energies_outside_the_float_float_range(cg):
    # |eps| * beta up to 50 in some kinds: their exponentials are formed in double
    g = GRAPHS["widths 63, 64, 65, 129"](np.random.default_rng(9))
    _both(cg, g, *_inputs(g, 600, spread=5.0), modes=(0, 1))


def test_times_outside_the_period(cg):
    # one sample in ten outside [-beta, beta]: its chunk is formed in double (within 1e-5 of
    # the sum of |path| values of the oracle, as every FP32 result)
    g = GRAPHS["fan-in 1..9"](np.random.default_rng(10))
    eps, t = _inputs(g, 400, seed=11)
    t[::10, 1] += 2.0 * BETA
    gr = cg.Graph.from_workload_graph(g)
    gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    assert _on_chip(cg, gr, 1)
    out, _ = _evaluate(gr, 1, 400)
    R, A = oracle.evaluate(g, eps, BETA, t)
    assert np.all(np.abs(out - R) <= TOL[1] * A)
    gr.close()


def test_batch_members_on_and_off_chip(cg):
    """A batch whose members run on chip in several launch shapes, and one that does not
    (a launch shape of its own): every member equals its single evaluation."""
    rng = np.random.default_rng(12)
    graphs, outs, refs = [], [], []
    for n, (widths, S) in enumerate([([1, 4, 1], 5000), ([1, 300, 300, 1], 3000), ([1, 30, 5000, 30, 1], 700),
                                     ([1, 50, 50, 1], 1), ([1, 64, 1], 2048)]):
        g = make_graph(widths, FaninSpec("uniform", 4), 5, 4, rng)
        eps, t = _inputs(g, S, seed=n)
        h = cg.Graph.from_workload_graph(g)
        h.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
        if n == 4:
            h.set_tuning(rows_per_warp=8)
        assert _on_chip(cg, h, 1) == (n != 4)
        refs.append(_evaluate(h, 1, S))
        graphs.append(h)
        outs.append(torch.empty(S, dtype=torch.float64, device="cuda"))
    b = cg.Batch(graphs, 1, outs)
    for _ in range(4):   # direct launch, capture, replays
        for o in outs:
            o.fill_(-1.0)
        b.launch()
        means = b.results()
        for o, m, ref in zip(outs, means, refs):
            np.testing.assert_array_equal(o.cpu().numpy(), ref[0])
            assert m == ref[1]
    b.close()
    for h in graphs:
        h.close()


def test_capture_without_mean(cg):
    # an evaluation without mean_out may be captured into a CUDA graph and replayed
    w = tiny(num_samples=900)
    gr = cg.Graph.from_workload_graph(w.graph)
    gr.set_samples(torch.from_numpy(w.samples.t).cuda(), w.samples.eps, w.samples.beta, cg.COS_T_SAMPLE_MAJOR)
    assert _on_chip(cg, gr, 0)
    ref, mean = _evaluate(gr, 0, 900)
    out = torch.zeros(900, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gr.evaluate(0, out=out, want_mean=False, stream=torch.cuda.current_stream())
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
        assert gr.get_result() == mean
    gr.close()
