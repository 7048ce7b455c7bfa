"""Forms of the on-chip walk that the shapes of test_gpu_chip.py do not reach: levels that go
through TMEM in pieces of 4 and 8 bytes, FP64 wherever it is meant to run on chip, members
of a batch that do run there, launches of two streams on one SM, energies of a capturing
stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_chip import ABS, GRAPHS, _both, _evaluate, _inputs, _on_chip, cg  # noqa: E402, F401
from workloads import medium, tiny  # noqa: E402
from workloads.generate import BETA, FaninSpec, make_graph  # noqa: E402

pytestmark = pytest.mark.gpu


# Two neighbouring levels, each more than half of what 227 KB leave: the second goes through
# TMEM.  30,000 rows: FP32 in rows and pieces of 4 bytes; 15,000: rows of 8 (FP32 and counts in
# pieces of 8, R and A in pieces of 4); 7,500: rows of 16 (R and A in pieces of 8).
@pytest.mark.parametrize("width,modes", [(30000, (1,)), (15000, (0, 1, 2, 1 | ABS)), (7500, (0, 2, 1 | ABS))])
def test_narrow_rows_through_staged_levels(cg, width, modes):  # noqa: F811
    g = make_graph([1, 100, width, width - 77, 50, 1], FaninSpec("uniform", 3), 6, 4, np.random.default_rng(width))
    eps, t = _inputs(g, 301)
    gr = cg.Graph.from_workload_graph(g)
    gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    for mode in modes:
        assert _on_chip(cg, gr, mode), mode
    gr.close()
    _both(cg, g, eps, t, modes, oracle_rows=8)


# (the exponentials of 300 kinds and 1,025 samples are left to the general kernels)
@pytest.mark.parametrize("name,S", [(n, S) for n in GRAPHS for S in (31, 1025) if (n, S) != ("300 kinds", 1025)])
def test_fp64_runs_on_chip(cg, name, S):  # noqa: F811
    g = GRAPHS[name](np.random.default_rng(3))
    eps, t = _inputs(g, S)
    gr = cg.Graph.from_workload_graph(g)
    gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    assert _on_chip(cg, gr, 0)
    gr.close()


@pytest.mark.parametrize("mode", [0, 1, 2, 1 | ABS])
def test_batch_members_that_run_on_chip(cg, mode):  # noqa: F811
    rng = np.random.default_rng(21)
    graphs, outs, refs = [], [], []
    for n, (widths, S) in enumerate([([1, 4, 1], 5000), ([1, 60, 60, 1], 3000), ([1, 30, 700, 30, 1], 400), ([1, 64, 1], 2048)]):
        g = make_graph(widths, FaninSpec("uniform", 4), 5, 4, rng)
        eps, t = _inputs(g, S, seed=n)
        h = cg.Graph.from_workload_graph(g)
        h.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
        h.set_tuning(schedule=1)
        refs.append(_evaluate(h, mode, S))
        if n < 3:
            h.set_tuning()
        graphs.append(h)
        outs.append(torch.empty(refs[-1][0].shape, dtype=torch.int64 if mode == 2 else torch.float64, device="cuda"))
    b = cg.Batch(graphs, mode, outs)
    for _ in range(4):   # direct launch, capture, replays
        for o in outs:
            o.fill_(-1)
        b.launch()
        means = b.results()
        assert b.info() == {"members": 4, "on_chip": 3,
                            "on_chip_values": 6 * 5000 + 122 * 3000 + 762 * 400}
        for o, m, ref in zip(outs, means, refs):
            np.testing.assert_array_equal(o.cpu().numpy(), ref[0])
            assert tuple(np.atleast_1d(m)) == tuple(np.atleast_1d(ref[1]))
    b.close()
    for h in graphs:
        h.close()


def test_two_streams_share_the_sms(cg):  # noqa: F811
    """Evaluations of two handles on two streams at once, one with levels through TMEM and one
    whose CTAs share an SM: each equals its evaluation alone."""
    wl = medium(num_samples=3000)
    a = cg.Graph.from_workload_graph(wl.graph)
    small = GRAPHS["widths 63, 64, 65, 129"](np.random.default_rng(3))
    b = cg.Graph.from_workload_graph(small)
    c = a.share()
    eps, t = _inputs(small, 40000)
    for h in (a, c):
        h.set_samples(torch.from_numpy(wl.samples.t).cuda(), wl.samples.eps, wl.samples.beta, cg.COS_T_SAMPLE_MAJOR)
    b.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    handles, sizes = (a, b, c), (3000, 40000, 3000)
    for h in handles:
        assert _on_chip(cg, h, 1)
    refs = [_evaluate(h, 1, S)[0] for h, S in zip(handles, sizes)]
    streams = [torch.cuda.Stream() for _ in handles]
    outs = [torch.full((S,), -1.0, dtype=torch.float64, device="cuda") for S in sizes]
    torch.cuda.synchronize()
    for _ in range(20):
        for h, o, st in zip(handles, outs, streams):
            h.evaluate(1, out=o, want_mean=False, stream=st)
    torch.cuda.synchronize()
    for o, ref in zip(outs, refs):
        np.testing.assert_array_equal(o.cpu().numpy(), ref)
    for h in (c, a, b):
        h.close()


def test_captured_sample_sets_read_the_energies_at_replay(cg):  # noqa: F811
    # on a capturing stream the energies are a copy node of the host's array, which each replay
    # reads; elsewhere they travel with the launch
    wl = tiny(num_samples=900)
    s = wl.samples
    t = torch.from_numpy(s.t).cuda()
    gr = cg.Graph.from_workload_graph(wl.graph)
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    ref, _ = _evaluate(gr, 1, 900)
    gr.set_samples(t, -0.5 * s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    other, _ = _evaluate(gr, 1, 900)
    out = torch.zeros(900, dtype=torch.float64, device="cuda")
    eps = torch.from_numpy(s.eps.copy()).pin_memory().numpy()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gr.set_samples(t, eps, s.beta, cg.COS_T_SAMPLE_MAJOR, stream=torch.cuda.current_stream())
        gr.evaluate(1, out=out, want_mean=False, stream=torch.cuda.current_stream())
    for scale, want in ((1.0, ref), (-0.5, other), (1.0, ref)):
        eps[:] = scale * s.eps
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    gr.close()


@pytest.mark.parametrize("S,on_chip", [(4 << 30, True), (8 << 30, False)])
def test_chunks_beyond_32_bits_stay_off_chip(cg, S, on_chip):  # noqa: F811
    # levels of 8,000 rows: four FP32 samples per chunk (nothing is evaluated: the times, borrowed,
    # are not there)
    g = make_graph([1, 100, 8000, 8000, 8000, 100, 1], FaninSpec("uniform", 4), 6, 1, np.random.default_rng(2))
    gr = cg.Graph.from_workload_graph(g)
    t = torch.zeros(128, dtype=torch.float64, device="cuda")
    gr.set_samples(t, np.zeros(6), BETA, cg.COS_T_BORROW, num_samples=S)
    assert _on_chip(cg, gr, 1) == on_chip
    gr.close()
