"""Plans whose device buffers cannot grow (the allocations are refused on the host while
COS_TEST_FAIL_ALLOC is set): the call reports it, and the next plan, however small, runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import medium  # noqa: E402
from workloads.generate import BETA, FaninSpec, make_graph  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg
    from paper_2501_00675_gb300 import _build
    _build.build()
    cg.load_library()
    return cg


def _member(cg, widths, S, seed):
    rng = np.random.default_rng(seed)
    g = make_graph(widths, FaninSpec("uniform", 3), 4, 5, rng)
    h = cg.Graph.from_workload_graph(g)
    h.set_samples(torch.from_numpy(rng.uniform(0.0, BETA, (S, 5))).cuda(), rng.uniform(-2, 2, 4), BETA, cg.COS_T_SAMPLE_MAJOR)
    return h


@pytest.mark.parametrize("on_chip", [True, False])
def test_batch_after_a_failed_growth(cg, monkeypatch, on_chip):
    members = [_member(cg, [1, 20, 90, 20, 1], 300, 0), _member(cg, [1, 30, 300, 300, 30, 1], 9000, 1),
               _member(cg, [1, 7, 50, 7, 1], 3000, 2)]
    if not on_chip:
        for h in members:
            h.set_tuning(rows_per_warp=8)
    refs = [h.evaluate(1) for h in members]
    batch = cg.Batch(members[:1], 1)
    batch.launch()
    assert batch.results()[0] == refs[0]
    monkeypatch.setenv("COS_TEST_FAIL_ALLOC", "1")
    batch.reset(members)
    with pytest.raises(cg.CosError) as e:
        batch.launch()
    assert e.value.code == cg.COS_ERR_OOM
    monkeypatch.delenv("COS_TEST_FAIL_ALLOC")
    for some in (members[:1], members, members[1:]):
        batch.reset(some)
        want = [refs[members.index(h)] for h in some]
        for _ in range(3):   # direct, capture, replay
            batch.launch()
            assert list(batch.results()) == want
    batch.close()
    for h in members:
        h.close()


def test_work_queue_after_a_failed_growth(cg, monkeypatch):
    h = _member(cg, [1, 20, 90, 20, 1], 300, 3)
    big = _member(cg, [1, 20, 90, 90, 90, 20, 1], 9000, 4)
    for g in (h, big):
        g.set_tuning(schedule=1)
    refs = [g.evaluate(0) for g in (h, big)]
    for g in (h, big):
        g.set_tuning(schedule=2)
    monkeypatch.setenv("COS_TEST_FAIL_ALLOC", "1")
    for g in (h, big):
        with pytest.raises(cg.CosError) as e:
            g.evaluate(0)
        assert e.value.code == cg.COS_ERR_OOM
    monkeypatch.delenv("COS_TEST_FAIL_ALLOC")
    assert [g.evaluate(0) for g in (h, big)] == refs
    h.close()
    big.close()


def test_tabulated_evaluation_without_memory_for_a_plan(cg, monkeypatch):
    # FP64 with tables takes the work queue for its speed alone: without memory for its plan
    # the level-synchronous kernel, which needs none, evaluates as it does from the same samples
    wl = medium(num_samples=8192)
    s = wl.samples
    table = 0.5 * np.tanh(np.random.default_rng(7).normal(size=(wl.graph.num_kinds, 2, 18)))
    gr = cg.Graph.from_workload_graph(wl.graph)
    gr.set_propagator_table(table, s.beta)
    gr.set_samples(torch.from_numpy(s.t).cuda(), s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    assert not gr.info()["on_chip"] & 1 and gr.get_tuning(0)["schedule"] == 2
    out, ref = (torch.empty(8192, dtype=torch.float64, device="cuda") for _ in range(2))
    gr.set_tuning(schedule=1)
    mean = gr.evaluate(0, out=ref)
    gr.set_tuning()
    monkeypatch.setenv("COS_TEST_FAIL_ALLOC", "1")
    assert gr.evaluate(0, out=out) == mean
    assert torch.equal(out, ref)
    monkeypatch.delenv("COS_TEST_FAIL_ALLOC")
    assert gr.evaluate(0, out=out) == mean
    assert torch.equal(out, ref)
    gr.close()
