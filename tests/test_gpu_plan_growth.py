"""Plans whose device buffers cannot grow (the allocations are refused on the host while
COS_TEST_FAIL_ALLOC is set): the call reports it, and the next plan, however small, runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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
