"""A sample set whose buffers cannot be allocated (more than the device holds; the request
is refused on the host and no sample is read): the handle is left without samples, every
use of them is refused, and the next sample set works."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import tiny  # noqa: E402

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


def _times(gr, cg, t, s, S):      # 6 times of 8 bytes: 3 TB
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR, num_samples=1 << 36)


def _partials(gr, cg, t, s, S):   # two partial sums and an arrival word per 1,024 samples: 400 GB
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_BORROW, num_samples=1 << 44)


def _workspace(gr, cg, t, s, S):  # over 2^30 x 256 bytes
    gr.set_tuning(tile_samples=1 << 30)
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR, num_samples=S)


def _uniform(gr, cg, t, s, S):
    gr.set_samples_uniform(1 << 36, 1, s.eps, s.beta)


@pytest.mark.parametrize("grow", [_times, _partials, _workspace, _uniform])
def test_a_failed_growth_leaves_no_samples(cg, grow):
    wl = tiny(num_samples=700)
    s, S = wl.samples, 700
    t = torch.from_numpy(s.t).cuda()
    gr = cg.Graph.from_workload_graph(wl.graph)
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    out = torch.empty(2 * S, dtype=torch.float64, device="cuda")
    mean = gr.evaluate(0, out=out)
    ref = out[:S].cpu().numpy()
    batch = cg.Batch([gr], 0, [out])
    batch.launch()
    torch.cuda.synchronize()
    with pytest.raises(cg.CosError) as e:
        grow(gr, cg, t, s, S)
    assert e.value.code == cg.COS_ERR_OOM
    for use in (lambda: gr.evaluate(0, out=out), lambda: gr.evaluate(1 | cg.COS_EVAL_ABS, out=out), lambda: batch.launch(),
                lambda: gr.copy_times(out), lambda: gr.autotune(1, out=out)):
        with pytest.raises(cg.CosError) as e:
            use()
        assert e.value.code == cg.COS_ERR_STATE
    gr.set_tuning()
    gr.set_samples(t, s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    out.fill_(-1.0)
    torch.cuda.synchronize()
    assert gr.evaluate(0, out=out) == mean
    np.testing.assert_array_equal(out[:S].cpu().numpy(), ref)
    out.fill_(-1.0)
    batch.launch()
    assert batch.results() == [mean]
    np.testing.assert_array_equal(out[:S].cpu().numpy(), ref)
    batch.close()
    gr.close()


def test_a_refused_sample_set_leaves_the_one_before(cg):
    wl = tiny(num_samples=700)
    s = wl.samples
    t = torch.from_numpy(s.t).cuda()
    gr = cg.Graph.from_workload_graph(wl.graph)
    gr.set_samples(t[:300], s.eps, s.beta, cg.COS_T_SAMPLE_MAJOR)
    mean = gr.evaluate(0)
    for call in (lambda: gr.set_samples(t, s.eps, -1.0, cg.COS_T_SAMPLE_MAJOR),
                 lambda: gr.set_samples_uniform(100000, 1, s.eps, -1.0)):
        with pytest.raises(cg.CosError) as e:
            call()
        assert e.value.code == cg.COS_ERR_INVALID
        assert gr.evaluate(0) == mean
    gr.close()
