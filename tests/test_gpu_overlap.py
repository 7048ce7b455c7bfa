"""On-chip evaluations whose arrival words are shared by calls that overlap on the GPU
(calls of the static entry share one array; calls on one handle share the handle's)."""
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


SIZES = (300, 20011, 9000)   # one block of samples (summed at the end), and blocks counted one by one


def _setup(cg):
    wl = tiny(num_samples=max(SIZES))
    gr = cg.Graph.from_workload_graph(wl.graph)
    t_ld = (max(SIZES) + 127) // 128 * 128
    t = torch.zeros((wl.samples.t.shape[1], t_ld), dtype=torch.float64, device="cuda")
    t[:, :max(SIZES)] = torch.from_numpy(np.ascontiguousarray(wl.samples.t.T)).cuda()
    eps = torch.from_numpy(np.ascontiguousarray(wl.samples.eps, dtype=np.float64)).cuda()
    refs = {}
    for S in SIZES:   # the general kernel
        gr.set_samples(torch.from_numpy(wl.samples.t[:S]).cuda(), wl.samples.eps, wl.samples.beta, cg.COS_T_SAMPLE_MAJOR)
        gr.set_tuning(schedule=1)
        out = torch.empty(S, dtype=torch.float64, device="cuda")
        mean = gr.evaluate(1, out=out)
        refs[S] = (out.cpu().numpy(), mean)
        gr.set_tuning()
        assert gr.info()["on_chip"] >> 1 & 1
    return wl, gr, t, t_ld, eps, refs


def test_overlapping_evaluations_on_a_handle_end(cg):
    # what they return is undefined; that they return is not
    wl, gr, _, _, _, _ = _setup(cg)
    S = 20011
    gr.set_samples(torch.from_numpy(wl.samples.t[:S]).cuda(), wl.samples.eps, wl.samples.beta, cg.COS_T_SAMPLE_MAJOR)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.empty(S, dtype=torch.float64, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    for _ in range(200):
        for out, stream in zip(outs, streams):
            gr.evaluate(1, out=out, want_mean=False, stream=stream)
    torch.cuda.synchronize()
    gr.close()
