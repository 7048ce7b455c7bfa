"""On-chip evaluations whose arrival words are shared by calls that overlap on the GPU:
such calls may spoil their own results, but the ones that follow, in order, may not see
it (calls of the static entry share one array; calls on one handle share the handle's)."""
import ctypes

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


def test_static_calls_after_overlapping_ones(cg):
    wl, gr, t, t_ld, eps, refs = _setup(cg)
    lib = cg.load_library()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.empty(max(SIZES), dtype=torch.float64, device="cuda") for _ in streams]
    torch.cuda.synchronize()

    def call(S, out, stream, mean):
        rc = lib.cos_evaluate_static(gr.handle, 1, S, t.data_ptr(), t_ld, eps.data_ptr(), float(wl.samples.beta),
                                     out.data_ptr(), mean, stream.cuda_stream)
        assert rc == cg.COS_OK, lib.cos_last_error()

    for _ in range(20):
        for n in range(21):
            call(SIZES[n % 3], outs[n % 2], streams[n % 2], None)
        torch.cuda.synchronize()
        for S in SIZES:
            outs[0].fill_(-1.0)
            torch.cuda.synchronize()
            mean = ctypes.c_double(-1.0)
            call(S, outs[0], streams[0], ctypes.addressof(mean))
            np.testing.assert_array_equal(outs[0][:S].cpu().numpy(), refs[S][0])
            assert mean.value == refs[S][1], S
    gr.close()


def test_evaluations_after_overlapping_ones_on_a_handle(cg):
    wl, gr, _, _, _, refs = _setup(cg)
    S = 20011
    gr.set_samples(torch.from_numpy(wl.samples.t[:S]).cuda(), wl.samples.eps, wl.samples.beta, cg.COS_T_SAMPLE_MAJOR)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.empty(S, dtype=torch.float64, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    for _ in range(20):
        for _ in range(10):
            for out, stream in zip(outs, streams):
                gr.evaluate(1, out=out, want_mean=False, stream=stream)
        torch.cuda.synchronize()
        outs[0].fill_(-1.0)
        torch.cuda.synchronize()
        assert gr.evaluate(1, out=outs[0], stream=streams[0]) == refs[S][1]
        np.testing.assert_array_equal(outs[0].cpu().numpy(), refs[S][0])
        gr.evaluate(1, out=outs[0], want_mean=False, stream=streams[0])   # the mean through the control block
        assert gr.get_result(stream=streams[0]) == refs[S][1]
    gr.close()


def test_replays_of_a_captured_evaluation_between_direct_calls(cg):
    # a captured launch carries one number: its words are cleared by the replay
    wl, gr, _, _, _, refs = _setup(cg)
    S = 20011
    gr.set_samples(torch.from_numpy(wl.samples.t[:S]).cuda(), wl.samples.eps, wl.samples.beta, cg.COS_T_SAMPLE_MAJOR)
    out = torch.empty(S, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gr.evaluate(1, out=out, want_mean=False, stream=torch.cuda.current_stream())
    for n in range(6):
        out.fill_(-1.0)
        if n % 3 == 2:
            assert gr.evaluate(1, out=out) == refs[S][1]
        else:
            graph.replay()
            torch.cuda.synchronize()
            assert gr.get_result() == refs[S][1]
        np.testing.assert_array_equal(out.cpu().numpy(), refs[S][0])
    gr.close()
