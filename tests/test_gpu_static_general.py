"""cos_evaluate_static where the on-chip walk does not serve it: the values of its tiles in
the static array against the oracle, and bit for bit against the allocating entry's
level-synchronous kernel."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from workloads import medium  # noqa: E402
from workloads.generate import BETA, FaninSpec, make_graph  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5}


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg
    from paper_2501_00675_gb300 import _build
    _build.build()
    cg.load_library()
    return cg


def _medium(S):
    wl = medium(num_samples=S)
    return wl.graph, wl.samples.eps, wl.samples.t


def _wide(S):   # several tiles: 64 MiB hold 64 samples in FP64, 128 in FP32
    rng = np.random.default_rng(17)
    g = make_graph([1, 200, 40000, 40000, 200, 1], FaninSpec("uniform", 3), 6, 4, rng)
    return g, rng.uniform(-2.0, 2.0, 6), rng.uniform(0.0, BETA, (S, 4))


@pytest.mark.parametrize("mode,case,S", [(0, _medium, 16384), (0, _wide, 1100), (1, _wide, 3001), (2, _wide, 3001)])
def test_static_values_off_chip(cg, mode, case, S):
    g, eps, t = case(S)
    lib = cg.load_library()
    gr = cg.Graph.from_workload_graph(g)
    gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    assert not gr.info()["on_chip"] >> mode & 1
    dtype = torch.int64 if mode == 2 else torch.float64
    gr.set_tuning(schedule=1)
    ref = torch.empty(S, dtype=dtype, device="cuda")
    ref_mean = gr.evaluate(mode, out=ref)
    gr.set_tuning()
    t_ld = (S + 127) // 128 * 128
    tdev = torch.zeros((t.shape[1], t_ld), dtype=torch.float64, device="cuda")
    tdev[:, :S] = torch.from_numpy(np.ascontiguousarray(t.T)).cuda()
    eps_dev = torch.from_numpy(eps).cuda()
    rows = min(S, 64)
    for _ in range(2):
        out = torch.full((S,), -3, dtype=dtype, device="cuda")
        mean = ctypes.c_double(0.0)
        rc = lib.cos_evaluate_static(gr.handle, mode, S, tdev.data_ptr(), t_ld, eps_dev.data_ptr(), BETA, out.data_ptr(),
                                     ctypes.addressof(mean), torch.cuda.current_stream().cuda_stream)
        assert rc == cg.COS_OK, lib.cos_last_error()
        assert torch.equal(out, ref) and mean.value == ref_mean
        got = out[:rows].cpu().numpy()
        if mode == 2:
            assert np.all(got == gr.info()["count"])
        else:
            R, A = oracle.evaluate(g, eps, BETA, t[:rows])
            assert np.all(np.abs(got - R) <= TOL[mode] * A)
    gr.close()
