"""The launch that puts a call's times and energies into the handle's layout, at the edges
of its tiles (64 samples, 32 times) and of the energies that travel as parameters (64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from workloads.generate import BETA, FaninSpec, make_graph  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,K", [(2, 1), (31, 63), (32, 64), (33, 65), (70, 3)])
def test_times_and_energies_arrive(D, K):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg

    rng = np.random.default_rng(D)
    g = make_graph([1, 5, 9, 1], FaninSpec("uniform", 3), K, D, rng)
    gr = cg.Graph.from_workload_graph(g)
    for S in (1000, 1, 63, 64, 65, 129):   # (the longest first: the buffer holds its times)
        t, eps = rng.uniform(0.0, BETA, (S, D)), rng.uniform(-2.0, 2.0, K)
        R, A = oracle.evaluate(g, eps, BETA, t)
        tt = np.ascontiguousarray(t.T)
        got, out = np.empty((D, S)), torch.empty(S, dtype=torch.float64, device="cuda")
        for src, flags in ((torch.from_numpy(t).cuda(), cg.COS_T_SAMPLE_MAJOR), (t, cg.COS_T_SAMPLE_MAJOR | cg.COS_T_HOST),
                           (torch.from_numpy(tt).cuda(), 0), (tt, cg.COS_T_HOST)):
            gr.set_samples(src, eps, BETA, flags, num_samples=S)
            gr.copy_times(got)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(got, tt)
            gr.evaluate(0, out=out)
            assert np.all(np.abs(out.cpu().numpy() - R) <= 1e-12 * A)
    gr.set_samples_uniform(130, 5, eps, BETA)
    gr.copy_times(got := np.empty((D, 130)))
    torch.cuda.synchronize()
    R, A = oracle.evaluate(g, eps, BETA, np.ascontiguousarray(got.T))
    gr.evaluate(0, out=(out := torch.empty(130, dtype=torch.float64, device="cuda")))
    assert np.all(np.abs(out.cpu().numpy() - R) <= 1e-12 * A)
    gr.close()
