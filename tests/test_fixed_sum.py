"""Integer sums of doubles (csrc/cos_fixed.h), by which every kernel forms the block sums
and means of R(s), against exact rational sums: a sum is rounded once, after bits below
2^-116 of the largest value (2^-96 with room for more values) were dropped."""
import math
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("needs a C++ compiler")
    exe = str(tmp_path_factory.mktemp("probe") / "fixed_sum_probe")
    subprocess.run([cxx, "-std=c++17", "-O1", os.path.join(HERE, "native", "fixed_sum_probe.cc"), "-o", exe], check=True)
    return exe


def sums(probe, sets):
    text = "".join(f"{extra} {len(x)} " + " ".join(struct.pack(">d", v).hex() for v in x) + "\n" for extra, x in sets)
    out = subprocess.run([probe], input=text, check=True, capture_output=True, text=True).stdout.split()
    return [None if o == "range" else struct.unpack(">d", bytes.fromhex(o))[0] for o in out]


def cases():
    rng = np.random.default_rng(7)
    for n in (1, 2, 31, 1024):
        for extra in (0, 20):
            yield extra, rng.standard_normal(n)
            yield extra, rng.standard_normal(n) * 2.0 ** rng.integers(-140, 140, n)      # below and at the dropped bits
            yield extra, -np.abs(rng.standard_normal(n)) * 1e250
            yield extra, np.full(n, float(2**53 - 1))                                     # every mantissa bit, full headroom
            yield extra, -np.full(n, float(2**53 - 1))
    x = rng.standard_normal(512)
    yield 0, np.concatenate([x, -x])                                                      # exact cancellation
    yield 0, np.concatenate([x * 2.0**60, -x * 2.0**60, x])                               # cancellation to the small ones
    for tie in (1.0, 1.0 + 2.0**-52):                                                     # halfway: to even, either way
        yield 0, np.array([tie, 2.0**-53])
        yield 0, np.array([tie, 2.0**-53, 2.0**-100])
        yield 0, np.array([-tie, -(2.0**-53), 2.0**-100])
    yield 0, np.array([2.0 - 2.0**-52, 2.0**-53])                                         # rounds up to the next power
    yield 0, np.array([1.0, 0.0, -0.0, 5e-324])
    yield 0, np.array([2.0**-822, 2.0**-870]) * 1.0                                       # near the low end of the range


def test_sums_are_rounded_once(probe):
    sets = list(cases())
    for (extra, x), got in zip(sets, sums(probe, sets)):
        exact = sum((Fraction(float(v)) for v in x), Fraction(0))
        dropped = len(x) * Fraction(2) ** (extra - 116) * Fraction(float(np.max(np.abs(x)))) * 2
        assert got is not None
        assert abs(Fraction(got) - exact) <= Fraction(math.ulp(got)) / 2 + dropped
        if abs(exact) * Fraction(2) ** -60 > dropped:   # nothing dropped can decide the rounding but at a near tie
            assert got == math.fsum(x) or abs(Fraction(got) - exact) <= Fraction(math.ulp(got)) / 2 * (1 + Fraction(1, 64))


def test_out_of_range_values_are_left_to_the_floating_point_sum(probe):
    sets = [(0, [float("inf"), 1.0]), (0, [float("nan"), 1.0]), (0, [0.0, -0.0]), (0, [5e-324, 1e-300]), (0, [1e308, 1e308])]
    assert sums(probe, sets) == [None] * len(sets)


@pytest.mark.gpu
@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("S", [1, 1023, 1024, 9000, 140001])
def test_means_of_every_kernel_are_the_rounded_sum(S, schedule):
    """The mean of R(s) equals the correctly rounded quotient of the correctly rounded sum
    of the block sums; a block with a value that is not finite takes the floating-point
    sum, whose NaN the mean then is."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_00675_gb300 as cg
    from workloads import tiny
    from workloads.generate import BETA

    g = tiny(num_samples=1).graph
    rng = np.random.default_rng(S)
    t, eps = rng.uniform(0.0, BETA, (S, g.num_times)), rng.uniform(-2.0, 2.0, g.num_kinds)
    gr = cg.Graph.from_workload_graph(g)
    gr.set_tuning(schedule=schedule)
    out = torch.empty(S, dtype=torch.float64, device="cuda")
    for mode in (0, 1):
        gr.set_samples(torch.from_numpy(t).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
        mean = gr.evaluate(mode, out=out)
        x = out.cpu().numpy()
        want = math.fsum(math.fsum(x[b:b + 1024]) for b in range(0, S, 1024)) / S
        # (a sum that lies closer to a halfway point than the dropped bits may round either way)
        assert abs(mean - want) <= 2 * math.ulp(want)
    bad = t.copy()
    bad[S // 2, 0] = float("nan")
    gr.set_samples(torch.from_numpy(bad).cuda(), eps, BETA, cg.COS_T_SAMPLE_MAJOR)
    mean = gr.evaluate(0, out=out)
    assert math.isnan(float(out[S // 2])) and math.isnan(mean)
    gr.close()
