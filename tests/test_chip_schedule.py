"""Row schedule of the on-chip walk (``build_chip`` in csrc/cos_chip.h) on the CPU,
through a host-only probe that walks the schedule with the kernel's index arithmetic
under every launch shape: each row's in-edges appear once, in the graph's order, and
every index stays inside its buffer, against a direct fold over the edge list."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from workloads import complete_layered_graph, medium, tiny
from workloads.generate import FaninSpec, make_graph

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "native", "chip_schedule_probe.cc")
MASK = (1 << 64) - 1


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("needs a C++ compiler")
    exe = str(tmp_path_factory.mktemp("probe") / "chip_schedule_probe")
    subprocess.run([cxx, "-std=c++17", "-O2", SRC, "-o", exe], check=True, capture_output=True)
    return exe


def _csr(g):
    e = g.edges.astype(np.int64)
    off = g.offsets()
    keys = (e[:, 2] * g.num_times + e[:, 3]) * g.num_times + e[:, 4]
    slots, slot = np.unique(keys, return_inverse=True)
    order = np.argsort(e[:, 1], kind="stable")
    level = np.searchsorted(off, e[:, 1], side="right") - 1
    src = e[:, 0] - off[level - 1]
    row_ptr = np.searchsorted(e[order, 1], np.arange(g.num_nodes + 1))
    return row_ptr, src[order], slot.reshape(-1)[order], len(slots)


def _direct(g, row_ptr, src, slot):
    off, val = g.offsets(), [1]
    for l in range(1, g.num_levels):
        new = []
        for r in range(off[l], off[l + 1]):
            v = 0
            for q in range(row_ptr[r], row_ptr[r + 1]):
                v = (v * 1000003 + val[src[q]] * (int(slot[q]) + 1)) & MASK
            new.append(v)
        val = new
    return val[0]


GRAPHS = {
    "tiny": lambda: tiny(num_samples=1).graph,
    "medium": lambda: medium(num_samples=1).graph,
    "two levels": lambda: complete_layered_graph([1, 1], 2, 3, np.random.default_rng(0)),
    "complete, 40 in-edges": lambda: complete_layered_graph([1, 40, 33, 1], 3, 4, np.random.default_rng(1)),
    "fan-in 1..9, odd widths": lambda: make_graph([1, 17, 513, 2047, 31, 1], FaninSpec("uniform", 9), 4, 5,
                                                  np.random.default_rng(2)),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("phase_rows", [1, 2, 4, 8, 16, 32])
def test_schedule_walks_every_in_edge_in_order(probe, name, phase_rows):
    g = GRAPHS[name]()
    row_ptr, src, slot, P = _csr(g)
    text = f"{g.num_levels} {P} {phase_rows}\n" + " ".join(map(str, g.widths)) + "\n" + " ".join(map(str, row_ptr)) + "\n"
    text += "\n".join(f"{a} {b}" for a, b in zip(src, slot)) + "\n"
    r = subprocess.run([probe], input=text, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    got = set(r.stdout.split())
    assert got == {str(_direct(g, row_ptr, src, slot))}


def test_rows_without_in_edges_and_refused_sizes(probe):
    # level widths 1, 3, 1: the middle node has no in-edge and holds 0
    text = "3 2 4\n1 3 1\n0 0 1 1 2 4\n0 0\n0 1\n0 0\n2 1\n"
    r = subprocess.run([probe], input=text, capture_output=True, text=True)
    assert r.returncode == 0 and set(r.stdout.split()) == {str(1 * 1000003 + 2 * 2)}
    wide = "2 70000 4\n1 1\n0 0 1\n0 0\n"          # more slots than 16 bits hold: no schedule
    assert subprocess.run([probe], input=wide, capture_output=True, text=True).stdout.strip() == "none"
