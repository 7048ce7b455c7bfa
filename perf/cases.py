"""Evaluations that programs ask of this library, with inputs, work and 64-bit values.

A case is one pass of a Monte Carlo program through the public entry points: attach a
batch of vertex times to a resident graph and evaluate it, launch a batch of graphs,
advance Metropolis walkers.  Graphs are the synthetic leveled graphs of `workloads`
(tiny, medium, large, batched, and the serving pool's, by expansion order and node
count); times and energies are drawn from the seed on the GPU.

Fields of a case
  entry    "evaluate" (cos_set_samples + cos_evaluate), "static" (cos_evaluate_static),
           "batch" (cos_batch_launch + cos_batch_results), "mc" (cos_mc_run + readback)
  graph    "tiny", "medium", "large", or "order" with order, nodes, fanin and graph_seed;
           for "batch": graphs, nodes, samples bound a mix drawn with graph_seed
  mode     "fp64", "mixed" (FP32 bulk, FP64 sink and sample sums), "count" (int64)
  abs      also accumulate A(s), the sum of |path| values, in the same walk
  table    intervals of user-tabulated propagators (0: the free-fermion formula)
  samples  Monte Carlo samples (or walkers) of one pass
  times    "device" ([S][D] on the GPU), "host" ([S][D], page-locked), "borrow" ([D][t_ld]
           used in place), "uniform" (drawn by the library from a seed)
  mean     the program waits for the mean over samples
"""
import ctypes
import functools
import math

import numpy as np
import torch

import paper_2501_00675_gb300 as cg
from workloads import generate as wg

BETA = wg.BETA
MODES = {"fp64": cg.COS_MODE_FP64, "mixed": cg.COS_MODE_FP32_MIXED, "count": cg.COS_MODE_COUNT_I64}
FANINS = {"uniform3": wg.FaninSpec("uniform", 3), "uniform4": wg.FaninSpec("uniform", 4),
          "geometric6": wg.FaninSpec("geometric", 6, 0.31)}


def _case(name, entry, graph, mode, samples, **more):
    c = dict(name=name, entry=entry, graph=graph, mode=mode, samples=samples, abs=0, table=0, times="device", mean=False)
    c.update(more)
    return c


def listed():
    return [
        # one small evaluation whose mean a program waits for: latency and launches count
        _case("tiny_fp64_mean", "evaluate", "tiny", "fp64", 1024, mean=True),
        # a latency-bound loop that may not allocate; a sample count that fills no block
        _case("tiny_mixed_static", "static", "tiny", "mixed", 1000, times="borrow"),
        # a low-order graph (2n+2 = 6 levels), its times coming from a host program, odd sizes
        _case("order2_mixed_host", "evaluate", "order", "mixed", 10007, order=2, nodes=1000, fanin="geometric6",
              graph_seed=5, times="host", mean=True),
        # the medium graph in double precision: the ordinary Monte Carlo batch
        _case("medium_fp64", "evaluate", "medium", "fp64", 65536),
        # the same batch in FP32 bulk
        _case("medium_mixed", "evaluate", "medium", "mixed", 65536),
        # exact path counting on the same lanes
        _case("medium_count", "evaluate", "medium", "count", 65536),
        # R(s) with its error scale A(s) in one walk, a ragged batch
        _case("medium_mixed_abs", "evaluate", "medium", "mixed", 50001, abs=1),
        # propagators given as numbers
        _case("medium_fp64_table", "evaluate", "medium", "fp64", 16384, table=256),
        # Metropolis walkers: a block of four steps, then readback of walkers and tallies
        _case("medium_fp64_walkers", "mc", "medium", "fp64", 16384, steps=4),
        # a typical serving request: order 6, 100k nodes, times drawn on the device
        _case("order6_mixed_uniform", "evaluate", "order", "mixed", 30000, order=6, nodes=100000, fanin="geometric6",
              graph_seed=6, times="uniform"),
        # the large graph (2.1M nodes, levels of 262,144): node values far beyond L2
        _case("large_mixed", "evaluate", "large", "mixed", 131072),
        # graphs of uneven size and sample count in one launch
        _case("batch_mixed", "batch", "mix", "mixed", 65536, graphs=32, nodes=200000, graph_seed=3, times="borrow",
              mean=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["evaluate"] * 7 + ["static", "batch", "mc"])
    if entry == "batch":
        return dict(entry="batch", graph="mix", mode=rng.choice(["mixed", "fp64"]), samples=_log_int(rng, 8192, 65536),
                    graphs=rng.randint(4, 32), nodes=_log_int(rng, 2e3, 1e5), graph_seed=rng.randrange(1 << 16), abs=0,
                    table=0, times="borrow", mean=True)
    order = rng.randint(2, 8)
    nodes = _log_int(rng, 100, 5000 if entry == "static" else 300000)
    c = dict(entry=entry, graph="order", order=order, nodes=nodes, fanin=rng.choice(["uniform4", "geometric6"]),
             graph_seed=rng.randrange(1 << 16), mode=rng.choice(["fp64", "mixed", "mixed", "count"]), abs=0, table=0,
             times="device", mean=rng.random() < 0.3)
    samples = _log_int(rng, 1, 131072)
    c["samples"] = max(1, min(samples, int(5e10 / (2.5 * nodes))))
    if entry == "static":
        c.update(times="borrow", mean=False, samples=min(c["samples"], 8192))
    elif entry == "mc":
        c.update(mode="fp64", mean=False, steps=rng.randint(1, 4), samples=max(64, min(c["samples"], 32768) // 4))
    else:
        c["times"] = rng.choice(["device", "device", "host", "borrow", "uniform"])
        if c["mode"] != "count":
            c["abs"] = int(rng.random() < 0.2)
            c["table"] = rng.choice([0, 0, 0, rng.randint(16, 1024)])
    return c


# ---------------------------------------------------------------------------- graphs


@functools.lru_cache(maxsize=64)
def _graph(kind, order, nodes, fanin, graph_seed, seed):
    if kind == "tiny":
        return wg.tiny(seed=0 + seed, num_samples=1).graph
    if kind == "medium":
        return wg.medium(seed=1 + seed, num_samples=1).graph
    if kind == "large":
        return wg.large(seed=2 + seed, num_samples=1).graph
    levels = 2 * order + 2
    return wg.make_graph(wg.widths_for_target(levels, nodes), FANINS[fanin], 32, levels,
                         np.random.default_rng(graph_seed + seed))


def _graph_of(case, seed=0):
    """The case's graph.  A count depends on the graph alone, so there every seed has its own."""
    return _graph(case["graph"], case.get("order", 0), case.get("nodes", 0), case.get("fanin", ""),
                  case.get("graph_seed", 0), seed if case["mode"] == "count" else 0)


@functools.lru_cache(maxsize=4)
def _mix(graphs, nodes, samples, graph_seed):
    """Graphs of order 2..8 with log-uniform node and sample counts (the batched workload's)."""
    rng = np.random.default_rng(graph_seed)
    out = []
    for _ in range(graphs):
        levels = 2 * int(rng.integers(2, 9)) + 2
        n = int(round(math.exp(rng.uniform(math.log(1e3), math.log(max(nodes, 1001))))))
        s = int(round(math.exp(rng.uniform(math.log(4096), math.log(max(samples, 4097))))))
        out.append((wg.make_graph(wg.widths_for_target(levels, n), FANINS["uniform4"], 16, levels, rng), s))
    return out


def _mix_of(case):
    return _mix(case["graphs"], case["nodes"], case["samples"], case["graph_seed"])


# ---------------------------------------------------------------------------- inputs


def _inputs(num_kinds, num_times, samples, seed):
    """eps_k ~ U[-2, 2] (host) and times t ~ U[0, beta) as [S][D] on the GPU."""
    eps = np.random.default_rng([seed, 1]).uniform(-2.0, 2.0, size=num_kinds)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    t = BETA * torch.rand((samples, num_times), generator=gen, dtype=torch.float64, device="cuda")
    return eps, t


def _tables(num_kinds, intervals, seed):
    """Smooth propagators with a jump at tau = 0: [K][2][T+1] on tau >= 0, then tau < 0."""
    rng = np.random.default_rng([seed, 2])
    x = np.linspace(0.0, 1.0, intervals + 1)
    a, b, f = (rng.uniform(0.2, 1.0, size=(num_kinds, 2, 1)) for _ in range(3))
    sign = np.array([-1.0, 1.0]).reshape(1, 2, 1)
    return sign * (a * np.exp(-2.0 * b * x) + 0.2 * np.cos(6.0 * f * x))


def _padded(t):
    """[D][t_ld] copy of t [S][D], t_ld = S rounded up to 128."""
    s, d = t.shape
    buf = torch.zeros((d, max(128, (s + 127) // 128 * 128)), dtype=torch.float64, device="cuda")
    buf[:, :s] = t.T
    return buf


def prepare(case, seed):
    mode = MODES[case["mode"]] | (cg.COS_EVAL_ABS if case["abs"] else 0)
    dtype = torch.int64 if case["mode"] == "count" else torch.float64
    st = {"case": case, "mode": mode}
    if case["entry"] == "batch":
        st["graphs"], st["keep"], st["outs"] = [], [], []
        for n, (g, s) in enumerate(_mix_of(case)):
            eps, t = _inputs(g.num_kinds, g.num_times, s, seed + 1000 * n)
            buf = _padded(t)
            h = cg.Graph.from_workload_graph(g)
            h.set_samples(buf, eps, BETA, cg.COS_T_BORROW, num_samples=s)
            st["graphs"].append(h)
            st["keep"].append(buf)
            st["outs"].append(torch.empty(s, dtype=dtype, device="cuda"))
        st["batch"] = cg.Batch(st["graphs"], mode, st["outs"])
        return st
    g = _graph_of(case, seed)
    s = case["samples"]
    h = st["graph"] = cg.Graph.from_workload_graph(g)
    if case["table"]:
        h.set_propagator_table(_tables(g.num_kinds, case["table"], seed), BETA)
    st["eps"], t = _inputs(g.num_kinds, g.num_times, s, seed)
    st["out"] = torch.empty(s * (2 if case["abs"] else 1), dtype=dtype, device="cuda")
    if case["entry"] == "mc":
        h.set_samples(t, st["eps"], BETA, cg.COS_T_SAMPLE_MAJOR)
        st["walkers"] = cg.Metropolis(h, mode, seed)
        st["times_out"] = torch.empty((g.num_times, s), dtype=torch.float64, device="cuda")
    elif case["entry"] == "static":
        st["t"] = _padded(t)
        st["eps_dev"] = torch.from_numpy(st["eps"]).cuda()
    elif case["times"] == "host":
        st["t"], st["flags"] = t.cpu().pin_memory(), cg.COS_T_HOST | cg.COS_T_SAMPLE_MAJOR
    elif case["times"] == "borrow":
        st["t"], st["flags"] = _padded(t), cg.COS_T_BORROW
    elif case["times"] == "uniform":
        st["seed"] = seed
    else:
        st["t"], st["flags"] = t, cg.COS_T_SAMPLE_MAJOR
    return st


def run(st):
    case, mode = st["case"], st["mode"]
    if case["entry"] == "batch":
        st["batch"].launch()
        return {"values": st["outs"], "means": st["batch"].results()}
    h, out, s = st["graph"], st["out"], case["samples"]
    if case["entry"] == "mc":
        w = st["walkers"]
        w.run(case["steps"])
        tallies = w.stats()
        h.copy_times(st["times_out"])
        return {"values": w.values(out), "times": st["times_out"], "tallies": tallies}
    if case["entry"] == "static":
        t = st["t"]
        rc = cg.load_library().cos_evaluate_static(
            h.handle, mode, s, t.data_ptr(), t.shape[1], st["eps_dev"].data_ptr(), ctypes.c_double(BETA), out.data_ptr(),
            None, torch.cuda.current_stream().cuda_stream)
        if rc != cg.COS_OK:
            raise RuntimeError(f"cos_evaluate_static: {rc}")
        return {"values": out}
    if case["times"] == "uniform":
        h.set_samples_uniform(s, st["seed"], st["eps"], BETA)
    else:
        h.set_samples(st["t"], st["eps"], BETA, st["flags"], num_samples=s)
    mean = h.evaluate(mode, out=out, want_mean=case["mean"])
    return {"values": out, "mean": mean} if case["mean"] else {"values": out}


# ---------------------------------------------------------------------------- work


def _graph_work(g, case, samples):
    """Inputs read once (times, energies or tables, edges) and outputs written once; one
    multiply-add per edge and sample (an addition when counting), one more for A."""
    values = 2 if case["abs"] else 1
    edge_bytes = 8 * g.num_edges + 4 * (g.num_nodes + 1)
    times = 0 if case["mode"] == "count" else 8 * g.num_times * samples
    tables = 8 * g.num_kinds * (2 * (case["table"] + 1) if case["table"] else 1)
    flops = (1 if case["mode"] == "count" else 2 * values) * g.num_edges * samples
    return edge_bytes + times + tables + 8 * values * samples, flops


def work(case):
    if case["entry"] == "batch":
        parts = [_graph_work(g, case, s) for g, s in _mix_of(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _graph_work(_graph_of(case), case, case["samples"])
    n = case.get("steps", 1)
    return {"bytes": b * n, "flops": f * n}


# ---------------------------------------------------------------------------- 64-bit values


def _levels(g):
    """Per level: rows in order of decreasing fan-in, and for r = 0, 1, ... the parents and
    slots of the rows' r-th in-edges; slots index the distinct (kind with sign, i, j)."""
    e = g.edges.astype(np.int64)
    slots, slot_of = np.unique(e[:, 2:5], axis=0, return_inverse=True)
    slot_of = slot_of.reshape(-1)
    off, first, out = g.offsets(), 0, []
    for l in range(1, g.num_levels):
        n = int(g.edge_counts[l])
        src, dst, slot = e[first:first + n, 0] - off[l - 1], e[first:first + n, 1] - off[l], slot_of[first:first + n]
        first += n
        by_dst = np.argsort(dst, kind="stable")
        src, dst, slot = src[by_dst], dst[by_dst], slot[by_dst]
        w = int(g.widths[l])
        deg = np.bincount(dst, minlength=w)
        start = np.concatenate([[0], np.cumsum(deg)[:-1]])
        rows = np.argsort(-deg, kind="stable")
        ranks = []
        for r in range(int(deg.max()) if w else 0):
            at = start[rows[:int((deg > r).sum())]] + r
            ranks.append((torch.from_numpy(src[at]).cuda(), torch.from_numpy(slot[at]).cuda()))
        out.append((torch.from_numpy(rows).cuda(), ranks, w))
    return slots, out


def _factors(slots, t, eps, tables):
    """G of every slot for times t [D][s], in 64 bits."""
    k, i, j = (torch.from_numpy(np.ascontiguousarray(slots[:, c])).cuda() for c in range(3))
    sign = torch.where((k & (1 << 30)) != 0, -1.0, 1.0).double()[:, None]
    k = k & ((1 << 30) - 1)
    tau = t[i] - t[j]
    pos = tau >= 0
    if tables is None:
        e = torch.from_numpy(eps).cuda()[k][:, None]
        return sign * torch.where(pos, -torch.exp(-e * tau), torch.exp(-e * (tau + BETA))) / (1.0 + torch.exp(-BETA * e))
    tab = torch.from_numpy(tables).cuda()
    n = tab.shape[2] - 1
    x = torch.where(pos, tau, tau + BETA) * (n / BETA)
    m = x.floor().clamp(0, n - 1).long()
    half = torch.where(pos, 0, 1)
    kk = k[:, None].expand_as(m)
    a, b = tab[kk, half, m], tab[kk, half, m + 1]
    return sign * (a + (x - m).clamp(0.0, 1.0) * (b - a))


def _walk(levels, factors, samples, dtype=torch.float64):
    val = torch.ones((1, samples), dtype=dtype, device="cuda")
    for rows, ranks, w in levels:
        acc = torch.zeros((w, samples), dtype=dtype, device="cuda")
        for src, slot in ranks:
            part = val.index_select(0, src)
            if factors is None:
                acc[:src.numel()] += part
            else:
                acc[:src.numel()].addcmul_(part, factors.index_select(0, slot))
        val = torch.empty_like(acc)
        val[rows] = acc
    return val[0]


def _values(g, t, eps, tables=None, with_abs=False, count=False):
    """The sink value of every sample, t [D][S]; with_abs: the sums of |path| values after them."""
    slots, levels = _levels(g)
    s = t.shape[1]
    step = int(max(64, min(8192, (1 << 27) // max(int(g.widths.max()), len(slots)))))
    out, out_abs = [], []
    for a in range(0, s, step):
        tt = t[:, a:a + step]
        if count:
            out.append(_walk(levels, None, tt.shape[1], torch.int64))
            continue
        f = _factors(slots, tt, eps, tables)
        out.append(_walk(levels, f, tt.shape[1]))
        if with_abs:
            out_abs.append(_walk(levels, f.abs(), tt.shape[1]))
    return torch.cat(out + out_abs)


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 (Salmon et al., SC'11) over int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(a, c):   # high and low words of the 64-bit product, without overflow
        lo16, hi16 = (a & 0xFFFF) * c, (a >> 16) * c
        mid = hi16 + (lo16 >> 16)
        return (mid >> 16) & mask, ((mid << 16) | (lo16 & 0xFFFF)) & mask

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mul(c0, 0xD2511F53)
        h1, l1 = mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1, c2, c3


def _unit(high, low):
    """53 bits of a word pair scaled to [0, 1)."""
    return ((high << 21) | (low >> 11)).double() * 2.0 ** -53


def _uniform_times(seed, samples, num_times):
    n = torch.arange(samples, dtype=torch.int64, device="cuda")
    zero = torch.zeros_like(n)
    rows = []
    for m in range((num_times + 1) // 2):
        w0, w1, w2, w3 = _philox(n, zero, zero + m, zero, seed)
        rows += [BETA * _unit(w1, w0), BETA * _unit(w3, w2)]
    return torch.stack(rows[:num_times])


def _metropolis(g, t, eps, seed, steps):
    """The walkers' values, times and tallies after the steps (t [D][S] is changed)."""
    d, s = t.shape
    walker = torch.arange(s, dtype=torch.int64, device="cuda")
    cur = _values(g, t, eps)
    accepted = positive = negative = 0
    for n in range(steps):
        w0, w1, w2, w3 = _philox(walker, torch.zeros_like(walker), torch.full_like(walker, n),
                                 torch.full_like(walker, 1 << 31), seed)
        i = (w0 * d) >> 32
        old = t[i, walker].clone()
        t[i, walker] = BETA * _unit(w2, w1)
        new = _values(g, t, eps)
        keep = (w3.double() + 0.5) * 2.0 ** -32 * cur.abs() < new.abs()
        cur = torch.where(keep, new, cur)
        t[i, walker] = torch.where(keep, t[i, walker], old)
        accepted += int(keep.sum())
        positive += int((cur > 0).sum())
        negative += int((cur < 0).sum())
    return {"values": cur, "times": t, "tallies": {"steps": steps, "accepted": accepted, "n_pos": positive, "n_neg": negative}}


def exact(case, seed):
    if case["entry"] == "batch":
        values, means = [], []
        for n, (g, s) in enumerate(_mix_of(case)):
            eps, t = _inputs(g.num_kinds, g.num_times, s, seed + 1000 * n)
            values.append(_values(g, t.T.contiguous(), eps))
            means.append(float(values[-1].mean()))
        return {"values": values, "means": np.array(means)}
    g, s = _graph_of(case, seed), case["samples"]
    eps, t = _inputs(g.num_kinds, g.num_times, s, seed)
    t = t.T.contiguous()
    if case["entry"] == "mc":
        return _metropolis(g, t, eps, seed, case["steps"])
    if case["times"] == "uniform":
        t = _uniform_times(seed, s, g.num_times)
    tables = _tables(g.num_kinds, case["table"], seed) if case["table"] else None
    v = _values(g, t, eps, tables, bool(case["abs"]), case["mode"] == "count")
    if not case["mean"]:
        return {"values": v}
    mean = float(v[:s].double().mean())
    return {"values": v, "mean": (mean, float(v[s:].mean())) if case["abs"] else mean}
