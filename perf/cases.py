"""The work that the performance of this library is judged by: seeded cases of
sampling and random walks, each run through the Python binding as a program
would call it.

Graphs are the seeded RMAT graphs of ``paper_2009_09103_gb300.inputs`` (scale
s: 2^s vertices, edge factor: drawn edges per vertex before symmetrising), the
stand-ins for the social and web graphs that such samplers run on.  A case's
``kind`` says which entry points it takes:

  walk    ``csaw.walk`` over a resident graph.  form "plain": the default
          call; "build": build_cdf=True, the cumulative array built inside the
          call; "kept": over an array built once with ``Graph.build_cdf``.
          mem "host": numpy starts in, numpy paths out
  plan    ``csaw.SamplePlan``: a batch of instances through a captured plan.
          mem "host": edges copied to the host with ``result()``; "device":
          used where they are, by the view that ``csaw_sample_plan_get_view``
          gives
  sample  ``csaw.sample``: one call, edges left on the device
  layer   ``csaw.layer_sample``, edges left on the device
  mdrw    ``csaw.mdrw`` over device pools
  serve   ``csaw.Server``: a burst of mixed requests, submitted and polled

How many edges a sampling call returns depends on its draws.  As a training
loop with static buffers does, those edges go into buffers of a fixed size
(the most that the seeds and fanouts can give), filled with -1 past the end.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2009_09103_gb300 import csaw, inputs


def listed():
    return [
        # One training step's neighbourhood of a GNN minibatch: 256 seed
        # vertices, two layers, on a small graph.  Latency decides.
        {"name": "plan_minibatch_s12", "kind": "plan", "scale": 12, "ef": 16, "wmax": 100, "form": "plain",
         "bias": "edge_weight", "mem": "host", "instances": 1, "seeds_lo": 256, "seeds_hi": 256,
         "fanout": "10,5"},
        # Thousands of independent instances of very unequal size at once, as
        # a data-parallel trainer or an offline embedding job samples them;
        # the biases are degree gathers.
        {"name": "plan_batched_s22", "kind": "plan", "scale": 22, "ef": 16, "wmax": 255, "form": "plain",
         "bias": "neighbor_degree", "mem": "device", "instances": 2048, "seeds_lo": 64, "seeds_hi": 8192,
         "fanout": "25,10"},
        # A one-off call of three layers from a training loop that keeps the
        # weights' cumulative array: odd seed counts, edges used on the device.
        {"name": "sample_kept_s18", "kind": "sample", "scale": 18, "ef": 16, "wmax": 255, "form": "kept",
         "bias": "edge_weight", "instances": 37, "seeds_lo": 100, "seeds_hi": 600, "fanout": "15,10,5"},
        # A few short walks from a user's seed list, numpy in and out: the
        # smallest walk call.
        {"name": "walk_small_s14", "kind": "walk", "scale": 14, "ef": 16, "wmax": 255, "form": "plain", "mem": "host",
         "bias": "edge_weight", "walkers": 1000, "length": 20},
        # The default weighted walk call over a mid-sized graph, one walker
        # per vertex (DeepWalk-style corpus).
        {"name": "walk_default_s18", "kind": "walk", "scale": 18, "ef": 16, "wmax": 255, "form": "plain", "mem": "device",
         "bias": "edge_weight", "walkers": 1 << 18, "length": 40},
        # The weighted walk of the benchmark: a million walkers, 80 steps, the
        # array's construction inside the call.
        {"name": "walk_build_s20", "kind": "walk", "scale": 20, "ef": 16, "wmax": 255, "form": "build", "mem": "device",
         "bias": "edge_weight", "walkers": 1 << 20, "length": 80},
        # Degree-biased walks from an odd number of starts over an array that
        # a long-running program keeps.
        {"name": "walk_kept_degree_s20", "kind": "walk", "scale": 20, "ef": 16, "wmax": 255, "form": "kept",
         "mem": "device", "bias": "neighbor_degree", "walkers": 600011, "length": 64},
        # node2vec corpus (p = 2, q = 0.5): one walker per vertex on a dense
        # graph; the second-order bias depends on the previous vertex.
        {"name": "walk_node2vec_s20", "kind": "walk", "scale": 20, "ef": 32, "wmax": 15, "form": "plain", "mem": "device",
         "bias": "node2vec", "walkers": 1 << 20, "length": 40},
        # Random walk with restart (personalised PageRank by simulation):
        # many walkers from a few start vertices.
        {"name": "walk_restart_s18", "kind": "walk", "scale": 18, "ef": 16, "wmax": 255, "form": "restart",
         "mem": "device", "bias": "edge_weight", "walkers": 100003, "length": 50},
        # Layer-wise importance sampling: 2000 minibatches, 512 vertices a layer.
        {"name": "layer_s20", "kind": "layer", "scale": 20, "ef": 16, "wmax": 255, "form": "plain", "bias": "edge_weight",
         "instances": 2000, "seeds_lo": 64, "seeds_hi": 64, "fanout": "512,512"},
        # Frontier sampling of a graph's statistics: pools of 2000 vertices,
        # one long dependent chain per instance.
        {"name": "mdrw_s20", "kind": "mdrw", "scale": 20, "ef": 16, "wmax": 255, "form": "plain", "instances": 2000,
         "pool": 2000, "steps": 2000},
        # A burst of mixed requests to the server: half layered sampling, half
        # weighted walks, sizes spread over four orders of magnitude.
        {"name": "serve_burst_s18", "kind": "serve", "scale": 18, "ef": 16, "wmax": 255, "form": "plain",
         "requests": 20, "slots": 8},
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "node2vec", "plan", "sample", "layer", "mdrw", "serve"])
    c = {"kind": kind, "ef": rng.randint(8, 16), "wmax": _log(rng, 15, 60000), "form": "plain"}
    if kind == "walk":
        c["scale"] = rng.randint(12, 20)
        c["bias"] = rng.choice(["edge_weight", "edge_weight", "neighbor_degree", "uniform"])
        c["form"] = rng.choice(["plain", "build", "kept", "restart"])
        c["mem"] = rng.choice(["device", "device", "host"])
        c["walkers"] = _log(rng, 64, 1 << c["scale"])
        c["length"] = rng.randint(5, 80)
    elif kind == "node2vec":
        c.update(kind="walk", bias=kind, mem="device", scale=rng.randint(12, 19), ef=rng.randint(8, 32), wmax=_log(rng, 1, 1000))
        c["form"] = rng.choice(["plain", "plain", "kept"])
        c["walkers"] = _log(rng, 64, 1 << c["scale"])
        c["length"] = rng.randint(5, 40)
    elif kind in ("plan", "sample"):
        c["scale"] = rng.randint(12, 20)
        c["bias"] = rng.choice(["edge_weight", "neighbor_degree", "uniform"])
        c["form"] = rng.choice(["plain", "kept"])
        c["mem"] = "device"
        c["instances"] = _log(rng, 1, 1000)
        c["seeds_lo"] = _log(rng, 1, 200)
        c["seeds_hi"] = min(_log(rng, c["seeds_lo"], 4000), 1 << (c["scale"] - 2))
        c["fanout"] = ",".join(str(_log(rng, 2, 25)) for _ in range(rng.randint(1, 2 if kind == "plan" else 3)))
        # no more edges than the largest listed batch may give
        while c["instances"] > 1 and c["instances"] * c["seeds_hi"] * math.prod(_fanout(c)) > 1 << 29:
            c["instances"] //= 2
        while c["seeds_hi"] * math.prod(_fanout(c)) > 1 << 29:
            c["seeds_hi"] = max(1, c["seeds_hi"] // 2)
            c["seeds_lo"] = min(c["seeds_lo"], c["seeds_hi"])
    elif kind == "layer":
        c["scale"] = rng.randint(14, 20)
        c["bias"] = rng.choice(["edge_weight", "neighbor_degree", "uniform"])
        c["form"] = rng.choice(["plain", "plain", "kept"])
        c["instances"] = _log(rng, 1, 2000)
        c["seeds_lo"] = c["seeds_hi"] = _log(rng, 1, 64)
        c["fanout"] = ",".join(str(_log(rng, 8, 512)) for _ in range(rng.randint(1, 2)))
    elif kind == "mdrw":
        c["scale"] = rng.randint(14, 20)
        c["instances"] = _log(rng, 16, 2000)
        c["pool"] = _log(rng, 16, 4000)
        c["steps"] = _log(rng, 50, 2000)
    else:
        c["scale"] = rng.randint(14, 18)
        c["form"] = rng.choice(["plain", "kept"])
        c["requests"] = rng.randint(4, 20)
        c["slots"] = rng.choice([2, 4, 8])
    return c


def _fanout(case):
    return [int(x) for x in case["fanout"].split(",")]


def _dev(a):
    """Host uint32/uint64 array as a device tensor of the same bits."""
    return torch.from_numpy(a.view(np.int32 if a.dtype == np.uint32 else np.int64)).cuda()


class _Array:
    """Device memory of the library, by address, for torch to look at; keeps its owner."""

    def __init__(self, ptr, n, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "data": (int(ptr), False), "version": 2}


def _plan_view(plan):
    """The last run's offsets, sizes and per-layer device edges."""
    v = csaw.SampleView()
    st = csaw.lib().csaw_sample_plan_get_view(plan._h, ctypes.byref(v))
    if st != csaw.OK:
        raise csaw.CsawError(st, csaw.lib().csaw_last_error().decode())
    groups, n = v.depth * v.n_instances, v.n_instances
    offs = np.ctypeslib.as_array(v.edge_offsets, shape=(groups + 1,)).copy().view(np.int64)
    sizes = np.ctypeslib.as_array(v.frontier_sizes, shape=(groups,)).copy().view(np.int64)
    out = [offs, sizes]
    for layer in range(v.depth):
        count = int(offs[(layer + 1) * n] - offs[layer * n])
        for ptr in (v.src[layer], v.dst[layer]):
            out.append(torch.as_tensor(_Array(ptr, count, plan), device="cuda") if count else
                       torch.empty(0, dtype=torch.int32, device="cuda"))
    return out


def _layer_bounds(case, seeds, instances, fanout):
    """The most edges that each layer can give."""
    out, f = [], seeds
    for k in fanout:
        out.append(instances * k if case["kind"] == "layer" else f * k)
        f = min(out[-1], instances * (1 << case["scale"]))
    return out


def _sizes(case):
    """Seeds per instance: a case has the same sizes whatever its inputs' seed."""
    lo, hi = case["seeds_lo"], case["seeds_hi"]
    if lo == hi:
        return np.full(case["instances"], lo, dtype=np.uint64)
    return inputs.loguniform_sizes(case["instances"], math.log2(lo), math.log2(hi / lo), 4, 2)


def _keep(bufs, edges):
    """The edges in the caller's fixed buffers."""
    for b, x in zip(bufs, edges):
        if isinstance(b, np.ndarray):
            b[:len(x)] = x
        else:
            b[:x.numel()].copy_(x)
    return list(bufs)


class _State:
    """What a program holds: the resident graph, its inputs, a plan or a server."""


def prepare(case, seed):
    g = inputs.rmat_csr(case["scale"], case["ef"], case["wmax"], 1000 + seed)
    st = _State()
    st.case = case
    st.seed = 1 + seed
    st.G = csaw.Graph(g.off, g.col, g.w)
    live = np.flatnonzero(np.diff(g.off) > 0).astype(np.uint32)
    kind = case["kind"]
    if case["form"] == "kept" and case.get("bias", "edge_weight") != "uniform":
        kept = case.get("bias", "edge_weight")
        st.G.build_cdf("edge_weight" if kept == "node2vec" else kept)
    if kind == "walk":
        n = case["walkers"]
        if case["form"] == "restart":
            # many walkers per start vertex
            few = live[inputs.uniform_vertices(max(1, n // 100), len(live), seed, 1)]
            starts = np.resize(few, n)
        elif n == g.V:
            starts = np.arange(n, dtype=np.uint32)
        else:
            starts = inputs.uniform_vertices(n, g.V, seed, 1)
        st.starts = _dev(starts) if case["mem"] == "device" else starts
    elif kind in ("plan", "sample", "layer"):
        sizes = _sizes(case)
        idx, offs = inputs.distinct_seeds(sizes, len(live), seed, 3)
        st.seeds, st.offs = _dev(live[idx]), _dev(offs)
        bounds = _layer_bounds(case, len(idx), case["instances"], _fanout(case))
        if kind == "plan" and case["mem"] == "host":
            st.out = [np.full(sum(bounds), -1, dtype=np.int32) for _ in range(2)]
        else:
            st.out = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in bounds for _ in range(2)]
        if kind == "plan":
            st.plan = csaw.SamplePlan(st.G, case["instances"], len(idx), _fanout(case), case["bias"])
    elif kind == "mdrw":
        n, m = case["instances"], case["pool"]
        st.pools = _dev(live[inputs.uniform_vertices(n * m, len(live), seed, 4)].reshape(n, m))
    else:
        # the serving mix's sizes, with seeds and starts of these inputs
        st.reqs, st.out = [], []
        for i, r in enumerate(inputs.serving_requests(g.V, case["requests"])):
            v = inputs.uniform_vertices(len(r[1]), g.V, seed, 10 + i)
            st.reqs.append((r[0], v) + r[2:-1] + (r[-1] + seed,))
            n = sum(_layer_bounds(case, len(v), 1, r[3])) if r[0] == "sample" else 0
            st.out.append([np.full(n, -1, dtype=np.int32) for _ in range(2)])
        st.server = csaw.Server(st.G, 40 << 30, case["slots"])
    return st


def run(st):
    c = st.case
    kind = c["kind"]
    if kind == "walk":
        kw = {}
        if c["bias"] == "node2vec":
            kw["mult"] = (1, 2, 4)
        if c["form"] == "build":
            kw["build_cdf"] = True
        elif c["form"] == "restart":
            kw.update(teleport="restart", teleport_q32=int(0.15 * 2**32))
        path = csaw.walk(st.G, st.starts, c["length"], c["bias"], st.seed, **kw)
        return path.view(np.int32) if c["mem"] == "host" else path
    if kind == "plan":
        st.plan.run(st.seeds, st.offs, st.seed)
        if c["mem"] == "device":
            offs, sizes, *edges = _plan_view(st.plan)
            return [offs, sizes, *_keep(st.out, edges)]
        r = st.plan.result()
        return [r.edge_offsets.view(np.int64), r.frontier_sizes.view(np.int64),
                *_keep(st.out, (r.src.view(np.int32), r.dst.view(np.int32)))]
    if kind in ("sample", "layer"):
        call = csaw.sample if kind == "sample" else csaw.layer_sample
        r = call(st.G, st.seeds, st.offs, _fanout(c), c["bias"], st.seed, to_host=False)
        edges = [x for pair in zip(r.src, r.dst) for x in pair]
        return [r.edge_offsets.view(np.int64), r.frontier_sizes.view(np.int64), *_keep(st.out, edges)]
    if kind == "mdrw":
        return csaw.mdrw(st.G, st.pools, c["steps"], st.seed)
    tickets = []
    for r in st.reqs:
        if r[0] == "sample":
            tickets.append(st.server.submit_sample(r[1], r[2], r[3], "edge_weight", r[4]))
        else:
            tickets.append(st.server.submit_walk(r[1], r[2], "edge_weight", r[3]))
    out = []
    for t, bufs in zip(tickets, st.out):
        r = st.server.poll(t)
        if r.path is not None:
            out.append(r.path.view(np.int32))
        else:
            out += [r.sample.edge_offsets.view(np.int64),
                    *_keep(bufs, (r.sample.src.view(np.int32), r.sample.dst.view(np.int32)))]
    return out


def _edges(case):
    """About how many directed edges the graph has: duplicates go, both directions stay."""
    return 2 * 0.94 * case["ef"] * (1 << case["scale"])


def work(case):
    """Bytes: the inputs (of the graph what the picks can touch: 16 bytes of
    offsets and 8 of column and weight for each pick's vertex and edge, or the
    whole graph once where that is less) and the outputs.  Operations: the ten
    rounds of two wide multiplies of each draw."""
    kind = case["kind"]
    graph = 8 * (1 << case["scale"]) + 8 * _edges(case)
    if kind == "walk":
        n, steps = case["walkers"], case["walkers"] * case["length"]
        picks, io = steps, 4 * n + 4 * n * (case["length"] + 1)
    elif kind in ("plan", "sample", "layer"):
        fan = _fanout(case)
        lo, hi = case["seeds_lo"], case["seeds_hi"]
        seeds = case["instances"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
        picks, f = 0.0, seeds
        for k in fan:
            e = case["instances"] * k if kind == "layer" else f * min(k, 8)   # most rows are short
            picks += e
            f = min(e, 0.6 * case["instances"] * (1 << case["scale"]))
        io = 4 * seeds + 8 * picks
    elif kind == "mdrw":
        picks = case["instances"] * case["steps"]
        io = 4 * case["instances"] * case["pool"] + 8 * picks
    else:
        # a mean request: about 1700 seeds of 50 edges, or 5900 walkers of 45 steps
        picks = case["requests"] * 175000.0
        io = 6 * picks
    return {"bytes": io + min(graph, 24 * picks), "flops": 40 * picks}


def exact(case, seed):
    """Every output is a vertex number or a count: none is a computed real."""
    return None
