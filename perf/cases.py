"""Cases for timing the library through its public entry points.

A case names a call a program makes (``call``), the graph it makes it on and
its options:

* ``refine``: levels 0..k of a graph already loaded into a handle, each level
  then copied into a device tensor (the rebuild of a resident graph);
* ``build``: load and refine from the caller's arrays (CSR or unsorted COO
  edges; CUDA tensors or pinned host arrays), and the levels read back to where
  the arrays came from;
* ``many``: one batched build of independent graphs, each graph's last level
  read back;
* ``update``: a maintenance batch and the batch that undoes it, so that the
  graph is the same before every pass, each followed by reading the levels;
* ``labels``: the allocation-free label partition.

Graphs are drawn on the GPU from the seed, in the shapes of
``paper_1210_0748_gb300.synth``: ``uniform`` (out-degrees Zipf(2.0) capped at
10,000, uniform targets and labels) and ``powerlaw`` (Pareto out-degrees with
hubs, preferential-attachment targets, Zipf labels).
"""
import math

import numpy as np
import torch

from paper_1210_0748_gb300 import synth
from paper_1210_0748_gb300.kbisim import KBisim, label_partition_noalloc
from paper_1210_0748_gb300.serve import handle_budget

UNIFORM = {"shape": "uniform", "node_labels": 8, "edge_labels": 4}
# the 16M-node / 256M-edge workload's distributions, and the 256M / 2B one's
POWERLAW = {"shape": "powerlaw", "alpha": 2.1, "node_labels": 16, "node_zipf": 1.2, "edge_labels": 32, "edge_zipf": 1.5}
POWERLAW_2 = {"shape": "powerlaw", "alpha": 2.0, "node_labels": 64, "node_zipf": 1.3, "edge_labels": 16, "edge_zipf": 1.3}


def listed():
    return [
        # the smallest graph of the batched workload, refined on its own: launches and waits are all there is
        {"name": "refine_uniform_1k", "call": "refine", "nodes": 125, "edges": 1000, "k": 10, **UNIFORM},
        # the 100K-node / 1M-edge workload
        {"name": "refine_uniform_1m", "call": "refine", "nodes": 100_000, "edges": 1_000_000, "k": 5, **UNIFORM},
        # the benchmark workload's shape at 1/16 of its size: the identifiers fit L2 many times
        {"name": "refine_powerlaw_16m", "call": "refine", "nodes": 1_000_000, "edges": 16_000_000, "k": 10, **POWERLAW},
        # the benchmark workload
        {"name": "refine_powerlaw_256m", "call": "refine", "nodes": 16_000_000, "edges": 256_000_000, "k": 10,
         **POWERLAW},
        # the 256M-node / 2B-edge workload's shape at 1/10 of its size, odd counts: heavier hubs, half the edges per node
        {"name": "refine_powerlaw2_200m", "call": "refine", "nodes": 25_600_001, "edges": 200_000_003, "k": 10,
         **POWERLAW_2},
        # many edge labels (RDF predicates) in 32 bits: label and identifier don't fit a 32-bit word
        {"name": "refine_wide_labels_10m", "call": "refine", "nodes": 1_000_000, "edges": 10_000_000, "k": 5,
         **UNIFORM, "edge_labels": 5000},
        # a graph that a GPU program has just made as an edge list: ragged sizes, grouping by source on the device
        {"name": "build_coo_4m", "call": "build", "nodes": 413_777, "edges": 4_100_003, "k": 5, "form": "coo",
         "where": "device", **UNIFORM},
        # end to end from pinned host memory to levels on the host, a graph of the serving workload's upper range
        {"name": "build_host_32m", "call": "build", "nodes": 3_200_000, "edges": 32_000_000, "k": 5, "form": "csr",
         "where": "host", **UNIFORM},
        # the batched workload's shape, 256 of its 4096 graphs
        {"name": "many_256", "call": "many", "graphs": 256, "edges_min": 1000, "edges_max": 1_000_000, **UNIFORM},
        # small maintenance batches on a resident graph, with the handle's own (default) choice of the path
        {"name": "update_16m", "call": "update", "nodes": 1_000_000, "edges": 16_000_000, "k": 3, "batch": 1000,
         "maintain": True, **POWERLAW},
        # an update of the serving loop (recomputes, under the handle's memory budget), mid-size batch
        {"name": "update_serve_10m", "call": "update", "nodes": 1_000_000, "edges": 10_000_000, "k": 5,
         "batch": 30_000, "maintain": False, **UNIFORM},
        # the label partition at its size limit, which a caller queues among its own kernels
        {"name": "labels_262144", "call": "labels", "nodes": 262_144, "node_labels": 1000},
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["refine", "refine", "refine", "build", "build", "many", "update", "labels"])
    if call == "labels":
        return {"call": call, "nodes": logint(1000, 262_144), "node_labels": logint(2, 3000)}
    if call == "many":
        return {"call": call, "graphs": logint(8, 300), "edges_min": 1000, "edges_max": logint(10_000, 1_000_000),
                **UNIFORM}
    shape = dict(rng.choice([UNIFORM, POWERLAW, POWERLAW_2, {**UNIFORM, "edge_labels": logint(300, 10_000)}]))
    edges = logint(1000, 64_000_000 if call == "refine" else 20_000_000)
    case = {"call": call, "nodes": max(16, int(edges / rng.uniform(6, 20))), "edges": edges, "k": rng.randint(1, 10),
            **shape}
    if call == "build":
        case.update(form=rng.choice(["csr", "coo"]), where=rng.choice(["device", "host"]))
    if call == "update":
        case.update(batch=min(logint(100, 1_000_000), edges // 4), maintain=rng.choice([True, False]), k=rng.randint(1, 5))
    return case


# --- graphs -----------------------------------------------------------------
def _zipf_cdf(num, s):
    c = np.cumsum(np.arange(1, num + 1, dtype=np.float64) ** (-s))
    return torch.from_numpy(c / c[-1]).cuda()


def _uniform01(count, gen):
    return torch.rand(count, dtype=torch.float64, device="cuda", generator=gen)


def _labels(count, num, zipf, gen):
    if zipf:
        lab = torch.searchsorted(_zipf_cdf(num, zipf), _uniform01(count, gen), right=True).clamp_(max=num - 1)
    else:
        lab = torch.randint(num, (count,), device="cuda", generator=gen)
    return lab


def _degrees(n, m, case, gen):
    """Out-degrees that sum to m: the shape's draw scaled to m, the rest handed out one by one to random nodes."""
    if case["shape"] == "uniform":
        raw = torch.searchsorted(_zipf_cdf(10_000, 2.0), _uniform01(n, gen), right=True) + 1
        cap = min(10_000, m)
    else:
        raw = (1.0 - _uniform01(n, gen)).pow_(-1.0 / (case["alpha"] - 1.0)).round_().clamp_(1, 2.0 ** 40).to(torch.int64)
        cap = min(1_000_000, m)
    deg = (raw.to(torch.float64) * (m / float(raw.sum()))).floor_().clamp_(1, cap).to(torch.int64)
    left = m - int(deg.sum())
    while left > 0:
        take = torch.randperm(n, device="cuda", generator=gen)[:left]
        deg[take] += 1
        left -= take.numel()
    while left < 0:
        big = torch.nonzero(deg > 1).flatten()
        take = big[torch.randperm(big.numel(), device="cuda", generator=gen)[:-left]]
        deg[take] -= 1
        left += take.numel()
    return deg


def _targets(n, m, case, gen):
    if case["shape"] == "uniform":
        return torch.randint(n, (m,), device="cuda", generator=gen, dtype=torch.int32)
    perm = torch.randperm(n, device="cuda", generator=gen, dtype=torch.int32)
    e = 1.0 - 1.0 / (case["alpha"] - 1.0)
    u = _uniform01(m, gen)
    if abs(e) > 1e-12:
        r = u.mul_((n + 1.0) ** e - 1.0).add_(1.0).pow_(1.0 / e)
    else:
        r = u.mul_(math.log(n + 1.0)).exp_()
    return perm[r.sub_(1.0).to(torch.int64).clamp_(0, n - 1)]


def _graph(n, m, case, gen):
    """(offsets int64, dst int32, edge label uint8 or int32, node label int32) on the GPU."""
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(_degrees(n, m, case, gen), 0, out=off[1:])
    lab = _labels(m, case["edge_labels"], case.get("edge_zipf"), gen)
    lab = lab.to(torch.uint8 if case["edge_labels"] <= 256 else torch.int32)
    nlab = _labels(n, case["node_labels"], case.get("node_zipf"), gen).to(torch.int32)
    return off, _targets(n, m, case, gen), lab, nlab


def _sources(off):
    n = off.numel() - 1
    return torch.repeat_interleave(torch.arange(n, dtype=torch.int32, device="cuda"), off[1:] - off[:-1])


def _pinned(t):
    """A pinned host copy, as the unsigned numpy array a host program would hold."""
    a = torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()
    return a if a.dtype == np.uint8 else a.view(np.uint64 if a.itemsize == 8 else np.uint32)


def _arrays(case, gen):
    """The caller's arrays of a graph: keyword arguments of KBisim.load and KBisim.build."""
    n = case["nodes"]
    off, dst, lab, nlab = _graph(n, case["edges"], case, gen)
    if case.get("form") == "coo":
        mix = torch.randperm(dst.numel(), device="cuda", generator=gen)
        arrays = {"src": _sources(off)[mix], "dst": dst[mix], "edge_label": lab[mix], "node_label": nlab}
    else:
        arrays = {"offsets": off, "dst": dst, "edge_label": lab, "node_label": nlab}
    if case.get("where") == "host":
        arrays = {key: _pinned(t) for key, t in arrays.items()}
    return {"num_nodes": n, **arrays}


def _batches(case, arrays, gen):
    """A batch (half insertions of random edges, half deletions of edges there are) and the one that undoes it."""
    n, m = case["nodes"], arrays["dst"].numel()
    ni = case["batch"] // 2
    at = torch.randperm(m, device="cuda", generator=gen)[:case["batch"] - ni]
    dels = (torch.searchsorted(arrays["offsets"], at, right=True) - 1, arrays["dst"][at], arrays["edge_label"][at])
    ins = tuple(torch.randint(hi, (ni,), device="cuda", generator=gen) for hi in (n, n, case["edge_labels"]))
    ins, dels = (tuple(x.cpu().numpy().astype(np.uint32) for x in b) for b in (ins, dels))
    return [{"ins": ins, "dels": dels}, {"ins": dels, "dels": ins}]


def _many(case, gen):
    """Disjoint union of the case's graphs as KBisim.build_many takes it, and each graph's k."""
    g = case["graphs"]
    sizes = np.random.default_rng([g, case["edges_max"]])  # a case's sizes and k are its own, whatever the seed
    edges = np.exp(sizes.uniform(math.log(case["edges_min"]), math.log(case["edges_max"]), g)).astype(int).tolist()
    ks = sizes.integers(1, 11, g).tolist()
    parts, starts, base = [], [0], 0
    for m in edges:
        off, dst, lab, nlab = _graph(m // 8, m, case, gen)
        parts.append((off[:-1] + base, dst + starts[-1], lab, nlab))
        starts.append(starts[-1] + m // 8)
        base += m
    off, dst, lab, nlab = (torch.cat(x) for x in zip(*parts))
    off = torch.cat([off, torch.tensor([base], device="cuda")])
    return (synth.Graph(starts[-1], off, dst, lab, nlab), np.array(starts, dtype=np.uint64)), ks


# --- one pass ----------------------------------------------------------------
def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    call, state = case["call"], {"case": case}
    if call == "labels":
        state["labels"] = _labels(case["nodes"], case["node_labels"], None, gen).to(torch.int32)
        state["pid0"] = torch.empty_like(state["labels"])
        state["count"] = torch.empty(1, dtype=torch.int32, device="cuda")
        return state
    state["handle"] = kb = KBisim(maintain=case.get("maintain", True))
    if call == "many":
        state["union"], state["ks"] = _many(case, gen)
        return state
    arrays = _arrays(case, gen)
    if call != "build" or case["where"] == "device":
        state["levels"] = torch.empty(case["k"] + 1, case["nodes"], dtype=torch.int32, device="cuda")
    if call == "build":
        state["arrays"] = arrays
    elif call == "refine":
        kb.load(**arrays)
    else:
        state["batches"] = _batches(case, arrays, gen)
        kb.build(k=case["k"], **arrays)
        if not case["maintain"]:
            kb.set_hbm_budget(handle_budget(kb.device_bytes))
    return state


def _read(state, res):
    """Block counts and levels 0..k."""
    kb, out = state["handle"], state.get("levels")
    return {"counts": np.array(res.counts, dtype=np.int64),
            "levels": [kb.pids(i).view(np.int32) if out is None else kb.pids(i, out=out[i]) for i in range(state["case"]["k"] + 1)]}


def run(state):
    case = state["case"]
    call, k = case["call"], case.get("k")
    if call == "labels":
        label_partition_noalloc(state["labels"], state["pid0"], state["count"])
        return {"pid0": state["pid0"], "count": state["count"]}
    kb = state["handle"]
    if call == "refine":
        return _read(state, kb.refine(k))
    if call == "build":
        return _read(state, kb.build(k=k, **state["arrays"]))
    if call == "many":
        ks = state["ks"]
        kb.build_many(None, ks, union=state["union"])
        return {"counts": np.concatenate([kb.many_info(j)[1] for j in range(len(ks))]).astype(np.int64),
                "pids": np.concatenate([kb.many_pids(j, ks[j]) for j in range(len(ks))]).view(np.int32)}
    out = {}
    for name, batch in zip(("changed", "undone"), state["batches"]):
        res, missing = kb.update(k, **batch)
        got = _read(state, res)
        out[name] = {"missing": missing, "counts": got["counts"], "last": got["levels"][-1]}
        if name == "changed":  # the second batch's levels go into the same buffer
            out[name]["last"] = out[name]["last"].clone()
    return out


def work(case):
    call = case["call"]
    if call == "labels":
        return {"bytes": 8.0 * case["nodes"], "flops": 0}
    if call == "many":
        lo, hi = case["edges_min"], case["edges_max"]
        m = case["graphs"] * (hi - lo) / math.log(hi / lo)
        n, k, passes = m / 8, 5, 1
    else:
        n, m, k, passes = case["nodes"], case["edges"], case["k"], 2 if call == "update" else 1
    edge = 5 if case["edge_labels"] <= 256 else 8
    # these graphs are stable after about 4 rounds; a round reads the edge table, the offsets and the level before and
    # writes its level, and level 0 reads and writes 4 bytes per node
    rounds = min(k, 4)
    moved = rounds * (m * edge + n * 16) + n * 8
    if call in ("build", "many"):
        moved += m * (edge + (4 if case.get("form") == "coo" else 0)) + n * 12
    return {"bytes": float(passes * moved), "flops": 0}


# --- the same levels in plain torch ---------------------------------------------
def _canonical(key):
    """Classes of equal rows (or values) numbered by their first row."""
    inv = torch.unique(key, dim=0 if key.dim() > 1 else None, return_inverse=True)[1]
    n, c = inv.numel(), int(inv.max()) + 1 if inv.numel() else 0
    first = torch.full((c,), n, dtype=torch.int64, device=inv.device).scatter_reduce_(
        0, inv, torch.arange(n, device=inv.device), "amin")
    rank = torch.empty_like(first)
    rank[torch.argsort(first)] = torch.arange(c, device=inv.device)
    return rank[inv], c


def _sets(n, src, elem):
    """One number per source for its set of elements: sorted lists without repeats, folded pair by pair; each
    pass numbers the distinct pairs, so equal numbers are equal lists."""
    key = torch.unique(torch.stack([src, elem], 1), dim=0)
    src, val = key[:, 0].contiguous(), torch.unique(key[:, 1], return_inverse=True)[1] + 1
    while src.numel():
        start = torch.searchsorted(src, torch.arange(n, device=src.device))
        at = torch.arange(src.numel(), device=src.device) - start[src]
        if int(at.max()) == 0:
            break
        left = at % 2 == 0
        nxt = torch.cat([val[1:], val.new_zeros(1)])
        has = torch.cat([(src[1:] == src[:-1]), src.new_zeros(1, dtype=torch.bool)])
        pair = torch.stack([val[left], torch.where(has, nxt, 0)[left]], 1)
        src, val = src[left], torch.unique(pair, dim=0, return_inverse=True)[1] + 1
    out = torch.zeros(n, dtype=torch.int64, device=src.device)
    out[src] = val
    return out


def exact(case, seed):
    if case["call"] not in ("refine", "build", "labels") or case.get("edges", 0) > 5_000_000:
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["call"] == "labels":
        pid, c = _canonical(_labels(case["nodes"], case["node_labels"], None, gen))
        return {"pid0": pid, "count": torch.tensor([c])}
    n = case["nodes"]
    arrays = {key: torch.as_tensor(v if isinstance(v, torch.Tensor) else v.astype(np.int64)).cuda().long()
              for key, v in _arrays(case, gen).items() if key != "num_nodes"}
    src = arrays["src"] if "src" in arrays else _sources(arrays["offsets"]).long()
    pid, c = _canonical(arrays["node_label"])
    levels, counts = [pid], [c]
    for _ in range(case["k"]):
        elem = (arrays["edge_label"] << 32) | levels[-1][arrays["dst"]]
        pid, c = _canonical(torch.stack([levels[-1], _sets(n, src, elem)], 1))
        levels.append(pid)
        counts.append(c)
    return {"counts": np.array(counts, dtype=np.int64), "levels": levels}
