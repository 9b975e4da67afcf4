"""What the performance of this library is measured on.

The cases go through the public binding the way a user's program calls it: planning one network from
host arrays (create, solve, destroy), re-solving with a handle and a workspace that the program
keeps, batches of small instances on either side of the bus, scoring and sampling candidate plans,
the paper's two-stage heuristic, and the search under the full objective.  Sizes and value
distributions are those of the named configurations of `workloads.py` (and of the paper's own
evaluation setting), drawn afresh for every seed.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare(case, seed)` makes
inputs, `run(state)` is one pass, `work(case)` the operations and bytes of one, `tolerance(case)`
how far two correct implementations may differ.
"""
from __future__ import annotations

import ctypes

import numpy as np
import torch

import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import workloads

MB = 1_000_000
CHAINS = ("uniform", "cnn", "stages", "blocks", "blocks_unequal", "geometric")


def listed():
    return [
        # one small network planned from scratch: the latency of a whole call, nothing else
        {"name": "plan_tiny", "kind": "plan", "chain": "uniform", "L": 12, "k": 6},
        # the paper's example model on ten devices, planned once from host arrays
        {"name": "plan_resnet50_shaped", "kind": "plan", "chain": "cnn", "L": 50, "k": 10},
        # a deep chain with an odd number of cut points (hundreds of layers, as EfficientNet-like models have)
        {"name": "plan_deep_chain", "kind": "plan", "chain": "stages", "L": 337, "k": 13},
        # a planner that keeps its handle and workspace and solves again and again on the device
        {"name": "solve_deeper_cnn", "kind": "solve", "chain": "stages", "L": 100, "k": 14},
        # the benchmark instance: a stack of identical blocks on 18 unequal nodes
        {"name": "solve_large", "kind": "solve", "chain": "blocks", "L": 200, "k": 18},
        # the same size with layers of unequal memory, what a real model looks like
        {"name": "solve_large_unequal", "kind": "solve", "chain": "blocks_unequal", "L": 200, "k": 18},
        # many small instances already on the device (a sweep over networks)
        {"name": "batch_4096", "kind": "batch", "B": 4096, "L": 24, "k": 8, "where": "device"},
        # a smaller batch of longer, odd-sized chains that lives in host arrays
        {"name": "batch_ragged_host", "kind": "batch", "B": 300, "L": 45, "k": 7, "where": "host"},
        # bulk scoring of candidate plans in compressed rows
        {"name": "score_packed", "kind": "score", "chain": "blocks", "L": 200, "k": 18, "B": 262144, "rows": "packed"},
        # the paper's random baseline: plans generated on the device and scored
        {"name": "sample_and_score", "kind": "sample", "chain": "geometric", "L": 50, "k": 14, "B": 100_003},
        # the paper's heuristic (Algorithm 1, then Algorithms 2 and 3) on its 50 devices, from host arrays
        {"name": "heuristic_50_nodes", "kind": "heuristic", "L": 50, "k": 50, "cap_mb": 16, "trials": 24, "classes": 3},
        # the search under Eq. 1 (compute times in the bottleneck), from host arrays
        {"name": "eq1_geometric", "kind": "eq1", "chain": "geometric", "L": 50, "k": 12},
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def relaxations(L, k):
    """(min, max) relaxations of the dense programme over (node set, last node, last layer)."""
    return k * (k - 1) * (1 << (k - 2)) * L if k >= 2 else 0


def draw(rng):
    kind = rng.choices(("plan", "solve", "batch", "score", "sample", "heuristic", "eq1"), (6, 5, 3, 2, 1, 1.5, 1.5))[0]
    if kind == "plan":
        while True:
            case = {"kind": kind, "chain": rng.choice(CHAINS), "L": _log_int(rng, 8, 400), "k": rng.randint(3, 14)}
            if relaxations(case["L"], case["k"]) <= relaxations(337, 13):
                return case
    if kind == "solve":
        while True:
            case = {"kind": kind, "chain": rng.choice(CHAINS[1:]), "L": _log_int(rng, 40, 240), "k": rng.randint(10, 18)}
            if relaxations(case["L"], case["k"]) <= relaxations(200, 18):
                return case
    if kind == "batch":
        k = rng.randint(4, 8)
        return {"kind": kind, "B": _log_int(rng, 16, 4096 if rng.random() < 0.7 else 512), "L": rng.randint(9, 32) if
                rng.random() < 0.7 else rng.randint(33, 60 if k < 8 else 48), "k": k,
                "where": rng.choice(("device", "host"))}
    if kind == "score":
        return {"kind": kind, "chain": rng.choice(CHAINS), "L": _log_int(rng, 24, 200), "k": rng.randint(6, 18),
                "B": _log_int(rng, 1000, 262144), "rows": rng.choice(("packed", "int32"))}
    if kind == "sample":
        return {"kind": kind, "chain": rng.choice(CHAINS), "L": _log_int(rng, 24, 200), "k": rng.randint(6, 18),
                "B": _log_int(rng, 1000, 200_000)}
    if kind == "heuristic":
        return {"kind": kind, "L": rng.randint(25, 100), "k": rng.randint(20, 50), "cap_mb": rng.randint(14, 40),
                "trials": rng.randint(8, 24), "classes": rng.randint(2, 4)}
    return {"kind": kind, "chain": rng.choice(CHAINS), "L": _log_int(rng, 12, 60), "k": rng.randint(5, 12)}


# ---- inputs ---------------------------------------------------------------------------------------

def _split(weights, total):
    parts = np.floor(weights / weights.sum() * total).astype(np.uint64)
    parts[-1] = np.uint64(total - int(parts[:-1].sum()))
    return parts


def _lognormal(rng, n, mean, sigma, lo, hi):
    x = np.exp(np.log(mean) - sigma * sigma / 2 + sigma * rng.standard_normal(n))
    return np.clip(np.rint(x), lo, hi)


def _symmetric(k, values):
    bw = np.zeros((k, k), dtype=np.uint32)
    bw[np.triu_indices(k, 1)] = values.astype(np.uint32)
    return bw + bw.T


def _instance(chain, L, k, rng, cap_mb=64):
    """One network of the family `chain` (the distributions of the configurations of workloads.py)."""
    pairs = k * (k - 1) // 2
    if chain == "uniform":
        bits = rng.integers(100_000, 20_000_001, L)
        mem = rng.integers(1 * MB, 40 * MB + 1, L)
        # the configurations have two or three layers to a node: longer chains get larger nodes
        cap = rng.integers(40 * MB, 160 * MB + 1, k) * max(1.0, L / (3.0 * k))
        bw = _symmetric(k, rng.integers(1000, 12001, pairs))
    elif chain in ("cnn", "geometric"):
        bits = _lognormal(rng, L, 10.2e6, 0.75, 1e5, 1.2e8)
        mem = _split(64.0 ** (np.arange(L) / L) * (0.8 + 0.4 * rng.random(L)), 102_400_000)
        if chain == "cnn":
            cap = rng.integers(24 * MB, 48 * MB + 1, k)
            bw = _symmetric(k, _lognormal(rng, pairs, 6000.0, 0.5, 500, 50000))
        else:
            cap = np.full(k, cap_mb * MB)
            bw, _ = workloads.geometric_bandwidths(k, int(rng.integers(1 << 30)), "pairwise")
    elif chain == "stages":
        raw = 2.0 ** (-(np.arange(L) * 5 // L)) * np.exp(0.35 * rng.standard_normal(L))
        bits = np.maximum(np.rint(raw * (8.0e6 / raw.mean())), 1)
        mem = _split((np.arange(L) + 1.0) * (0.9 + 0.2 * rng.random(L)), 240_000_000)
        cap = rng.integers(64 * MB, 224 * MB + 1, k)  # no node holds the whole chain
        bw = _symmetric(k, np.where(rng.random(pairs) < 0.2, 500, rng.integers(2000, 20001, pairs)))
    else:
        bits = np.rint(8_388_608 * (0.9 + 0.2 * rng.random(L)))
        mem = np.full(L, np.floor(1.2e9 / L))
        if chain == "blocks_unequal":
            mem = np.rint(mem * (0.5 + rng.random(L)))
        cap = rng.integers(128 * MB, 512 * MB + 1, k)
        bw = _symmetric(k, rng.integers(1000, 50001, pairs))
    u64 = lambda a: np.ascontiguousarray(a).astype(np.uint64)
    return workloads.Instance(L, k, u64(bits), u64(mem), u64(cap), np.ascontiguousarray(bw, dtype=np.uint32), chain)


def _device(a):
    """A host array's bytes on the GPU (unsigned types travel as signed ones of the same width)."""
    a = np.ascontiguousarray(a)
    if a.dtype.kind == "u" and a.dtype.itemsize > 1:
        a = a.view("i%d" % a.dtype.itemsize)
    return torch.from_numpy(a).cuda()


def _problem(inst):
    p = pp.Problem.from_instance(inst)
    p.set_stream(torch.cuda.current_stream().cuda_stream)
    return p


def _plans(L, k, B, g):
    """Candidate plans as `workloads.random_plans` draws them (any number of segments, random cuts,
    random distinct nodes, one row in twenty invalid), made on the GPU: nseg [B], ends, nodes [B, k]."""
    mmax = min(k, L)
    rand = lambda *shape: torch.rand(*shape, device="cuda", generator=g)
    nseg = 1 + (rand(B) * mmax).long().clamp(max=mmax - 1)
    at = torch.arange(k, device="cuda")[None, :]
    cuts = torch.full((B, k), L, device="cuda")
    if mmax > 1:
        cuts[:, : mmax - 1] = rand(B, L - 1).argsort(1)[:, : mmax - 1]
    ends = torch.where(at < nseg[:, None] - 1, cuts, L).sort(1).values
    ends = torch.where(at < nseg[:, None] - 1, ends, torch.where(at == nseg[:, None] - 1, L - 1, -1))
    nodes = torch.where(at < nseg[:, None], rand(B, k).argsort(1), -1)
    bad, kind = rand(B) < 0.05, (rand(B) * 3).long()
    nodes[:, 0] = torch.where(bad & (kind == 0), k, nodes[:, 0])               # no such node
    last = nodes.gather(1, (nseg - 1)[:, None])[:, 0]
    nodes[:, 0] = torch.where(bad & (kind == 1) & (nseg > 1), last, nodes[:, 0])  # a node used twice
    nseg = torch.where(bad & (kind == 2), 0, nseg)                             # no segment
    return nseg.to(torch.uint8), ends.to(torch.int32).contiguous(), nodes.to(torch.int32).contiguous()


def prepare(case, seed):
    rng = np.random.default_rng([seed, 20221])
    kind, L, k = case["kind"], case["L"], case["k"]
    if kind == "plan":
        return {"kind": kind, "inst": _instance(case["chain"], L, k, rng)}
    if kind == "solve":
        p = _problem(_instance(case["chain"], L, k, rng))
        p.set_workspace(torch.empty(p.workspace_bytes(), dtype=torch.uint8, device="cuda"))
        sol = torch.zeros(ctypes.sizeof(pp.pp_solution) // 4, dtype=torch.int32, device="cuda")
        return {"kind": kind, "p": p, "sol": sol, "out": (sol[:2].view(torch.float64), sol[2:])}
    if kind == "batch":
        B = case["B"]
        bw = np.zeros((B, k, k), dtype=np.uint32)
        iu = np.triu_indices(k, 1)
        bw[:, iu[0], iu[1]] = rng.integers(1000, 12001, (B, len(iu[0])))
        cap = rng.integers(40 * MB, 160 * MB + 1, (B, k)) * max(1.0, L / (3.0 * k))
        arrays = (rng.integers(100_000, 20_000_001, (B, L)).astype(np.uint64),
                  rng.integers(1 * MB, 40 * MB + 1, (B, L)).astype(np.uint64), cap.astype(np.uint64),
                  bw + bw.transpose(0, 2, 1))
        if case["where"] == "host":
            return {"kind": "batch_host", "L": L, "k": k, "arrays": arrays}
        new = lambda n, t: torch.empty(n, dtype=t, device="cuda")
        out = (new(B, torch.float64), new(B, torch.int32), new(B * (k - 1), torch.int32), new(B * k, torch.int32),
               new(B, torch.int8))
        return {"kind": kind, "B": B, "L": L, "k": k, "in": [_device(a) for a in arrays], "out": out}
    if kind == "score":
        p = _problem(_instance(case["chain"], L, k, rng))
        B = case["B"]
        nseg, ends, nodes = _plans(L, k, B, torch.Generator("cuda").manual_seed(seed))
        out = (torch.empty(B, dtype=torch.float64, device="cuda"), torch.empty(B, dtype=torch.uint8, device="cuda"))
        if case["rows"] == "int32":
            return {"kind": "score_int32", "p": p, "B": B, "in": (nseg, ends, nodes), "out": out}
        keep = torch.arange(k, device="cuda")[None, :] < nseg[:, None]
        off = torch.zeros(B + 1, dtype=torch.int32, device="cuda")
        off[1:] = nseg.long().cumsum(0)
        rows = (nseg, off, ends[keep].to(torch.int16), nodes[keep].to(torch.uint8))
        return {"kind": "score_packed", "p": p, "B": B, "total": rows[2].numel(), "in": rows, "out": out}
    if kind == "sample":
        p = _problem(_instance(case["chain"], L, k, rng))
        B = case["B"]
        draws = _device(rng.integers(0, 1 << 32, (B, 2 * k), dtype=np.uint32))
        new = lambda n, t: torch.empty(n, dtype=t, device="cuda")
        out = (new(B, torch.uint8), new(B * k, torch.int32), new(B * k, torch.int32), new(B, torch.float64),
               new(B, torch.uint8))
        return {"kind": kind, "p": p, "B": B, "draws": draws, "out": out}
    if kind == "heuristic":
        inst = _instance("geometric", L, k, rng, case["cap_mb"])
        draws = rng.integers(0, 1 << 32, (case["trials"], k), dtype=np.uint32)
        return {"kind": kind, "inst": inst, "draws": draws, "classes": case["classes"]}
    inst = _instance(case["chain"], L, k, rng)
    # layers cost work in proportion to their memory, nodes differ threefold in speed
    return {"kind": kind, "inst": inst, "work": (inst.layer_mem_bytes // np.uint64(1024)).astype(np.uint64),
            "speed": rng.integers(500, 1501, k).astype(np.uint32)}


# ---- one pass -------------------------------------------------------------------------------------

def _ptrs(tensors):
    return [t.data_ptr() for t in tensors]


def _solution(s):
    return {"status": s.status, "beta_ms": s.beta_ms, "m": s.m, "cuts": s.cuts, "placement": s.placement}


def run(state):
    kind = state["kind"]
    if kind == "plan":
        with pp.Problem.from_instance(state["inst"]) as p:
            return _solution(p.solve_exact())
    if kind == "solve":
        state["p"].solve_exact_dev(state["sol"].data_ptr())
        return state["out"]
    if kind == "batch":
        pp.solve_exact_batch_dev(state["B"], state["L"], state["k"], *_ptrs(state["in"]), *_ptrs(state["out"]),
                                 torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if kind == "batch_host":
        s = pp.solve_exact_batch(state["L"], state["k"], *state["arrays"])
        return s.beta_ms, s.m, s.cuts, s.placement, s.status
    if kind == "score_packed":
        state["p"].eval_plans_packed_dev(state["B"], state["total"], *_ptrs(state["in"]), *_ptrs(state["out"]))
        return state["out"]
    if kind == "score_int32":
        state["p"].eval_plans_dev(state["B"], *_ptrs(state["in"]), *_ptrs(state["out"]))
        return state["out"]
    if kind == "sample":
        nseg, ends, nodes, beta, status = _ptrs(state["out"])
        state["p"].random_plans_dev(state["B"], state["draws"].data_ptr(), nseg, ends, nodes)
        state["p"].eval_plans_dev(state["B"], nseg, ends, nodes, beta, status)
        return state["out"]
    if kind == "heuristic":
        inst = state["inst"]
        part = pp.partition_minsum_batch(inst.layer_out_bits[None, :], inst.layer_mem_bytes[None, :],
                                         inst.node_mem_bytes[:1], inst.L)
        m = int(part.m[0])
        status, nodes, thr = pp.kpath_matching(inst.bw_kbps, part.sizes[0, : m - 1], state["classes"], state["draws"])
        placed = np.full((2, inst.L), -1, dtype=np.int64)  # one row of nodes, one of thresholds, for any number of cuts
        placed[0, :m], placed[1, : m - 1] = nodes, thr
        return part.cost, part.m, part.cuts, part.sizes, part.status, status, placed
    return _solution(pp.solve_exact_compute(state["inst"], state["work"], state["speed"]))


# ---- what a pass needs ----------------------------------------------------------------------------

def work(case):
    """Bytes: the inputs once and the results once.  Operations: for a search, a maximum and a minimum
    per relaxation and three per state of the dense programme; for the other calls, one division and
    one comparison per cut or candidate."""
    kind, L, k = case["kind"], case["L"], case["k"]
    network = 16 * L + 8 * k + 4 * k * k
    search = 2 * relaxations(L, k) + 3 * k * (1 << (k - 1)) * L if k <= 20 else 0
    if kind in ("plan", "solve"):
        return {"bytes": network + 176, "flops": search}
    if kind == "batch":
        return {"bytes": case["B"] * (network + 13 + 4 * (2 * k - 1)), "flops": case["B"] * search}
    m = (min(k, L) + 1) / 2  # segments of a plan, on average
    if kind == "score":
        row = 5 + 3 * m - 2 if case["rows"] == "packed" else 1 + 8 * m - 4
        return {"bytes": network + case["B"] * (row + 9), "flops": case["B"] * 2 * m}
    if kind == "sample":
        return {"bytes": network + case["B"] * (8 * m + 1 + 8 * k + 9), "flops": case["B"] * 2 * m}
    if kind == "heuristic":
        return {"bytes": network + 4 * k * case["trials"] + 12 * L + 8 * k, "flops": L * L / 2}
    # Eq. 1: the compute time of every window is one more maximum per (set, node, window)
    return {"bytes": network + 8 * L + 4 * k + 176, "flops": search}


def tolerance(case):
    # values are selected, never accumulated: beta is one of the input quotients, bit for bit, and the
    # plan is canonical
    return "exact"
