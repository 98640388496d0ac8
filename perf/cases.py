"""The work that users have this library do, as timed cases.

listed() and draw() describe cases as plain values, prepare() makes what a
user's program holds before the call (inputs in device or pinned host memory),
run() is one pass through the public Python entry points, work() the bytes and
operations that pass cannot do without, and exact() its results computed from
the generating order alone, in 64 bits with plain torch.

Inputs are the kinds of list that the paper and this repository's own
configurations name: lists in random order, lists shuffled inside windows of
256 positions, the identity order, forests of a few long and many short lists,
Euler tours of random trees with weights +1 and -1, and batches of independent
lists of log-uniform sizes.  int32 weights lie in [-1000, 1000], int64 weights
in [0, 2^20).
"""
import math
import random

import torch

import paper_2606_09318_gb300 as lr

_BYTES = {"none": 0, "int32": 4, "int64": 8}


def listed():
    return [
        # A short list ranked on its own: the latency of one call.
        {"name": "list_1k", "kind": "list", "order": "random", "n": 1000, "weights": "none", "validate": False},
        # A weighted list of a few ten thousand elements: latency, a few levels.
        {"name": "list_20k_i64", "kind": "list", "order": "random", "n": 20011, "weights": "int64",
         "validate": False},
        # The smallest single-list size of the published configurations (plus a
        # ragged end): everything fits in L2.
        {"name": "list_1m", "kind": "list", "order": "random", "n": (1 << 20) + 7, "weights": "none",
         "validate": False},
        # Weighted ranking of a list well beyond L2.
        {"name": "list_16m_i32", "kind": "list", "order": "random", "n": 1 << 24, "weights": "int32",
         "validate": False},
        # The headline: one random list of 2^28 elements.
        {"name": "list_268m", "kind": "list", "order": "random", "n": 1 << 28, "weights": "none",
         "validate": False},
        # A list whose order follows memory, as after a traversal or a sort.
        {"name": "local_67m_i32", "kind": "list", "order": "locality", "n": (1 << 26) + 13, "weights": "int32",
         "validate": False},
        # Many lists in one successor array, input checked for two predecessors.
        {"name": "forest_8m", "kind": "forest", "n": (1 << 23) + 1, "n_long": 4, "validate": True},
        # Tree computations: the Euler tour of a random tree, depths from +1/-1.
        {"name": "euler_4m", "kind": "euler", "vertices": 1 << 21},
        # Many independent weighted lists back to back, sizes 2^8 to 2^22.
        {"name": "batch_1024", "kind": "batch", "k": 1024, "lo": 8.0, "hi": 22.0, "sizes": 1, "weights": "int64"},
        # Waiting requests of a service, sizes 2^10 to 2^18, each in its own buffers.
        {"name": "requests_48", "kind": "requests", "k": 48, "lo": 10.0, "hi": 18.0, "sizes": 2, "weights": "int64"},
        # Terminal ids and head-relative ranks beside the ranks.
        {"name": "outputs_4m_i32", "kind": "outputs", "n": (1 << 22) - 1, "weights": "int32"},
        # A list in pinned host memory, ranked end to end.
        {"name": "host_4m", "kind": "host", "n": 4000037, "weights": "none"},
    ]


def _log_int(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["list", "list", "list", "list", "forest", "euler", "batch", "requests", "outputs", "host"])
    weights = rng.choice(["none", "int32", "int64"])
    if kind == "list":
        order = rng.choice(["random", "random", "random", "locality", "identity"])
        top = (1 << 27) + 5 if weights == "none" else 1 << 26
        return {"kind": kind, "order": order, "n": _log_int(rng, 500, top), "weights": weights,
                "validate": rng.random() < 0.2}
    if kind == "forest":
        return {"kind": kind, "n": _log_int(rng, 5000, 1 << 24), "n_long": rng.randint(0, 8),
                "validate": rng.random() < 0.5}
    if kind == "euler":
        return {"kind": kind, "vertices": _log_int(rng, 2000, 1 << 22)}
    if kind == "batch":
        hi = rng.uniform(11.0, 18.0)
        return {"kind": kind, "k": rng.randint(8, 512), "lo": 8.0, "hi": hi, "sizes": rng.randint(0, 1 << 30),
                "weights": weights}
    if kind == "requests":
        hi = rng.uniform(12.0, 20.0)
        return {"kind": kind, "k": rng.randint(4, 60), "lo": 10.0, "hi": hi, "sizes": rng.randint(0, 1 << 30),
                "weights": weights}
    if kind == "outputs":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 24), "weights": weights}
    return {"kind": "host", "n": _log_int(rng, 1000, 1 << 24), "weights": weights}


# ---------------------------------------------------------------- inputs
_DEV = "cuda"


def _gen(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed) & (2**63 - 1))
    return g


def _order(kind, n, g):
    """The ids in list order, front to back (int64)."""
    if kind == "random":
        return torch.randperm(n, device=_DEV, generator=g, dtype=torch.int64)
    ids = torch.arange(n, device=_DEV)
    if kind == "identity":
        return ids
    key = (ids >> 8) << 31 | torch.randint(0, 1 << 31, (n,), device=_DEV, generator=g)
    return torch.argsort(key)


def _successors(order, ends, base=None):
    """int32 successor array of the lists that visit `order`, cut after the
    positions marked in `ends` (None: one list); ids less `base` if given."""
    nxt = torch.roll(order, -1)
    if ends is None:
        nxt[-1] = order[-1]
    else:
        nxt = torch.where(ends, order, nxt)
    if base is not None:
        nxt = nxt - base
    succ = torch.empty(order.numel(), dtype=torch.int32, device=_DEV)
    succ[order] = nxt.to(torch.int32)
    return succ


def _weights(kind, n, g):
    if kind == "none":
        return None
    if kind == "int32":
        return torch.randint(-1000, 1001, (n,), device=_DEV, generator=g, dtype=torch.int32)
    return torch.randint(0, 1 << 20, (n,), device=_DEV, generator=g, dtype=torch.int64)


def _forest_ends(n, n_long, g):
    """Marks of the list ends: n_long lists that share half of the elements,
    then lists of geometric length with mean 64."""
    ends = torch.zeros(n, dtype=torch.bool, device=_DEV)
    long_len = n // (2 * n_long) if n_long else 0
    cut = n_long * long_len
    for j in range(n_long):
        ends[(j + 1) * long_len - 1] = True
    ends[cut:] = torch.rand(n - cut, device=_DEV, generator=g) < 1.0 / 64
    ends[-1] = True
    return ends


def _tree(vertices, g):
    """parent[v] uniform below v; parent[0] = 0."""
    v = torch.arange(vertices, device=_DEV)
    u = torch.rand(vertices, device=_DEV, generator=g, dtype=torch.float64)
    return torch.minimum((u * v).to(torch.int64), (v - 1).clamp(min=0))


def _euler(parent):
    """Successors and weights of the tour: arc 2(v-1) goes down to v (+1), arc
    2(v-1)+1 comes back up (-1); children in ascending order."""
    nv = parent.numel()
    kids = torch.arange(1, nv, device=_DEV)
    by_parent = torch.sort(parent[1:], stable=True).indices + 1
    par = parent[by_parent]
    same = par[1:] == par[:-1]
    first = torch.cat([torch.ones(1, dtype=torch.bool, device=_DEV), ~same])
    first_child = torch.full((nv,), -1, dtype=torch.int64, device=_DEV)
    first_child[par[first]] = by_parent[first]
    next_sib = torch.full((nv,), -1, dtype=torch.int64, device=_DEV)
    next_sib[by_parent[:-1][same]] = by_parent[1:][same]
    up = 2 * (kids - 1) + 1
    fc, ns, pv = first_child[kids], next_sib[kids], parent[kids]
    succ = torch.empty(2 * (nv - 1), dtype=torch.int32, device=_DEV)
    succ[up - 1] = torch.where(fc >= 0, 2 * (fc - 1), up).to(torch.int32)
    back = torch.where(pv == 0, up, 2 * (pv - 1) + 1)
    succ[up] = torch.where(ns >= 0, 2 * (ns - 1), back).to(torch.int32)
    weight = torch.ones(2 * (nv - 1), dtype=torch.int32, device=_DEV)
    weight[up] = -1
    return succ, weight


def _batch_lens(case):
    """The batch's k instance sizes, log-uniform (part of the case: every
    seed's inputs have the same sizes)."""
    r = random.Random(case["sizes"])
    return [int(2.0 ** r.uniform(case["lo"], case["hi"])) for _ in range(case["k"])]


def _batch_lists(case, g):
    """(offsets, order, ends, base): k random-order lists back to back."""
    lens = torch.tensor(_batch_lens(case), dtype=torch.int64, device=_DEV)
    offsets = torch.zeros(case["k"] + 1, dtype=torch.int64, device=_DEV)
    offsets[1:] = torch.cumsum(lens, 0)
    n = int(offsets[-1])
    inst = torch.repeat_interleave(torch.arange(case["k"], device=_DEV), lens, output_size=n)
    key = inst << 31 | torch.randint(0, 1 << 31, (n,), device=_DEV, generator=g)
    order = torch.argsort(key)
    del key
    ends = torch.zeros(n, dtype=torch.bool, device=_DEV)
    ends[offsets[1:] - 1] = True
    return offsets, order, ends, offsets[inst]


def _lists(case, seed):
    """What both the inputs and the exact results are made from:
    (order, ends, base, offsets, weight)."""
    g = _gen(seed)
    kind = case["kind"]
    offsets = base = ends = None
    if kind in ("batch", "requests"):
        offsets, order, ends, base = _batch_lists(case, g)
    else:
        order = _order(case.get("order", "random"), case["n"], g)
        if kind == "forest":
            ends = _forest_ends(case["n"], case["n_long"], g)
    weight = _weights(case.get("weights", "none"), order.numel(), g)
    return order, ends, base, offsets, weight


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "validate": case.get("validate", False), "weight": None}
    if kind == "euler":
        st["succ"], st["weight"] = _euler(_tree(case["vertices"], _gen(seed)))
        return st
    order, ends, base, offsets, weight = _lists(case, seed)
    succ = _successors(order, ends, base)
    if kind == "requests":
        cuts = offsets.tolist()
        st["succ"] = [succ[a:b].clone() for a, b in zip(cuts, cuts[1:])]
        if weight is not None:
            st["weight"] = [weight[a:b].clone() for a, b in zip(cuts, cuts[1:])]
        return st
    if kind == "host":
        st["succ"] = succ.cpu().pin_memory()
        st["weight"] = None if weight is None else weight.cpu().pin_memory()
        st["out"] = torch.empty(case["n"], dtype=torch.int32 if weight is None else torch.int64, pin_memory=True)
        return st
    st["succ"], st["weight"] = succ, weight
    if kind == "batch":
        st["offsets"] = offsets
        st["k"] = case["k"]
    return st


def run(state):
    kind = state["kind"]
    if kind in ("list", "forest"):
        return lr.rank(state["succ"], state["weight"], validate=state["validate"])
    if kind == "euler":
        return lr.rank(state["succ"], state["weight"], rank_dtype=torch.int32)
    if kind == "batch":
        return lr.rank_batch(state["offsets"], state["succ"], state["weight"], max_lists=state["k"])
    if kind == "requests":
        return lr.rank_batch_ptrs(state["succ"], state["weight"])
    if kind == "outputs":
        return lr.rank_outputs(state["succ"], state["weight"], term=True, prefix=True)
    return lr.rank_host(state["succ"], state["weight"], out=state["out"])


def work(case):
    """Each successor and weight read once, each result written once; one
    addition per element (and one more for a head-relative rank)."""
    kind = case["kind"]
    if kind == "euler":
        n = 2 * (case["vertices"] - 1)
        return {"bytes": n * (4 + 4 + 4), "flops": n}
    if kind in ("batch", "requests"):
        n = sum(_batch_lens(case))
    else:
        n = case["n"]
    wb = _BYTES[case.get("weights", "none")]
    rb = 8 if wb else 4
    per = 4 + wb + rb
    if kind == "outputs":
        per += 4 + rb                                   # terminal ids, head-relative ranks
    return {"bytes": n * per, "flops": n * (2 if kind == "outputs" else 1)}


# ---------------------------------------------------------------- exact results
def _exact_lists(order, ends, weight):
    """Ranks, terminals and head-relative ranks of the lists along `order`."""
    n = order.numel()
    w = torch.ones(n, dtype=torch.int64, device=_DEV) if weight is None else weight[order].to(torch.int64)
    if ends is None:
        ends = torch.zeros(n, dtype=torch.bool, device=_DEV)
        ends[-1] = True
    w[ends] = 0                                         # a terminal has no outgoing link
    before = torch.cumsum(w, 0) - w                     # weight of the links before each position
    del w
    last = torch.nonzero(ends).flatten()
    which = torch.cumsum(ends, 0) - ends.to(torch.int64)
    tail = last[which]
    first = torch.cat([torch.zeros(1, dtype=torch.int64, device=_DEV), last[:-1] + 1])[which]
    rank, term, prefix = (torch.empty(n, dtype=torch.int64, device=_DEV) for _ in range(3))
    rank[order] = before[tail] - before
    term[order] = order[tail]
    prefix[order] = before - before[first]
    return rank, term, prefix


def exact(case, seed):
    kind = case["kind"]
    if kind == "euler":
        parent = _tree(case["vertices"], _gen(seed))
        hop, depth = parent.clone(), (parent != torch.arange(parent.numel(), device=_DEV)).to(torch.int64)
        while int(hop.max()) > 0:                       # distance to the root, doubling
            depth = depth + depth[hop]
            hop = hop[hop]
        rank = torch.empty(2 * (parent.numel() - 1), dtype=torch.int64, device=_DEV)
        rank[0::2] = 2 - depth[1:]                      # from the arc down to v
        rank[1::2] = -depth[parent[1:]]                 # from the arc back up to v's parent
        return rank
    order, ends, _, offsets, weight = _lists(case, seed)
    rank, term, prefix = _exact_lists(order, ends, weight)
    if kind == "requests":
        cuts = offsets.tolist()
        return [rank[a:b] for a, b in zip(cuts, cuts[1:])]
    if kind == "outputs":
        return rank, term, prefix
    if kind == "host":
        return rank.cpu()
    return rank
