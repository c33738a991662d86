"""The work a user of this framework has it do, as timed cases.

Graphs are drawn on the device from the seed alone, in the two shapes of
``paper_2210_03211_gb300/workloads.py``: "power" (Chung-Lu power law with planted
overlapping communities: collaboration and social networks) and "planted"
(equal weights inside planted overlapping communities of 20-150 nodes, 2%
background: dense small networks, the batched and the served graphs).  Weights
are integers, so that a seed gives the same edges on every run.

Kinds of a case:
  call       one call from host edge lists to communities (``run_lazyfox``)
  detect     build from an edge list on the device, run, read the communities
  run        a run on a graph that is kept
  create     the preprocessing alone (triangles, vt, node order, cc)
  batch      many graphs packed in one handle, from host edge lists
  triangles  t and vt of an oriented CSR without any allocation
  f1         F1-score of a detected cover against a reference cover
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2210_03211_gb300 import lazyfox

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")


def listed():
    return [
        # A script that clusters one small network: latency and launches count.
        dict(name="call_300_q16", kind="call", shape="planted", n=300, degree=20.0, q=16, iters=50, stop=True),
        # Fox itself (queue size 1) on an e-mail network of a thousand people, run to convergence.
        dict(name="fox_1k_q1", kind="run", shape="planted", n=1000, degree=31.0, q=1, iters=50, stop=True),
        # The quality setting on a collaboration network: short queues, close to Fox.
        dict(name="run_84k_q64", kind="run", shape="power", n=83750, degree=6.45, q=64, iters=50, stop=True),
        # The throughput setting on a collaboration network of 335k authors, run to convergence.
        dict(name="run_335k_q1024", kind="run", shape="power", n=335000, degree=6.45, q=1024, iters=50, stop=True),
        # The same with the mean-field gain, the faster rule that users may choose.
        dict(name="run_335k_q1024_meanfield", kind="run", shape="power", n=335000, degree=6.45, q=1024, iters=50,
             stop=True, rule="meanfield"),
        # Preprocessing alone: triangle counts, local clustering and node order of the same network.
        dict(name="create_335k", kind="create", shape="power", n=335000, degree=6.45),
        # One dense planted network of the serving mix, from host edge lists to communities.
        dict(name="call_61k_q1024", kind="call", shape="planted", n=61003, degree=45.0, q=1024, iters=50, stop=True),
        # A batch of small networks of uneven size in one handle.
        dict(name="batch_128_q256", kind="batch", shape="planted", count=128, n_lo=200, n_hi=20000, q=256, iters=50,
             stop=True),
        # A social network of 767k users with hubs, ten passes over a kept graph: memberships pile up.
        dict(name="run_767k_q16384", kind="run", shape="power", n=767500, degree=136.0, q=16384, iters=10, stop=False),
        # The largest: 3.07M users and about 115M friendships, from edges on the device to communities.
        dict(name="detect_3M_q65536", kind="detect", shape="power", n=3070000, degree=136.0, q=65536, iters=3,
             stop=False),
        # Scoring a detected cover of the 335k network against its reference cover.
        dict(name="f1_335k", kind="f1", n=335000),
        # Triangle counts for a program that cannot allocate when it calls.
        dict(name="triangles_335k", kind="triangles", shape="power", n=335000, degree=6.45),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["call", "run", "run", "run", "detect", "create", "batch", "triangles", "f1"])
    if kind == "batch":
        return dict(kind=kind, shape="planted", count=logu(2, 96), n_lo=200, n_hi=logu(1000, 20000), q=logu(32, 4096),
                    iters=50, stop=True)
    if kind == "f1":
        return dict(kind=kind, n=logu(500, 1000000))
    if kind == "triangles":
        return dict(kind=kind, shape="power", n=logu(1000, 700000), degree=round(rng.uniform(3.0, 12.0), 2))
    if kind == "call":
        c = dict(kind=kind, shape="planted", n=logu(200, 60000), degree=round(rng.uniform(10.0, 60.0), 1), stop=True)
        lo, iters = 1, 25
    elif kind == "create":
        return dict(kind=kind, shape="power", n=logu(1000, 2000000), degree=round(rng.uniform(4.0, 80.0), 2))
    else:
        n = logu(1000, 1500000 if kind == "detect" else 700000)
        c = dict(kind=kind, shape="power", n=n, degree=round(rng.uniform(4.0, 120.0), 2), stop=n < 100000)
        if rng.random() < 0.25:
            c["rule"] = "meanfield"
        lo, iters = 1, 20
    # at most ~16,000 queues in a run; at most one queue per iteration
    lo = max(lo, math.ceil(c["n"] * iters / 16000))
    if not c["stop"]:
        lo = max(lo, c["n"] // 100)
    c["q"] = logu(lo, max(lo, min(65536, c["n"])))
    c["iters"] = 50 if c["stop"] else 3
    return c


# --- inputs -------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, count):
    return torch.rand(int(count), generator=g, device=DEV, dtype=torch.float64)


def _below(g, high):
    """Random integers in [0, high), `high` an int64 tensor."""
    u = torch.rand(high.shape, generator=g, device=DEV, dtype=torch.float64)
    return torch.minimum((u * high).long(), high - 1)


def _cover(g, n, shape, power_hi):
    """Planted memberships (community, node), sorted by community: 1-4 (power
    law of sizes) or 1-3 (sizes 20-150) communities per node."""
    u = _uniform(g, n)
    if shape == "power":
        r = 1 + (u > 0.55).long() + (u > 0.80).long() + (u > 0.93).long()
        lo, hi = (6, min(2000, max(7, n // 4))) if power_hi < 5000 else (10, 5000)
        total = int(r.sum())
        v = _uniform(g, 2 * total // lo + 16)
        a, b = 1.0 / lo, 1.0 / (hi + 1)
        sizes = (1.0 / (a + v * (b - a))).long().clamp(lo, hi)       # P(s) ~ s^-2
    else:
        r = 1 + (u * 3.0).long().clamp(max=2)
        total = int(r.sum())
        sizes = 20 + (_uniform(g, total // 20 + 16) * 131.0).long()
    ends = torch.cumsum(sizes, 0)
    k = int(torch.searchsorted(ends, torch.tensor([total], device=DEV))[0])
    slots = torch.repeat_interleave(torch.arange(n, device=DEV), r)
    slots = slots[torch.randperm(total, generator=g, device=DEV)]
    comm = torch.searchsorted(ends[:k + 1], torch.arange(total, device=DEV), right=True)
    key = torch.unique(comm * n + slots)                             # a node once per community
    return key // n, key % n, r


def _edges(shape, n, degree, seed):
    """(src, dst) int32 on the device: undirected edges with repeats, self-loops
    and gaps in the ids, as edge lists come."""
    g = _gen(seed)
    large = shape == "power" and degree > 40.0
    comm, node, r = _cover(g, n, shape, 5000 if large else 2000)
    k = int(comm[-1]) + 1
    if shape == "power":
        gamma, cap = (2.2, 95000.0) if large else (2.5, 700.0)
        w = (torch.arange(n, device=DEV, dtype=torch.float64) + 1.0) ** (-1.0 / (gamma - 1.0))
        w = w * (degree / w.mean())
        for _ in range(8):
            w = w.clamp(max=min(cap, n / 2.0))
            w = w * (degree / w.mean())
        w = w[torch.randperm(n, generator=g, device=DEV)]
        mu = 0.3
    else:
        w = torch.full((n,), float(degree), device=DEV, dtype=torch.float64)
        mu = 0.02
    wi = (w * 4096.0).long().clamp(min=1)
    a = torch.div(wi[node], r[node], rounding_mode="floor").clamp(min=1)
    cum = torch.cumsum(a, 0)
    size = torch.bincount(comm, minlength=k)
    end = torch.cumsum(size, 0)
    cum0 = torch.cat([torch.zeros(1, device=DEV, dtype=torch.int64), cum])
    lo, hi = cum0[end - size], cum0[end]
    mass = hi - lo
    target = n * degree / 2.0
    want = (1.0 - mu) * target * mass.double() / float(int(mass.sum()))
    ec = (want + _uniform(g, k)).long()
    if large:
        ec = torch.minimum(ec, size * (size - 1) // 4)               # small communities stay below saturation
    ec = torch.where(size >= 2, ec, torch.zeros_like(ec))
    of = torch.repeat_interleave(torch.arange(k, device=DEV), ec)
    ends = []
    for _ in range(2):
        at = lo[of] + _below(g, mass[of])
        ends.append(node[torch.searchsorted(cum, at, right=True)].int())
        del at
    del of
    gcum = torch.cumsum(wi, 0)
    nb = int(round(mu * target))
    whole = torch.full((nb,), int(gcum[-1]), device=DEV, dtype=torch.int64)
    for i in range(2):
        ends[i] = torch.cat([ends[i], torch.searchsorted(gcum, _below(g, whole), right=True).int()])
    # every node is the end of an edge
    ids = torch.arange(n, device=DEV, dtype=torch.int32)
    proper = ends[0] != ends[1]
    touched = torch.zeros(n, device=DEV, dtype=torch.bool)
    for e in ends:
        touched[e[proper].long()] = True
    lonely = ids[~touched]
    src = torch.cat([ends[0], lonely])
    dst = torch.cat([ends[1], (lonely + 1) % n])
    label = (7 + torch.cumsum(1 + (_uniform(g, n) * 3.0).long().clamp(max=2), 0)).int()
    return label[src.long()], label[dst.long()]


def _batch_sizes(case):
    """Nodes (log-uniform) and mean degree of every graph: the case's own, so
    that a batch has the same number of nodes for every seed."""
    u = np.random.default_rng([case["count"], case["n_hi"], case["q"]]).random((2, case["count"]))
    n = np.exp(u[0] * (math.log(case["n_hi"]) - math.log(case["n_lo"])) + math.log(case["n_lo"]))
    return np.round(n).astype(np.int64), 8.0 + 32.0 * u[1]


def _covers(n, seed):
    """A reference cover and a detected one: the reference with a fifth of its
    memberships dropped, some moved to other communities, and some split."""
    g = _gen(seed)
    comm, node, _ = _cover(g, n, "power", 2000)
    u = _uniform(g, comm.shape[0])
    keep = u > 0.2
    k = int(comm[-1]) + 1
    moved = torch.where(u > 0.9, _below(g, torch.full_like(comm, k)), comm)
    split = moved * 2 + ((moved % 3 == 0) & (node % 2 == 0)).long()
    out = []
    for c, v in ((split[keep], node[keep]), (comm, node)):
        key = torch.unique(c * n + v)
        c, v = key // n, key % n
        _, cnt = torch.unique(c, return_counts=True)
        off = torch.cat([torch.zeros(1, device=DEV, dtype=torch.int64), torch.cumsum(cnt, 0)])
        out.append((off.cpu().numpy(), v.int().cpu().numpy()))
    return out


def _num_detected(n):
    return n // 6 + 16


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "f1":
        state["det"], state["ref"] = _covers(case["n"], seed)
        state["best"] = np.full(_num_detected(case["n"]), -1, np.int32)
        return state
    if kind == "batch":
        state["graphs"] = []
        for i, (n, d) in enumerate(zip(*_batch_sizes(case))):
            s, t = _edges("planted", int(n), float(d), seed * 1009 + i)
            state["graphs"].append((s.cpu().numpy(), t.cpu().numpy()))
        state.update(_buffers(int(_batch_sizes(case)[0].sum()), case["iters"]))
        return state
    src, dst = _edges(case["shape"], case["n"], case["degree"], seed)
    if "iters" in case:
        state.update(_buffers(case["n"], case["iters"]))
    if kind == "call":
        state["src"], state["dst"] = src.cpu().numpy(), dst.cpu().numpy()
    elif kind == "run":
        state["graph"] = lazyfox.Graph(src, dst, gain_rule=case.get("rule"))
    elif kind == "triangles":
        with lazyfox.Graph(src, dst) as graph:
            off, adj = graph.oriented()
        state["off"] = torch.from_numpy(off).to(DEV)
        state["adj"] = torch.from_numpy(adj).to(DEV)
        state["t"] = torch.empty(off.shape[0] - 1, device=DEV, dtype=torch.int64)
        state["vt"] = torch.empty(off.shape[0] - 1, device=DEV, dtype=torch.int32)
    else:
        state["src"], state["dst"] = src, dst
        state["stream"] = torch.cuda.Stream()
        state["stream"].wait_stream(torch.cuda.current_stream())
    return state


# --- one pass -----------------------------------------------------------------

def _threshold(case):
    return 0.01 if case["stop"] else -math.inf


def _buffers(n, iters):
    """The caller's own arrays for a run's results, whose lengths differ from
    graph to graph: the values come first, then 0 (histories) or -1 (cover)."""
    return dict(wcc=np.zeros(iters), joins=np.zeros(iters, np.int64), leaves=np.zeros(iters, np.int64),
                offsets=np.full(n + 1, -1, np.int64), members=np.full(min(iters + 1, 16) * n, -1, np.int32), used={})


def _put(state, name, values, rest):
    k, buf = values.shape[0], state[name]
    buf[:k] = values
    buf[k:state["used"].get(name, 0)] = rest
    state["used"][name] = k
    return buf


def _result(state, st, offsets, members):
    return dict(wcc_initial=st.wcc_initial, wcc=_put(state, "wcc", st.wcc_history, 0.0),
                joins=_put(state, "joins", st.joins, 0), leaves=_put(state, "leaves", st.leaves, 0),
                offsets=_put(state, "offsets", offsets, -1), members=_put(state, "members", members, -1))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "f1":
        f1, best = lazyfox.cover_f1(state["det"], state["ref"])
        state["best"][:best.shape[0]] = best
        return dict(f1=f1, best=state["best"])
    if kind == "triangles":
        lazyfox.lf_triangles_noalloc(state["off"], state["adj"], state["t"], state["vt"])
        return dict(t=state["t"], vt=state["vt"])
    if kind == "create":
        with lazyfox.Graph(state["src"], state["dst"], stream=state["stream"]) as graph:
            t, vt, cc = graph.node_stats()
            return dict(t=t, vt=vt, cc=cc, order=graph.order())
    if kind == "batch":
        with lazyfox.Batch(state["graphs"]) as batch:
            st = batch.run(case["q"], _threshold(case), case["iters"])
            info = batch.info()
            offsets, members = batch.communities()
            return dict(wcc_initial=info["wcc_initial"], wcc_final=info["wcc_final"], cc=info["cc"],
                        iterations=info["iterations"], joins=_put(state, "joins", st.joins, 0),
                        leaves=_put(state, "leaves", st.leaves, 0), offsets=_put(state, "offsets", offsets, -1),
                        members=_put(state, "members", members, -1))
    if kind == "call":
        communities, st = lazyfox.run_lazyfox(state["src"], state["dst"], case["q"], _threshold(case), case["iters"])
        sizes = np.array([c.shape[0] for c in communities], dtype=np.int64)
        offsets = np.concatenate([np.zeros(1, np.int64), np.cumsum(sizes)])
        return _result(state, st, offsets, np.concatenate(communities) if communities else np.zeros(0, np.int32))
    if kind == "detect":
        with lazyfox.Graph(state["src"], state["dst"], stream=state["stream"], gain_rule=case.get("rule")) as graph:
            st = graph.run(case["q"], _threshold(case), case["iters"])
            return _result(state, st, *graph.communities())
    st = state["graph"].run(case["q"], _threshold(case), case["iters"])
    return _result(state, st, *state["graph"].communities())


# --- what a pass cannot do without ----------------------------------------------

def work(case):
    """Bytes: the edge list once; per iteration every neighbour id, every
    node's offset and position and its memberships (read and written); the
    cover once.  A run that stops by itself is taken as 6 (power) or 20
    (planted) iterations.  Operations: about 20 per (neighbour, membership)
    pair and iteration, two memberships per node."""
    kind = case["kind"]
    if kind == "f1":
        m = 1.6 * case["n"]
        return {"bytes": 2 * 4 * m + 8 * m / 10, "flops": 10 * m}
    if kind == "batch":
        ln = math.log(case["n_hi"] / case["n_lo"])
        n = case["count"] * ((case["n_hi"] - case["n_lo"]) / ln if ln > 0 else case["n_lo"])
        m = 12.0 * n
    else:
        n = float(case["n"])
        m = n * case["degree"] / 2.0
    if kind == "triangles":
        return {"bytes": 8 * n + 4 * m + 12 * n, "flops": 4 * m}
    if kind == "create":
        return {"bytes": 8 * m + 8 * m + 16 * n, "flops": 8 * m}
    iters = case["iters"] if not case["stop"] else 20 if case["shape"] == "planted" else 6
    once = 8 * m if kind != "run" else 0
    return {"bytes": once + iters * (8 * m + 12 * n + 32 * n) + 8 * n, "flops": iters * 80.0 * m}


# --- the same results in plain torch and numpy ----------------------------------

class _Plain:
    """The preprocessing, the initial clustering and, for small graphs, whole
    runs, written out in 64 bits."""

    def __init__(self, src, dst):
        src, dst = (torch.as_tensor(v).to(DEV).long() for v in (src, dst))
        keep = src != dst
        src, dst = src[keep], dst[keep]
        self.label, inv = torch.unique(torch.cat([src, dst]), return_inverse=True)
        n = self.n = self.label.shape[0]
        a, b = inv[:src.shape[0]], inv[src.shape[0]:]
        key = torch.unique(torch.cat([a * n + b, b * n + a]))
        self.row, self.col = key // n, key % n
        self.key = key
        self.deg = torch.bincount(self.row, minlength=n)
        self.off = torch.cat([torch.zeros(1, device=DEV, dtype=torch.int64), torch.cumsum(self.deg, 0)])
        self._triangles()
        d = self.deg.double()
        pairs = 0.5 * d * (d - 1.0)
        local = torch.where(self.deg > 1, self.t.double() / pairs.clamp(min=1.0), torch.zeros_like(d)).cpu().numpy()
        self.cc = math.fsum(local) / n if n else 0.0
        deg = self.deg.cpu().numpy()
        self.order = np.lexsort((np.arange(n), -deg, -local))

    def _triangles(self):
        n = self.n
        up = (self.deg[self.row] * n + self.row) < (self.deg[self.col] * n + self.col)
        ou, ov = self.row[up], self.col[up]
        okey = ou * n + ov
        odeg = torch.bincount(ou, minlength=n)
        ooff = torch.cat([torch.zeros(1, device=DEV, dtype=torch.int64), torch.cumsum(odeg, 0)])
        later = ooff[ou + 1] - torch.arange(ou.shape[0], device=DEV) - 1   # out-neighbours of u listed after v
        self.t = torch.zeros(n, device=DEV, dtype=torch.int64)
        mark = torch.zeros(ou.shape[0], device=DEV, dtype=torch.bool)
        total = torch.cumsum(later, 0)
        start, e = 0, ou.shape[0]
        while start < e:
            base = int(total[start - 1]) if start else 0
            stop = int(torch.searchsorted(total, torch.tensor([base + (1 << 26)], device=DEV), right=True)[0])
            stop = min(max(stop, start + 1), e)
            first = torch.repeat_interleave(torch.arange(start, stop, device=DEV), later[start:stop])
            k = torch.arange(first.shape[0], device=DEV) - (total - later)[first] + base
            second = first + 1 + k
            v, w = ov[first], ov[second]
            swap = (self.deg[v] * n + v) > (self.deg[w] * n + w)
            want = torch.where(swap, w * n + v, v * n + w)
            third = torch.searchsorted(okey, want).clamp(max=e - 1)
            hit = okey[third] == want
            first, second, third = first[hit], second[hit], third[hit]
            for node in (ou[first], ov[first], ov[second]):
                self.t += torch.bincount(node, minlength=n)
            for edge in (first, second, third):
                mark[edge] = True
            start = stop
        self.vt = torch.bincount(ou[mark], minlength=n) + torch.bincount(ov[mark], minlength=n)

    def clustering(self):
        """Community of every node: walking the order, a free node opens one
        and its free neighbours join it."""
        off, col = self.off.tolist(), self.col.cpu().numpy()
        of = np.full(self.n, -1, np.int64)
        k = 0
        for x in self.order.tolist():
            if of[x] < 0:
                nb = col[off[x]:off[x + 1]]
                of[nb[of[nb] < 0]] = k
                of[x] = k
                k += 1
        return of, k

    def terms(self, k, d, n, m2):
        """WCC-hat of members with k of their d neighbours inside a community
        of n members and m2/2 inner edges."""
        k, d = np.asarray(k, np.float64), np.asarray(d, np.float64)
        if n < 2 or not self.cc > 0.0:
            return np.zeros(k.shape)
        p = m2 / (float(n) * (n - 1.0))
        inside = np.where(k >= 1, 0.5 * (k * (k - 1.0)), 0.0) * p
        around = np.where(d >= 1, 0.5 * (d * (d - 1.0)), 0.0) * self.cc
        ok = around > 0.0
        r = inside / np.where(ok, around, 1.0) * (d / ((n - 1.0) + (d - k)))
        return np.where(ok, r, 0.0)

    def initial_total(self):
        of, k = self.clustering()
        ofd = torch.as_tensor(of, device=DEV)
        same = ofd[self.row] == ofd[self.col]
        inner = torch.bincount(self.row[same], minlength=self.n).cpu().numpy()
        size = np.bincount(of, minlength=k)
        m2 = np.bincount(of, weights=inner, minlength=k)
        n_, m_, d = size[of].astype(np.float64), m2[of], self.deg.cpu().numpy().astype(np.float64)
        p = m_ / np.maximum(n_ * (n_ - 1.0), 1.0)
        inside = np.where(inner >= 1, 0.5 * (inner * (inner - 1.0)), 0.0) * p
        around = 0.5 * (d * (d - 1.0)) * self.cc
        ok = (around > 0.0) & (n_ >= 2)
        return math.fsum(np.where(ok, inside / np.where(ok, around, 1.0) * (d / ((n_ - 1.0) + (d - inner))), 0.0))

    def whole_run(self, q, threshold, iters):
        off, col, deg = self.off.tolist(), self.col.cpu().numpy(), self.deg.cpu().numpy()
        nb = [col[off[x]:off[x + 1]].tolist() for x in range(self.n)]
        nbset = [set(v) for v in nb]
        of, k = self.clustering()
        members = [set(np.flatnonzero(of == c).tolist()) for c in range(k)]
        mine = [{int(c)} for c in of]

        def count(y, c):
            return len(nbset[y] & members[c])

        def sum_of(c):
            ys = list(members[c])
            ks = [count(y, c) for y in ys]
            return ys, ks, sum(ks)

        def total():
            out = []
            for c in range(k):
                if members[c]:
                    ys, ks, m2 = sum_of(c)
                    out.extend(self.terms(ks, deg[ys], len(ys), m2).tolist())
            return math.fsum(out)

        def gain(x, c, join, inside):
            ys, ks, m2 = inside
            kx = count(x, c)
            step = 1 if join else -1
            before = self.terms(ks, deg[ys], len(ys), m2)
            new_y = [y for y in ys if join or y != x]
            new_k = [kk + step * (y in nbset[x]) for y, kk in zip(ys, ks) if join or y != x]
            if join:
                new_y.append(x)
                new_k.append(kx)
            after = self.terms(new_k, deg[new_y], len(new_y), m2 + 2 * step * kx)
            return math.fsum(after.tolist() + (-before).tolist())

        t0 = last = total()
        wcc, joins, leaves = [], [], []
        order = self.order.tolist()
        for _ in range(iters):
            nj = nl = 0
            for s in range(0, self.n, q):
                acts, inside = [], {}
                for x in order[s:s + q]:
                    best = {True: (0.0, -1), False: (0.0, -1)}
                    for c in sorted(set().union(mine[x], *(mine[y] for y in nb[x]))):
                        if c not in inside:
                            inside[c] = sum_of(c)
                        join = c not in mine[x]
                        v = gain(x, c, join, inside[c])
                        if v > best[join][0]:
                            best[join] = (v, c)
                    acts.append((x, best[False][1], best[True][1]))
                for x, out, into in acts:
                    if out >= 0:
                        members[out].discard(x)
                        mine[x].discard(out)
                        nl += 1
                    if into >= 0:
                        members[into].add(x)
                        mine[x].add(into)
                        nj += 1
            for c in range(k):
                if len(members[c]) == 1:
                    mine[members[c].pop()].discard(c)
            now = total()
            wcc.append(now)
            joins.append(nj)
            leaves.append(nl)
            if (now - last) / last < threshold if last != 0.0 else now == 0.0:
                break
            last = now
        cover = [sorted(c) for c in members if c]
        out = _buffers(self.n, iters)
        out["wcc"][:len(wcc)], out["joins"][:len(wcc)], out["leaves"][:len(wcc)] = wcc, joins, leaves
        out["offsets"][:len(cover) + 1] = np.cumsum([0] + [len(c) for c in cover])
        inside = [x for c in cover for x in c]
        out["members"][:len(inside)] = self.label.cpu().numpy()[inside]
        out.pop("used")
        return dict(wcc_initial=t0, **out)


def _plain_f1(det, ref, room):
    (oa, ma), (ob, mb) = det, ref
    ka, kb = oa.shape[0] - 1, ob.shape[0] - 1
    sa, sb = np.diff(oa), np.diff(ob)
    ca, cb = np.repeat(np.arange(ka), sa), np.repeat(np.arange(kb), sb)
    by = np.argsort(mb, kind="stable")
    mbs, cbs = mb[by], cb[by]
    lo, hi = np.searchsorted(mbs, ma, "left"), np.searchsorted(mbs, ma, "right")
    cnt = hi - lo
    at = np.repeat(lo - (np.cumsum(cnt) - cnt), cnt) + np.arange(int(cnt.sum()))
    pair, both = np.unique(np.repeat(ca, cnt) * np.int64(kb) + cbs[at], return_counts=True)
    a, b = pair // kb, pair % kb
    p, r = both / sa[a], both / sb[b]
    f = 2.0 * (p * r) / (p + r)
    best, top = np.full(room, -1, np.int32), np.zeros(ka)
    for i in np.lexsort((-b, f)):      # the last write of a community: largest F1, then lowest index
        best[a[i]], top[a[i]] = b[i], f[i]
    return dict(f1=math.fsum(top) / ka if ka else 0.0, best=best)


def exact(case, seed):
    kind = case["kind"]
    if kind == "f1":
        return _plain_f1(*_covers(case["n"], seed), _num_detected(case["n"]))
    if kind == "batch":
        t0, cc = [], []
        for i, (n, d) in enumerate(zip(*_batch_sizes(case))):
            g = _Plain(*_edges("planted", int(n), float(d), seed * 1009 + i))
            t0.append(g.initial_total())
            cc.append(g.cc)
        return dict(wcc_initial=np.array(t0), wcc_final=None, cc=np.array(cc), iterations=None, joins=None,
                    leaves=None, offsets=None, members=None)
    if case["n"] > 400000 or case["n"] * case["degree"] > 8e6:
        return None
    g = _Plain(*_edges(case["shape"], case["n"], case["degree"], seed))
    if kind == "triangles":
        return dict(t=g.t, vt=g.vt.int())
    if kind == "create":
        return dict(t=g.t.cpu().numpy(), vt=g.vt.int().cpu().numpy(), cc=g.cc, order=g.order.astype(np.int32))
    if case["n"] <= 400 and case.get("rule") is None:
        return g.whole_run(case["q"], _threshold(case), case["iters"])
    return dict(wcc_initial=g.initial_total(), wcc=None, joins=None, leaves=None, offsets=None, members=None)
